"""The reciprocals, quotients and roots of the FP64 paths that start from float
pairs, and the fixed-point wave speeds of the transport, against IEEE arithmetic
within the bounds stated beside them (csrc/dfmath.cuh, csrc/transport_math.cuh):

* 1/b and a/b of the thermochemistry: the nearest double (but for one quotient
  in 2^35), outside 2^-70 .. 2^70 in magnitude exactly the IEEE quotient, zero,
  infinities and NaN included;
* 1/b, 1/sqrt(b) of the transport for positive b of any size and sqrt(t) of t in
  [1, 4]: within an ulp;
* doubles of magnitude up to 1 to fixed point (2^-62) cut off exactly, and back
  as the nearest double;
* wave speeds within 2^-50 of the bilinear table in double arithmetic, at the
  ends of its rows and columns too.

The headers are compiled into a small library of the test's own (nvcc)."""
import ctypes as C
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1304_7126_gb300", "csrc")
N = 1 << 21

HARNESS = r'''
#include "transport_math.cuh"
using namespace rtgb;
__global__ void k(int fn, long long n, const double *a, const double *b, double *y, long long *z, const long long *tab)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    switch (fn) {
    case 0: y[i] = dfm::fast_rcp(b[i]); break;
    case 1: y[i] = dfm::fast_div(a[i], b[i]); break;
    case 2: y[i] = trcp(b[i]); break;
    case 3: y[i] = trsqrt(b[i]); break;
    case 4: y[i] = tsqrt14(b[i]); break;
    case 5: z[i] = (long long)to_fix(b[i]); break;
    case 6: y[i] = from_fix((unsigned long long)z[i]); break;
    case 7: {   // f = a in [0, 1], mu = b
        unsigned long long v = to_fix(a[i]);
        if (v >= (1ULL << 62)) v = (1ULL << 62) - 1ULL;
        long long lo, hi;
        hll_lookup_fix(tab, (int)(v >> 54), v << 10, b[i], lo, hi);
        z[2 * i] = lo;
        z[2 * i + 1] = hi;
    }
    }
}
extern "C" int run(int fn, long long n, const double *a, const double *b, double *y, long long *z, const long long *tab)
{
    k<<<(unsigned)((n + 255) / 256), 256>>>(fn, n, a, b, y, z, tab);
    cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? (int)e : (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    from paper_1304_7126_gb300 import _build
    d = tmp_path_factory.mktemp("quotients")
    src, lib = str(d / "harness.cu"), str(d / "harness.so")
    open(src, "w").write(HARNESS)
    subprocess.check_call([_build.nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, "-I",
                           _build.INCLUDE] + _build.ARCH + [src, "-o", lib, "-lcudart"])
    L = C.CDLL(lib)
    L.run.argtypes = [C.c_int, C.c_longlong] + [C.c_void_p] * 5

    def call(fn, b, a=None, z=None, tab=None):
        dev = lambda v: None if v is None else torch.as_tensor(v).cuda()   # noqa: E731
        b, a, z, tab = dev(b), dev(a), dev(z), dev(tab)
        n = len(b if b is not None else z)
        y = torch.zeros(n, dtype=torch.float64, device="cuda")
        if z is None:
            z = torch.zeros(2 * n, dtype=torch.int64, device="cuda")
        torch.cuda.synchronize()
        p = lambda t: None if t is None else t.data_ptr()   # noqa: E731
        assert L.run(fn, n, p(a), p(b), p(y), p(z), p(tab)) == 0
        return y.cpu().numpy(), z.cpu().numpy()

    return call


def _random(rng, e0, e1, n, sign=True):
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(e0, e1, n))
    return x * rng.choice([-1.0, 1.0], n) if sign else x


def _same(got, ref):
    return (got == ref) | (np.isnan(got) & np.isnan(ref))


SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.0, -1.0, 2.0 ** -70, 2.0 ** 70, 2.0 ** 71, 1.5 * 2.0 ** -71,
                    np.nextafter(2.0 ** -70, 0), np.nextafter(2.0 ** 70, np.inf), 5e-324, 2.0 ** -1022, 1.7e308,
                    np.nextafter(1.0, 2)])


def test_thermochemistry_reciprocal_and_quotient(run):
    rng = np.random.default_rng(1)
    for e0, e1 in ((-70, 70), (-3, 3)):
        b = _random(rng, e0, e1, N)
        a = _random(rng, -400, 400, N)
        assert np.sum(run(0, b)[0] != 1.0 / b) <= 1
        assert np.sum(run(1, b, a)[0] != a / b) <= 1
    with np.errstate(all="ignore"):
        for lo, hi in ((-1000, -71), (71, 1000)):
            b = _random(rng, lo, hi, N // 8)
            a = _random(rng, -20, 20, N // 8)
            assert np.all(_same(run(0, b)[0], 1.0 / b)) and np.all(_same(run(1, b, a)[0], a / b))
        assert np.all(_same(run(0, SPECIAL)[0], 1.0 / SPECIAL))
        a = np.array([1.0, -3.0, 0.0, 1e-300])
        A, B = (v.reshape(-1).copy() for v in np.meshgrid(a, SPECIAL))
        assert np.all(_same(run(1, B, A)[0], A / B))
    # 1/(2 - 2^-52) lies 2^-107 above the middle of two doubles: too close for either
    # function to decide, so the bound is what the 2^-88 before rounding leave, half
    # an ulp (2^-54 here) and 2^-88
    b = np.nextafter(2.0, 1)
    for r in (run(0, np.array([b]))[0][0], run(1, np.array([b]), np.array([1.0]))[0][0]):
        assert abs(Fraction(r) - 1 / Fraction(b)) <= Fraction(1, 1 << 54) + Fraction(1, 1 << 88)


@pytest.mark.parametrize("fn", [2, 3])
def test_transport_reciprocal_and_root(run, fn):
    rng = np.random.default_rng(2)
    for e0, e1 in ((-1022, 1023), (-100, 100), (0, 2)):
        b = _random(rng, e0, e1, N, sign=False)
        ref = 1.0 / b if fn == 2 else np.asarray(1.0 / np.sqrt(b.astype(np.longdouble)), dtype=np.float64)
        ok = np.abs(ref) >= 2.0 ** -1022
        got = run(fn, b)[0]
        assert np.all(np.abs(got - ref)[ok] <= np.spacing(ref)[ok])
    with np.errstate(all="ignore"):
        b = np.array([0.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, 1.7e308])
        ref = 1.0 / b if fn == 2 else 1.0 / np.sqrt(b)
        got = run(fn, b)[0]
        fin = np.isfinite(ref) & (ref > 0)
        assert np.all(np.abs(got - ref)[fin] <= 2 * np.spacing(ref[fin])) and np.all(_same(got, ref)[~fin])


def test_transport_sqrt(run):
    rng = np.random.default_rng(3)
    t = np.concatenate([rng.uniform(1.0, 4.0, N), [1.0, 4.0, np.nextafter(1.0, 2), np.nextafter(4.0, 1), 2.0]])
    ref = np.sqrt(t)
    assert np.all(np.abs(run(4, t)[0] - ref) <= np.spacing(ref))


def test_fixed_point(run):
    rng = np.random.default_rng(4)
    x = np.concatenate([_random(rng, -70, 0, N), [0.0, -0.0, 1.0, -1.0, np.nextafter(1.0, 0), 5e-324]])
    z = run(5, x)[1][:len(x)].astype(np.uint64)
    ref = np.floor(np.abs(x) * 2.0 ** 62)          # exact: a scaling, then whole numbers below 2^62 or multiples of 2^9
    assert np.array_equal(z, ref.astype(np.uint64))
    v = np.concatenate([rng.integers(0, 1 << 62, N), (1 << rng.integers(0, 62, N)) + rng.integers(0, 3, N),
                        [0, 1, (1 << 62) - 1, 1 << 62, (1 << 63) - 1]]).astype(np.int64)
    y = run(6, None, z=v)[0]
    err = np.abs(np.asarray(y, dtype=np.longdouble) * np.longdouble(2.0) ** 62 - v.astype(np.longdouble))
    assert np.all(err <= 0.5 * np.spacing(np.maximum(v.astype(np.float64), 1.0))) and y[-5] == 0.0


def test_wave_speeds(run):
    from paper_1304_7126_gb300 import rt as R
    tab = R.rt_hll_table(257, 257)
    fix = (tab * 2.0 ** 62).astype(np.int64)       # towards zero, as the library makes it
    rng = np.random.default_rng(5)
    f = np.concatenate([rng.uniform(0, 1, N), rng.integers(0, 257, 4096) / 256.0, np.ones(4096), np.zeros(4096)])
    mu = rng.uniform(-1, 1, len(f))
    mu[::7] = rng.integers(-128, 129, len(mu[::7])) / 128.0
    mu[::11] = rng.choice([-1.0, 1.0], len(mu[::11]))
    z = run(7, mu, f, tab=fix.reshape(-1))[1].reshape(-1, 2)
    x, m = f * 256.0, (mu + 1.0) * 128.0
    i, j = np.minimum(x.astype(int), 255), np.minimum(m.astype(int), 255)
    u, w = (x - i)[:, None], (m - j)[:, None]
    ref = (1 - u) * ((1 - w) * tab[i, j] + w * tab[i, j + 1]) + u * ((1 - w) * tab[i + 1, j] + w * tab[i + 1, j + 1])
    assert np.max(np.abs(z * 2.0 ** -62 - ref)) <= 2.0 ** -50
