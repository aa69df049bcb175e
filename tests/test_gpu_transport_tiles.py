"""Transport on the 32 x 4 tiles of small boxes, and the FP64 closure and
wave speeds at the ends of their ranges.

A group's transport does not depend on the others, so a box of one group
(32 x 4 tiles) and the same box with its group eight times over (32 x 8
tiles) give identical bits per group, in FP64 and FP32, for GLF and HLL; the
FP64 state is within 1e-12 of the oracle (the transport tolerance of the
parity tests), every step from the oracle's state: where opposing beams
cancel, a cell is left with photons of rounding size and a flux of any
direction, whose wave speeds set its neighbours' HLL fluxes a step later.
Shapes, eight groups of which take the large tiles in FP32
(four CTAs per SM) as well but for the single cell: the largest box of the rule in FP64 at 152 SMs
(two CTAs each, 2 x 4 x 38 = 304) and the first beyond it, ragged ends of a
tile, single rows and a single cell."""
import numpy as np
import pytest

from parity import compare, oracle_problem

pytestmark = pytest.mark.gpu
C_LIGHT = 2.99792458e10


@pytest.fixture(scope="module")
def R():
    import torch
    assert torch.cuda.is_available()
    from paper_1304_7126_gb300 import rt
    rt.load()
    return rt


def _workload(shape, flux, G):
    from paper_1304_7126_gb300 import workloads as W
    nc = int(np.prod(shape))
    w = W.Workload(name="tr", shape=shape, dx=3e20, G=G, cr=C_LIGHT / 100, sigN=np.zeros((G, 3)),
                   sigE=np.zeros((G, 3)), egy=np.full(G, 3e-11), X=1.0, isothermal=True, otsa=True,
                   flux=flux, bc=(0, 1, 2, 2, 1, 0), steps=3)
    w.nH, w.xHII, w.T = np.full(nc, 1e-3), np.full(nc, 0.5), np.full(nc, 1e4)
    w.xHeII, w.xHeIII = np.zeros(nc), np.zeros(nc)
    w.src_ijk = np.array([[shape[2] // 2, shape[1] // 2, shape[0] // 2]], dtype=np.int32)
    w.src_L = np.full((1, G), 1e55)
    return w


def _photons(w, kind, seed=5):
    """N, F of one group: random, or the extremes of the closure: f = 0, f = 1
    and a few roundings below it along +-x, +-y, +-z (mu = +-1 and 0), opposing
    beams, and cells with next to no photons beside full ones."""
    nc = w.ncells
    rng = np.random.default_rng(seed)
    N = 10 ** rng.uniform(-3, 0, nc)
    d = rng.standard_normal((3, nc))
    d /= np.linalg.norm(d, axis=0)
    f = rng.uniform(0, 1, nc)
    if kind == "ends":
        k = rng.integers(0, 8, nc)
        axis = np.zeros((3, nc))
        axis[k % 3, np.arange(nc)] = np.where(rng.random(nc) < 0.5, 1.0, -1.0)
        d = np.where(k < 6, axis, d)
        f = np.where(k == 7, 0.0, np.where(k % 2 == 0, 1.0, 1.0 + 2e-16 * rng.integers(-4, 1, nc)))
        N = np.where(rng.random(nc) < 0.2, 1e-25, N)
    return N, w.cr * N * f * d


@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("shape,kind", [((38, 32, 32), "random"), ((39, 32, 32), "random"), ((10, 13, 40), "random"),
                                        ((20, 5, 33), "ends"), ((20, 16, 16), "ends"), ((39, 1, 1), "ends"),
                                        ((1, 1, 1), "random")])
def test_small_tiles(oracle_mod, R, flux, shape, kind):
    G = 8
    w1, w8 = _workload(shape, flux, 1), _workload(shape, flux, G)
    N, F = _photons(w1, kind)
    s1, s8 = w1.state(), w8.state()
    s1["N"], s1["F"] = N.copy(), F.reshape(-1).copy()
    s8["N"], s8["F"] = np.tile(N, G), np.tile(F.reshape(-1), G)
    for prec in (R.RT_FP64, R.RT_MIXED):
        a, b = R.RT.from_workload(w1, precision=prec), R.RT.from_workload(w8, precision=prec)
        a.set_state(s1)
        b.set_state(s8)
        dt = a.courant_dt()
        ref = {k: v.copy() for k, v in s1.items()}
        p = oracle_problem(oracle_mod, w1)
        for step in range(3):
            if step > 0:
                a.set_state(ref)
                b.set_state({k: np.tile(ref[k], G) if k in "NF" else ref[k] for k in ref})
            a.step(dt)
            b.step(dt)
            ga, gb = a.get_state(), b.get_state()
            for k in ("N", "F"):
                assert np.array_equal(np.tile(ga[k], G), gb[k]), (prec, step, k)
            assert np.all(np.isfinite(ga["N"])) and np.all(np.isfinite(ga["F"]))
            assert np.allclose(a.budget()[0], b.budget()[G - 1], rtol=1e-12, atol=1e-12 * a.budget()[0, 3])
            st, _, _, _ = p.step(ref, dt, w1.src_ijk, w1.src_L)
            assert st == 0
            if prec == R.RT_FP64:
                e = compare(ga, ref, ("N", "F"), cr=w1.cr, G=1)
                assert e["N"] < 1e-12 and e["F"] < 1e-12, (step, e)
