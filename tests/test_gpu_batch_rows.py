"""Boxes of a batch whose class has longer rows of N and F than the limit that
CUDA states for 2-D copies (2^31 - 1 bytes; N and F of a box are moved as rows of
the class arrays): what was set comes back, from host and device memory."""
import numpy as np
import pytest


pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("prec,nbig", [("RT_FP64", 16), ("RT_MIXED", 32)])   # 2^28, 2^29 cells of one group
def test_box_state_in_a_class_beyond_the_pitch_limit(prec, nbig, device):
    import torch
    from paper_1304_7126_gb300 import rt as R
    from paper_1304_7126_gb300 import workloads as W
    if torch.cuda.mem_get_info()[0] < 100 << 30:
        pytest.skip("needs 100 GB of free device memory")
    small, big = W.stromgren32(7), W.stromgren32(7)
    big.shape = (256, 256, 256)   # (zero state: only the small boxes at both ends are set)
    boxes = [small] + [big] * nbig + [small]
    bt = R.RTBatch(boxes, precision=getattr(R, prec))
    rng = np.random.default_rng(1)
    want = []
    for i in (0, nbig + 1):
        s = small.state()
        s["N"] = (10 ** rng.uniform(-12, 0, s["N"].size)).astype(np.float32).astype(np.float64)
        s["F"] = (rng.uniform(-0.5, 0.5, (3, s["N"].size)) * s["N"] * small.cr).astype(np.float32).reshape(-1).astype(np.float64)
        bt.set_box_state(i, {k: torch.as_tensor(v).cuda() for k, v in s.items()} if device else s)
        want.append((i, s))
    for i, s in want:
        got = bt.get_box_state(i)
        for k in s:
            assert np.array_equal(got[k], s[k]), (i, k)
    bt.close()


STAGING = """
import numpy as np
from paper_1304_7126_gb300 import rt as R
from paper_1304_7126_gb300 import workloads as W
w = W.stromgren32(152)                      # a row of 13.4 MB as float
w.G = 8
w.sigN, w.sigE, w.egy = np.repeat(w.sigN, 8, 0), np.repeat(w.sigE, 8, 0), np.repeat(w.egy, 8)
bt = R.RTBatch([w], precision=R.RT_MIXED)
rng = np.random.default_rng(2)
s = w.state()
for k in "NF":
    rng.random(out=s[k])
mb = lambda key: int([l for l in open("/proc/self/status") if l.startswith(key)][0].split()[1]) / 1024.0
now, peak = lambda: mb("VmRSS"), lambda: mb("VmHWM")   # (getrusage's peak starts at the parent's)
a = now()
bt.set_box_state(0, s)
b = peak()
c = now()
got = bt.get_box_state(0)
d = peak()
for k in s:
    assert np.array_equal(got[k], s[k].astype(np.float32).astype(np.float64) if k in "NF" else s[k]), k
print(b - a, d - c - sum(v.nbytes for v in got.values()) / 2**20)
"""


def test_host_staging_is_bounded():
    """RT_MIXED through host memory: N and F are rounded to float in chunks of
    rows (several here, the last one shorter), 64 MB of staging, not in a copy of
    all rows of F (322 MB); the process's memory peak says so."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", STAGING], cwd=root, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    put, get = map(float, r.stdout.split())
    print("MB beyond the state's own arrays: set %.0f, get %.0f" % (put, get))
    assert put < 160 and get < 160, (put, get)
