"""Box states of a batch, N and F moved as rows of the class arrays: what was
set comes back, for every box, whatever its place in its class and its size
(odd sizes: rows that start at no multiple of 16 bytes), from host and device
memory; in mixed precision N and F rounded to float, exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KEYS = ("nH", "xHII", "xHeII", "xHeIII", "T", "N", "F")


@pytest.mark.parametrize("prec", ["RT_FP64", "RT_MIXED"])
@pytest.mark.parametrize("device", [False, True])
def test_box_state_round_trip(prec, device):
    import torch
    from paper_1304_7126_gb300 import rt as R
    from paper_1304_7126_gb300 import workloads as W
    boxes = W.batched(8, seed0=5, steps=2, sides=(5, 7, 8, 13))
    bt = R.RTBatch(boxes, precision=getattr(R, prec))
    rng = np.random.default_rng(1)
    want = []
    for i, w in enumerate(boxes):
        s = w.state()
        s["N"] = 10 ** rng.uniform(-12, 0, s["N"].size)
        s["F"] = np.repeat(s["N"].reshape(w.G, 1, -1), 3, axis=1).reshape(-1) * w.cr * rng.uniform(-0.5, 0.5, s["F"].size)
        want.append(s)
        bt.set_box_state(i, {k: torch.as_tensor(s[k]).cuda() for k in KEYS} if device else s)
    for i, s in enumerate(want):
        got = bt.get_box_state(i)
        for k in KEYS:
            ref = s[k].astype(np.float32).astype(np.float64) if prec == "RT_MIXED" and k in "NF" else s[k]
            assert np.array_equal(got[k], ref), (i, k)
