"""A NaN of either sign or an infinity in the photon state ends as
RT_ENONFINITE, never as photons that are not there: states from device memory
are not checked on entry, so the step has to carry what it finds to where it is
reported.  One value of N or F replaced, in the middle of the box and in a
corner, for every precision, flux function and transport kernel (single box,
batch).  (A cell with an infinite N may sub-cycle up to the cap, set low
here; RT_ENONFINITE is reported before RT_ESUBCYCLE.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
KEYS = ("nH", "xHII", "xHeII", "xHeIII", "T", "N", "F")
VALUES = np.concatenate([np.array([0x7ff8000000000000, 0xfff8000000000000], dtype=np.uint64).view(np.float64),
                         [np.inf, -np.inf]])


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("flux", [0, 1])
@pytest.mark.parametrize("prec", ["RT_FP64", "RT_MIXED"])
def test_nonfinite_photons_reported(prec, flux, batch):
    import torch
    from paper_1304_7126_gb300 import rt as R
    from paper_1304_7126_gb300 import workloads as W
    w = W.small_cosmo(12, seed=3, nsrc=3, flux=flux)
    opts = dict(precision=getattr(R, prec), max_subcycles=4000)
    sim = R.RT.from_workload(w, **opts)
    dt = sim.courant_dt()
    for _ in range(3):
        sim.step(dt)
    s0 = sim.get_state()
    bt = R.RTBatch([w], **opts) if batch else None

    def code(s):
        dev = {k: torch.as_tensor(s[k]).cuda() for k in KEYS}
        try:
            if batch:
                bt.set_box_state(0, dev)
                bt.step(dt)
                bt.sync()
            else:
                sim.set_state(dev)
                sim.step(dt)
                sim.sync()
        except R.RTError as e:
            return e.code
        return R.RT_OK

    assert code(s0) == R.RT_OK
    nc = w.ncells
    for key, comp in (("N", 0), ("F", 0), ("F", 1), ("F", 2)):
        for v in VALUES:
            for cell in (0, (6 * 12 + 6) * 12 + 6):
                s = {k: a.copy() for k, a in s0.items()}
                s[key].view(np.uint64)[comp * nc + cell] = v.view(np.uint64)
                assert code(s) == R.RT_ENONFINITE, (key, comp, v, np.signbit(v), cell)
    assert code(s0) == R.RT_OK
