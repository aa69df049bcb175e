"""Routing and timing leave no trace in the result, in any precision, with and
without smoothing: a box whose queue is several times what the team kernels
hold at once, so that the teams take further cells from it and, once it is
empty, hand running ones to the second stage.  Which attempts of a cell run
where then depends on timing; x_HII, x_HeII, x_HeIII, T, N, F and the attempt
counts must be the same bits in repeated runs and for every routing.

Every cell is neutral gas in a strong photon field: x_HII grows from 1e-6 by at
most 10% per sub-step, more than 64 of them, so that every cell is queued after
its first attempt and a cell taken as the queue runs empty has many sub-steps
ahead whenever it looks (after two attempts).

And the team kernel's fast path gives way to the exact one, with the same bits
again, where its arguments are out of range.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
STATE = ("xHII", "xHeII", "xHeIII", "T", "N", "F")
N_SIDE = 64
ROUTINGS = ((1, 1, 1, 0), (1, 1, 1, 0),   # both stages, looking every two attempts; twice
            (1, 0, 0, 1 << 30),           # the second stage alone
            (3, 7, 8, 0),
            (1 << 20, 0, 0, -1))          # every attempt in the first pass


@pytest.mark.parametrize("smooth", [0, 1])
@pytest.mark.parametrize("prec", ["RT_FP64", "RT_MIXED", "RT_MIXED32"])
def test_long_queue_same_bits(prec, smooth):
    import torch
    from paper_1304_7126_gb300 import rt as R
    from paper_1304_7126_gb300 import workloads as W
    w = W.cosmo(N_SIDE, 5, 4, 10)
    # stage 1 holds 64 cells per block of 128 threads, 16 blocks per SM at most
    assert w.ncells > 64 * 16 * torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(11)
    s = w.state()
    s["nH"] = np.clip(s["nH"], 1e-4, 1e-2)
    s["N"] = 10 ** rng.uniform(-1.5, -0.5, s["N"].size)
    s["F"] = np.repeat(s["N"].reshape(w.G, 1, -1), 3, axis=1).reshape(-1) * w.cr * rng.uniform(-0.5, 0.5, s["F"].size)
    ref = None
    for routing in ROUTINGS:
        sim = R.RT.from_workload(w, precision=getattr(R, prec), smooth=smooth)
        sim.set_thermo_routing(*routing)
        sim.set_state(s)
        sim.step()
        got, sub = sim.get_state(), sim.subcycles().copy()
        sim.close()
        if ref is None:
            assert sub.min() > 64, sub.min()
            ref, ref_sub = got, sub
        assert np.array_equal(sub, ref_sub), routing
        for k in STATE:
            assert np.array_equal(got[k], ref[k]), (routing, k, int((got[k] != ref[k]).sum()))


@pytest.mark.parametrize("T", [2e18, 1e21])
def test_out_of_range_recombination_same_bits(T):
    """Recombination photons without the on-the-spot approximation in gas beyond
    the range of the team kernel's fast path (2^60 K): its attempts there are made
    again the exact way, with recombination rates of their own, and give the bits
    of the one-thread path.  No other photons, so that N is made of them."""
    from paper_1304_7126_gb300 import rt as R
    from paper_1304_7126_gb300 import workloads as W
    w = W.small_cosmo(12, seed=3, nsrc=3)
    w.otsa = False
    w.src_ijk, w.src_L = w.src_ijk[:0], w.src_L[:0]
    s = w.state()
    s["T"][:], s["xHII"][:], s["xHeII"][:] = T, 0.9, 0.5
    s["nH"] *= 1e6
    ref = None
    for routing in ((1 << 20, 0, 0, -1), (1, 1, 1, 0), (1, 0, 0, -1)):
        sim = R.RT.from_workload(w)
        sim.set_thermo_routing(*routing)
        sim.set_state(s)
        sim.step()
        got, sub = sim.get_state(), sim.subcycles().copy()
        sim.close()
        if ref is None:
            assert sub.min() > 64 and got["N"].max() > 0
            ref, ref_sub = got, sub
        assert np.array_equal(sub, ref_sub), routing
        for k in STATE:
            assert np.array_equal(got[k], ref[k]), (routing, k, int((got[k] != ref[k]).sum()))
