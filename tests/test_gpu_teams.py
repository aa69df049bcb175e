"""The team kernels of the thermochemistry (two and four lanes per cell) and
the adjoint's teams (one tangent per lane, eight or sixteen lanes per cell)
at every group count.

* FP64: a step with every attempt in the one-thread first pass, one with the
  attempts after the first in teams of two and four, and one with teams of
  four alone give identical bits for every field and attempt count, for 1 to
  8 groups (5: a lane of a team of two or four without a group in its last
  round), without helium, isothermal, without the on-the-spot approximation
  and smoothed.
* The one-step adjoint against central differences of the step, as in the
  three-group case (1e-5: the truncation and rounding of the differences),
  at 1 group, at 4 (the first count whose nine tangents need a second team
  of eight) and at 8.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
STATE = ("xHII", "xHeII", "xHeIII", "T", "N", "F")


@pytest.fixture(scope="module")
def R():
    import torch
    assert torch.cuda.is_available()
    from paper_1304_7126_gb300 import rt
    rt.load()
    return rt


def _box(G, n=12, helium=True, flux=0, **over):
    """Small cosmological box with G groups: the three black-body groups and
    harder and harder copies of them."""
    from paper_1304_7126_gb300 import workloads as W
    w = W.small_cosmo(n, seed=3, nsrc=3, flux=flux)
    i, s = np.arange(G) % 3, 1.0 / (1 + np.arange(G) // 3)
    w.G = G
    w.sigN, w.sigE, w.egy = w.sigN[i] * s[:, None], w.sigE[i] * s[:, None], w.egy[i] / s
    w.src_L = w.src_L[:, i] * s / G
    if not helium:
        w.X = 1.0
    for k, v in over.items():
        setattr(w, k, v)
    if w.isothermal:
        w.T = np.full(w.ncells, 1e4)
    return w


@pytest.mark.parametrize("G,over,opts", [(g, {}, {}) for g in range(1, 9)] + [
    (3, {"helium": False}, {}),
    (1, {"helium": False, "isothermal": True}, {}),
    (4, {"isothermal": True}, {}),
    (3, {"otsa": False}, {}),
    (5, {"otsa": False, "isothermal": True}, {}),
    (3, {}, {"smooth": 1}),
    (5, {"otsa": False}, {"smooth": 1})])
def test_teams_equal_one_thread(R, G, over, opts):
    w = _box(G, **over)
    sims = []
    for routing in ((1 << 20, 0, 0, -1),   # every attempt in the first pass
                    (1, 1, 1, 0),          # teams of two, cells handed to teams of four after two attempts
                    (1, 0, 0, -1)):        # the whole queue to teams of four
        sim = R.RT.from_workload(w, **opts)
        sim.set_thermo_routing(*routing)
        sims.append(sim)
    dt = sims[0].courant_dt()
    most = 0
    for step in range(3):
        for sim in sims:
            sim.step(dt)
        ref, sub = sims[0].get_state(), sims[0].subcycles()
        most = max(most, int(sub.max()))
        for sim in sims[1:]:
            got = sim.get_state()
            assert np.array_equal(sim.subcycles(), sub), step
            for k in STATE:
                assert np.array_equal(got[k], ref[k]), (step, k)
    assert most > 16


@pytest.mark.parametrize("G", [1, 4, 8])
def test_adjoint_teams_directional(R, G):
    import torch
    w = _box(G, n=8)
    sim = R.RT.from_workload(w)
    dt = sim.courant_dt()
    sim.run(dt, 3)
    s0 = sim.get_state()
    nc = w.ncells
    rng = np.random.default_rng(G)
    Nm = s0["N"].max()
    v = {"xHII": rng.standard_normal(nc), "xHeII": rng.standard_normal(nc), "xHeIII": rng.standard_normal(nc),
         "T": rng.standard_normal(nc) / 1e4, "N": rng.standard_normal(G * nc) / Nm,
         "F": rng.standard_normal(3 * G * nc) / (w.cr * Nm)}
    u = {"N": s0["N"] * rng.standard_normal(G * nc), "F": s0["F"] * rng.standard_normal(3 * G * nc) * 0.1,
         "xHII": np.minimum(s0["xHII"] - 1e-6, 1 - s0["xHII"]) * rng.standard_normal(nc),
         "T": s0["T"] * rng.standard_normal(nc), "nH": s0["nH"] * rng.standard_normal(nc)}

    def step(eps):
        sim.set_state({k: a + eps * u[k] if k in u else a for k, a in s0.items()})
        sim.step(dt)
        out = sim.get_state()
        return sum(float(v[k] @ out[k]) for k in v), sim.subcycles()

    (jp, sp), (jm, sm), (_, sub) = step(1e-7), step(-1e-7), step(0.0)
    assert np.array_equal(sp, sub) and np.array_equal(sm, sub) and sub.max() > 6
    dev = lambda a: torch.as_tensor(np.array(a, dtype=np.float64)).cuda()
    sim.set_state(s0)
    lam = {k: dev(v[k]) for k in v}
    g_nH, g_L = dev(np.zeros(nc)), dev(np.zeros((len(w.src_ijk), G)))
    assert sim.step_vjp(dt, lam, g_nH, g_L, check=True) == 0
    torch.cuda.synchronize()
    ad = sum(float(lam[k].cpu().numpy() @ u[k]) for k in ("N", "F", "xHII", "T")) + \
        float(g_nH.cpu().numpy() @ u["nH"])
    fd = (jp - jm) / 2e-7
    assert abs(ad - fd) <= 1e-5 * abs(fd), (ad, fd)
