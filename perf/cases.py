"""Workloads of the RT step for performance work: what users of the library
have it do, through its public entry points (the ctypes binding of the C-ABI
and torch.autograd), from the smallest box to the largest.

``listed()`` names the workloads, ``draw`` gives others of the same ranges,
``prepare`` makes the inputs of a seed, ``run`` is one pass, ``work`` the
bytes and operations that a pass cannot do without, ``tolerance`` how far
apart two correct implementations may be, and ``exact`` the same pass in
plain 64-bit torch / numpy, written from the method's equations (Rosdahl et
al. 2013: M1 moments, App. A thermochemistry, the rate fits of its appendix)
without the library.

A pass puts the state into the handle, takes ``steps`` RT steps and reads
the result, which is what a program does between two checkpoints (and what
the differentiable run does per segment), so that every pass of a case does
the same work whatever ran before it.

Inputs are synthetic and seeded: log-normal densities, ionised bubbles around
the sources with their photon field (`front` > 0, their mean radius in cells:
a run in progress), or neutral gas without photons (`front` = 0: the first steps).
"""
import math

import numpy as np
import torch

from paper_1304_7126_gb300 import adjoint as A
from paper_1304_7126_gb300 import rt as R
from paper_1304_7126_gb300 import workloads as W

C_LIGHT = 2.99792458e10          # cm/s
KPC = 3.0856775814913673e21      # cm
DEV = "cuda"
KEYS = ("nH", "xHII", "xHeII", "xHeIII", "T", "N", "F")
PREC = {"fp64": R.RT_FP64, "mixed": R.RT_MIXED, "mixed32": R.RT_MIXED32}
FLUX = {"GLF": R.RT_GLF, "HLL": R.RT_HLL}
OUT, REF, PER, INF = R.RT_BC_OUTFLOW, R.RT_BC_REFLECT, R.RT_BC_PERIODIC, R.RT_BC_INFLOW
BCS = {
    "outflow": (OUT,) * 6,
    "octant": (REF, OUT, REF, OUT, REF, OUT),     # the source in a reflecting corner
    "mixed": (REF, OUT, PER, PER, OUT, REF),
    "periodic": (PER,) * 6,
    "inflow": (INF,) + (OUT,) * 5,                # a plane-parallel flux through x = 0
}


def _case(kind, nx, ny, nz, **kw):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, G=3, flux="HLL", bc="outflow", precision="fp64", recipe="cosmo",
             otsa=True, nsrc=8, front=0.0, steps=2, budget=False)
    c.update(kw)
    return c


def listed():
    def named(name, c):
        return dict(name=name, **c)
    return [
        # one eager step of a very small box, read back: interactive use, unit-sized problems
        named("step16", _case("run", 16, 16, 16, nsrc=2, front=2.5, steps=1)),
        # Stromgren sphere in a reflecting corner (isothermal hydrogen, one group): many short steps between
        # two outputs, launched as a graph
        named("stromgren32", _case("run", 32, 32, 32, G=1, flux="GLF", bc="octant", recipe="stromgren", nsrc=1,
                                   front=13.0, steps=40)),
        # a ragged box with reflecting, periodic and open faces, an odd number of steps, the photon ledger read
        named("ragged_bc", _case("run", 37, 19, 51, bc="mixed", flux="GLF", nsrc=3, front=2.5, steps=3, budget=True)),
        # recombination photons followed (no on-the-spot approximation), a mid-sized box in progress
        named("nonotsa48", _case("run", 48, 48, 48, otsa=False, nsrc=4, front=2.5)),
        # cosmological field, FP64, 3 groups, HLL: the first steps from neutral gas
        named("cosmo128_start", _case("run", 128, 128, 128, nsrc=16)),
        # the same field well into the run: ionised bubbles around every source
        named("cosmo128_late", _case("run", 128, 128, 128, nsrc=16, front=3.0)),
        # the same in mixed precision with FP32 rate functions
        named("cosmo128_mixed32", _case("run", 128, 128, 128, nsrc=16, front=3.0, precision="mixed32")),
        # the largest box, mixed precision
        named("cosmo256_mixed", _case("run", 256, 256, 256, nsrc=64, front=3.0, precision="mixed")),
        # dense cloud in a plane-parallel flux: hydrogen only, no source, the ledger read
        named("shadow128", _case("run", 128, 128, 128, recipe="shadow", bc="inflow", nsrc=0, front=32.0, steps=4,
                                 budget=True)),
        # a batch of independent boxes of uneven sizes, 1 or 3 groups each, mixed precision
        named("batch48", _case("batch", 64, 64, 64, recipe="batch", precision="mixed", nsrc=48)),
        # gradient of the neutral hydrogen mass with respect to density, luminosities and initial temperature through
        # the run (checkpointed autograd), GLF
        named("train24", _case("train", 24, 24, 24, flux="GLF", nsrc=4, front=2.5)),
        # state in host memory in, one step, state out: a host program that owns the state
        named("host96", _case("host", 96, 96, 96, nsrc=8, front=2.5, steps=1)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more workload of the ranges above (boxes of 10^3 to 2 x 10^6 cells,
    sides odd or even)."""
    kind = rng.choice(["run"] * 7 + ["batch", "train", "host", "thermo"])
    flux = rng.choice(["HLL", "HLL", "GLF"])
    if kind == "batch":
        return _case("batch", rng.choice([32, 48, 64]), 0, 0, recipe="batch", flux=flux, nsrc=_log_int(rng, 4, 48),
                     precision=rng.choice(["mixed", "fp64", "mixed32"]), steps=rng.randint(1, 3))
    n = _log_int(rng, 10, {"run": 128, "host": 96, "thermo": 62, "train": 24}[kind])
    nx, ny, nz = (max(6, int(n * rng.uniform(0.8, 1.2))) for _ in range(3))
    if kind == "run":
        while nx * ny * nz > 2100000:
            nz -= 8
    if kind == "thermo":
        while nx * ny * nz > 262144:
            nz -= 4
    recipe = rng.choice(["cosmo"] * 4 + ["stromgren", "shadow"]) if kind in ("run", "host") else "cosmo"
    nsrc = 0 if recipe == "shadow" else _log_int(rng, 1, max(1, n // 6))
    bc = "inflow" if recipe == "shadow" else rng.choice(["outflow", "outflow", "octant", "mixed", "periodic"])
    otsa = kind != "run" or recipe != "cosmo" or rng.random() < 0.8
    front = {"cosmo": rng.uniform(1.5, 4.0), "stromgren": n * rng.uniform(0.2, 0.6), "shadow": nx * rng.uniform(0.1, 0.5)}
    return _case(kind, nx, ny, nz, G=1 if recipe == "stromgren" else rng.choice([1, 2, 3, 3]), flux=flux, bc=bc,
                 precision=rng.choice(["fp64", "fp64", "mixed", "mixed32"]) if kind == "run" and otsa else "fp64",
                 recipe=recipe, otsa=otsa, nsrc=nsrc, front=front[recipe], steps=rng.randint(1, 4),
                 budget=rng.random() < 0.3)


# ---------------------------------------------------------------------------
# inputs

def _groups(case):
    """sigma^N, sigma^E [G][3], mean energies [G], photon fractions [G]."""
    G = case["G"]
    if case["recipe"] == "stromgren":
        return np.array(W.H1_SIGN), np.array(W.H1_SIGE), np.array(W.H1_EGY_EV) * W.EV, np.ones(1)
    if G == 1:
        return np.array(W.BB1_SIGN), np.array(W.BB1_SIGE), np.array(W.BB1_EGY_EV) * W.EV, np.ones(1)
    f = np.array(W.BB3_PHOTON_FRACTION)[:G]
    return np.array(W.BB3_SIGN)[:G], np.array(W.BB3_SIGE)[:G], np.array(W.BB3_EGY_EV)[:G] * W.EV, f / f.sum()


def _density(shape, gen, mean):
    """Log-normal density, P(k) ~ k^-3, sigma_ln = 1."""
    w = torch.fft.rfftn(torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
    m = max(shape)
    kz, ky = (torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) * m for n in shape[:2])
    kx = torch.fft.rfftfreq(shape[2], device=DEV, dtype=torch.float64) * m
    k = torch.sqrt(kz[:, None, None] ** 2 + ky[None, :, None] ** 2 + kx[None, None, :] ** 2)
    k = torch.where(k > 0, k, torch.inf)
    g = torch.fft.irfftn(w * k ** -1.5, s=shape)
    rho = torch.exp((g - g.mean()) / g.std())
    return rho * (mean / rho.mean())


def _bubbles(shape, dx, cr, sigN, nH, src, L, radius, gen, he, age, xbg, Tbg, Nbg, octant):
    """Ionised bubbles of the given radii (cells) around sources: photon field
    L / (4 pi r^2 c_r), absorbed beyond the front by neutral gas of the mean
    density (the hard photons leak out), flux radial."""
    nz, ny, nx = shape
    G = L.shape[1]
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) for n in (nx, ny, nz)]
    N = torch.full((G,) + shape, Nbg, device=DEV, dtype=torch.float64)
    F = torch.zeros((G, 3) + shape, device=DEV, dtype=torch.float64)
    jit = torch.exp(0.05 * torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
    scale = torch.exp(0.05 * torch.randn((G, 1) + shape, generator=gen, device=DEV, dtype=torch.float64))
    tau = dx * float(nH.mean()) * (sigN[:, 0] + he * sigN[:, 1])    # per cell of neutral gas
    for s in range(len(src)):
        d = [ax[k] - float(src[s][k]) for k in range(3)]
        dz, dy, dxx = d[2][:, None, None], d[1][None, :, None], d[0][None, None, :]
        r2 = dz * dz + dy * dy + dxx * dxx
        r = torch.sqrt(r2)
        geo = (8.0 if octant else 1.0) / (4 * math.pi * (r2 + 0.25) * dx * dx * cr)
        f = 0.95 * cr * r / (r2 + 1.0)          # |F| / N / r: reduced flux 0.95 r^2 / (r^2 + 1)
        past = (r - radius[s]).clamp(min=0.0)
        for g in range(G):
            n = float(L[s, g]) * geo * torch.exp(-float(tau[g]) * past)
            n = torch.where(n > 1e-40, n, torch.zeros_like(n))
            N[g] += n
            F[g, 0] += n * f * dxx
            F[g, 1] += n * f * dy
            F[g, 2] += n * f * dz
    N *= scale[:, 0]
    F *= scale
    # fractions: in balance with the photon field (x^2 alpha n = (1 - x) Gamma), or still growing (`age` of light)
    gam = [sum(float(sigN[g, j]) * cr * N[g] for g in range(G)) + 1e-60 for j in range(3)]
    a = 2.0e-13 * nH
    x = 2.0 * gam[0] / (gam[0] + torch.sqrt(gam[0] ** 2 + 4.0 * a * gam[0])) * (1.0 - 1e-5 * jit)
    x = torch.clamp(torch.minimum(x, 1.0 - torch.exp(-age * gam[0])), xbg, 1.0)
    a = a * x + 1e-60
    r2, r3 = gam[1] / (1.1 * a), gam[2] / (6.0 * a)      # HeII / HeI, HeIII / HeII
    r2 = torch.minimum(r2, torch.expm1((age * gam[1]).clamp(max=80.0)))
    r3 = torch.minimum(r3, torch.expm1((0.5 * age * gam[2]).clamp(max=80.0)))
    y1 = 1.0 / (1.0 + r2 * (1.0 + r3))
    y3 = y1 * r2 * r3
    T = Tbg + 2e4 * torch.sqrt(x - xbg) * jit
    return N, F, x, (1.0 - y1 - y3).clamp(min=0.0), y3, T


def _box(case, seed):
    """The physical problem of a box: grid constants (numbers, numpy) and the
    initial state (CUDA tensors, library layout)."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1 + int(seed))
    rng = np.random.default_rng(int(seed))
    shape = (case["nz"], case["ny"], case["nx"])
    nz, ny, nx = shape
    nc = nx * ny * nz
    G, recipe, n = case["G"], case["recipe"], max(nx, ny, nz)
    sigN, sigE, egy, frac = _groups(case)
    p = dict(shape=shape, G=G, sigN=sigN, sigE=sigE, egy=egy, flux=case["flux"], bc=BCS[case["bc"]], X=0.76,
             isothermal=False, otsa=case["otsa"], cfl=0.8, inflow=None)
    zero = torch.zeros(shape, device=DEV, dtype=torch.float64)
    if recipe == "shadow":        # dense cloud in thin gas, a flux of 1e6 photons / cm^2 / s entering at x = 0
        p.update(X=1.0, dx=6.6 * KPC / n, cr=C_LIGHT / 10)
        ax = [(torch.arange(m, device=DEV, dtype=torch.float64) + 0.5) * p["dx"] for m in (nz, ny, nx)]
        c = [0.5 * nz * p["dx"], 0.5 * ny * p["dx"], (5.0 / 6.6) * nx * p["dx"]]
        r2 = sum((a.reshape([-1 if k == j else 1 for k in range(3)]) - c[j]) ** 2 for j, a in enumerate(ax))
        inside = (r2 <= (0.8 * KPC) ** 2).double()
        jit = torch.exp(0.1 * torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
        nH = (2e-4 + (4e-2 - 2e-4) * inside) * jit
        Fin = 1e6 * frac
        front = case["front"] * (0.9 + 0.2 * rng.random())
        lit = torch.sigmoid((front - torch.arange(nx, device=DEV, dtype=torch.float64)) / 1.5)
        lit = (lit * (lit > 1e-12))[None, None, :] + zero
        N = torch.stack([lit * float(f) / p["cr"] for f in Fin]) * jit
        F = torch.stack([torch.stack([N[g] * p["cr"] * 0.999, zero, zero]) for g in range(G)])
        x = torch.clamp(lit * (1 - 1e-3 * jit), 1e-6, 1.0)
        T = (8000.0 - 7960.0 * inside) * jit + 8e3 * lit
        inflow = np.zeros((6, G, 4))
        inflow[0, :, 0] = Fin / p["cr"]
        inflow[0, :, 1] = Fin
        p.update(src=np.zeros((0, 3), np.int32), L=np.zeros((0, G)), inflow=inflow)
        y2 = y3 = zero
    else:
        if recipe == "stromgren":
            p.update(X=1.0, isothermal=True, dx=6.6 * KPC / n, cr=C_LIGHT / 100)
            nH = torch.full(shape, 1e-3, device=DEV, dtype=torch.float64)
            nH *= torch.exp(0.02 * torch.randn(shape, generator=gen, device=DEV, dtype=torch.float64))
            src = np.zeros((1, 3), np.int32)
            lum = np.array([5e48 / 8])
            xbg, Tbg = 1.2e-3, 1e4
        elif recipe == "batch":
            p.update(dx=6.6 * KPC / 128, cr=C_LIGHT / 100)
            nH = _density(shape, gen, 10.0 ** rng.uniform(-4, -1))
            cells = rng.choice(nc, size=min(nc, int(rng.integers(1, 9))), replace=False)
            src = np.stack([cells % nx, cells // nx % ny, cells // (nx * ny)], 1).astype(np.int32)
            lum = 10.0 ** rng.uniform(48, 52, size=len(src))
            xbg, Tbg = 1e-6, 100.0
        else:                     # cosmological box: sources of 1e52 photons / s at the densest cells
            p.update(dx=0.8e3 * KPC / 128, cr=C_LIGHT / 10)
            nH = _density(shape, gen, 1e-3)
            top = torch.topk(nH.reshape(-1), min(nc, case["nsrc"])).indices.cpu().numpy()
            src = np.stack([top % nx, top // nx % ny, top // (nx * ny)], 1).astype(np.int32)
            lum = np.full(len(src), 1e52)
            xbg, Tbg = 1e-6, 100.0
        L = np.outer(lum, frac)
        p.update(src=src, L=L)
        if case["front"] > 0:
            radius = case["front"] * (0.7 + 0.6 * rng.random(len(src)))
            # without the on-the-spot approximation every cell holds recombination photons
            N, F, x, y2, y3, T = _bubbles(shape, p["dx"], p["cr"], sigN, nH, src, L, radius, gen,
                                          (1 - p["X"]) / (4 * p["X"]), 30 * p["dx"] / p["cr"], xbg, Tbg,
                                          0.0 if case["otsa"] else 1e-20, recipe == "stromgren")
            if p["X"] == 1.0:
                y2, y3 = zero, zero
            if p["isothermal"]:
                T = torch.full(shape, 1e4, device=DEV, dtype=torch.float64)
        else:
            N = torch.zeros((G,) + shape, device=DEV, dtype=torch.float64)
            F = torch.zeros((G, 3) + shape, device=DEV, dtype=torch.float64)
            x = torch.full(shape, xbg, device=DEV, dtype=torch.float64)
            y2, y3 = zero, zero
            T = torch.full(shape, Tbg, device=DEV, dtype=torch.float64)
    state = dict(zip(KEYS, (v.reshape(-1).clone() for v in (nH, x, y2, y3, T, N, F))))
    p["dt"] = p["cfl"] * p["dx"] / (3.0 * p["cr"])
    return p, state


def _batch_boxes(case, seed):
    """`nsrc` boxes of uneven sides up to nx, 1 or 3 groups each."""
    rng = np.random.default_rng(case["nsrc"])       # the sizes belong to the case, the fields to the seed
    sides = [s for s in (16, 24, 32, 48, 64) if s <= case["nx"]]
    got = []
    for b in range(case["nsrc"]):
        n = int(rng.choice(sides))
        c = dict(case, nx=n, ny=n, nz=n, G=int(rng.choice([1, 3])), nsrc=1, front=float(rng.choice([0.0, 2.5])))
        got.append(_box(c, 1000 * int(seed) + b))
    return got


def _opts(case, p):
    return dict(X=p["X"], isothermal=int(p["isothermal"]), otsa=int(p["otsa"]), flux=FLUX[p["flux"]], cfl=p["cfl"],
                precision=PREC[case["precision"]])


def _handle(case, p, stream):
    sim = R.RT(p["shape"], p["dx"], p["G"], p["cr"], p["sigN"], p["sigE"], p["egy"], bc=p["bc"], **_opts(case, p))
    sim.set_stream(stream.cuda_stream)
    sim.set_sources(p["src"], p["L"])
    if p["inflow"] is not None:
        for face in range(6):
            if p["bc"][face] == INF:
                sim.set_inflow(face, p["inflow"][face])
    return sim


def prepare(case, seed):
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        if case["kind"] == "batch":
            boxes = _batch_boxes(case, seed)
            ws = [W.Workload(name="box%d" % i, shape=p["shape"], dx=p["dx"], G=p["G"], cr=p["cr"], sigN=p["sigN"],
                             sigE=p["sigE"], egy=p["egy"], X=p["X"], isothermal=False, otsa=True,
                             flux=FLUX[p["flux"]], bc=p["bc"], steps=case["steps"]) for i, (p, _) in enumerate(boxes)]
            sim = R.RTBatch(ws, precision=PREC[case["precision"]])
            sim.set_stream(stream.cuda_stream)
            for i, (p, s) in enumerate(boxes):
                sim.set_box_state(i, s)
                sim.set_box_sources(i, p["src"], p["L"])
            st = dict(case=case, sim=sim, boxes=boxes, dt=boxes[0][0]["dt"], stream=stream)
        else:
            p, s = _box(case, seed)
            st = dict(case=case, p=p, state=s, dt=p["dt"], stream=stream)
            if case["kind"] == "thermo":
                st["opt"] = R.default_options(**_opts(case, p))
                st["work"] = {k: v.clone() for k, v in s.items()}
                st["sub"] = torch.zeros(s["nH"].numel(), dtype=torch.int32, device=DEV)
            else:
                st["sim"] = _handle(case, p, stream)
            if case["kind"] == "host":   # the program's own pinned buffers
                pin = {k: v.cpu().pin_memory() for k, v in s.items()}
                out = {k: torch.empty_like(v).pin_memory() for k, v in pin.items()}
                st["keep"] = (pin, out)
                st["in"] = {k: v.numpy() for k, v in pin.items()}
                st["out"] = {k: v.numpy() for k, v in out.items()}
            if case["kind"] == "train":
                st["L"] = torch.as_tensor(p["L"], device=DEV)
                st["nH0"] = s["nH"].clone().requires_grad_(True)
                st["L0"] = st["L"].clone().requires_grad_(True)
                st["T0"] = s["T"].clone().requires_grad_(True)
    stream.synchronize()
    return st


# ---------------------------------------------------------------------------
# one pass

def _cat_state(boxes, G):
    """Empty tensors for the boxes of one group count, and each box's slices."""
    sel = [i for i, (p, _) in enumerate(boxes) if p["G"] == G]
    ncs = [int(np.prod(boxes[i][0]["shape"])) for i in sel]
    per = dict(nH=1, xHII=1, xHeII=1, xHeIII=1, T=1, N=G, F=3 * G)
    out = {k: torch.empty(sum(ncs) * per[k], dtype=torch.float64, device=DEV) for k in KEYS}
    cuts = {k: torch.split(out[k], [n * per[k] for n in ncs]) for k in KEYS}
    return sel, out, [{k: cuts[k][j] for k in KEYS} for j in range(len(sel))]


def run(state):
    case = state["case"]
    with torch.cuda.stream(state["stream"]):
        return RUN[case["kind"]](case, state)


def _run_box(case, st):
    sim = st["sim"]
    sim.set_state(st["state"])
    if case["steps"] == 1:
        sim.step(st["dt"])
    else:
        sim.run(st["dt"], case["steps"])
    out = sim.get_state(device=True)
    if case["budget"]:
        out["budget"] = sim.budget()
    return out


def _run_batch(case, st):
    sim = st["sim"]
    for i, (_, s) in enumerate(st["boxes"]):
        sim.set_box_state(i, s)
    sim.run(st["dt"], case["steps"])
    got = {}
    for G in sorted({p["G"] for p, _ in st["boxes"]}):
        sel, out, cut = _cat_state(st["boxes"], G)
        for i, c in zip(sel, cut):   # rt_batch_get_box_state into device arrays
            rc = sim.L.rt_batch_get_box_state(sim.h, i, *[c[k].data_ptr() for k in KEYS], 1)
            if rc:
                raise R.RTError(rc, "rt_batch_get_box_state")
        got["G%d" % G] = out
    return got


def _run_train(case, st):
    s = st["state"]
    s0 = dict(s, T=st["T0"])
    out = A.run(st["sim"], st["dt"], case["steps"], st["p"]["src"], st["nH0"], st["L0"], s0, every=2)
    loss = A.neutral_hydrogen_mass(out, st["p"]["dx"])
    g = torch.autograd.grad(loss, [st["nH0"], st["L0"], st["T0"]])
    return dict(loss=loss.detach(), g_nH=g[0], g_L=g[1], g_T=g[2], **{k: out[k].detach() for k in KEYS[1:]})


def _run_host(case, st):
    sim = st["sim"]
    sim.set_state(st["in"])
    for _ in range(case["steps"]):
        sim.step(st["dt"])
    return dict(sim.get_state(st["out"]))


def _run_thermo(case, st):
    # a host framework's own device arrays, updated in place
    for k in KEYS:
        st["work"][k].copy_(st["state"][k])
    p = st["p"]
    rc = R.rt_thermo_step_noalloc(st["sub"].numel(), p["G"], st["opt"], p["cr"], p["sigN"], p["sigE"], p["egy"],
                                  st["dt"], st["work"], st["sub"], st["stream"].cuda_stream)
    if rc:
        raise R.RTError(rc, "rt_thermo_step_noalloc")
    return dict(st["work"], subcycles=st["sub"])


RUN = {"run": _run_box, "batch": _run_batch, "train": _run_train, "host": _run_host, "thermo": _run_thermo}


# ---------------------------------------------------------------------------
# what a pass cannot do without, and how far apart two of them may be

def work(case):
    """Per RT step: the state (5 gas fields, N and F of every group) read and
    written once; the method's own operation counts, 355 (HLL) or 222 (GLF)
    flops per cell and group of the transport and, one sub-step per cell at
    least, 1370 flops of the thermochemistry (hydrogen only: about 500)."""
    if case["kind"] == "batch":
        side = np.mean([s ** 3 for s in (16, 24, 32, 48, 64) if s <= case["nx"]])
        nc, G = case["nsrc"] * side, 2.0
    else:
        nc, G = case["nx"] * case["ny"] * case["nz"], case["G"]
    photon = 8.0 if case["precision"] == "fp64" else 4.0
    by = nc * (9 * 8.0 + 8 * G * photon)
    fl = nc * (500.0 if case["recipe"] in ("stromgren", "shadow") else 1370.0)
    if case["kind"] != "thermo":
        fl += nc * G * (355.0 if case["flux"] == "HLL" else 222.0)
    steps = 1 if case["kind"] == "thermo" else case["steps"]
    if case["kind"] == "train":   # forward, recomputed forward, and the adjoint of every step
        by, fl = 4 * by, 4 * fl
    return {"bytes": by * steps, "flops": fl * steps}


def tolerance(case):
    # FP64: the library is 1e-14 from exact() (gradients 1e-13); its rate functions are good to 1e-12, and a
    # sub-step schedule that differs in one cell by a rounding at the 10% threshold shows in "max" first.
    # FP32 photon state: 1e-7 in N and F after a few steps.
    if case["precision"] == "fp64":
        return {"rel": 1e-11 if case["kind"] != "train" else 1e-9, "max": 1e-6, "differ": 1e-3}
    return {"rel": 1e-6, "max": 1e-3, "differ": 1e-3}


# ---------------------------------------------------------------------------
# the same pass in 64 bits

K_B = 1.380649e-16               # erg / K
M_P = 1.67262192e-24             # g
EPS = np.array([13.60, 24.59, 54.42]) * W.EV


def exact(case, seed):
    torch.cuda.empty_cache()
    if case["kind"] == "batch":
        boxes = _batch_boxes(case, seed)
        got = {}
        for G in sorted({p["G"] for p, _ in boxes}):
            sel = [b for b in boxes if b[0]["G"] == G]
            for _ in range(case["steps"]):
                for p, s in sel:
                    _exact_photons(p, s)
                nc = [s["nH"].numel() for _, s in sel]
                cat = {k: torch.cat([s[k] for _, s in sel]) for k in ("nH", "xHII", "xHeII", "xHeIII", "T")}
                cat["N"] = torch.cat([s["N"].view(G, -1) for _, s in sel], 1)
                cat["F"] = torch.cat([s["F"].view(3 * G, -1) for _, s in sel], 1)
                _exact_gas(sel[0][0], cat)
                cat["N"], cat["F"] = cat["N"].view(G, -1), cat["F"].view(3 * G, -1)
                for j, (_, s) in enumerate(sel):
                    for k in KEYS[1:]:
                        s[k] = torch.split(cat[k], nc, -1)[j].reshape(-1)
            got["G%d" % G] = {k: torch.cat([s[k] for _, s in sel]) for k in KEYS}
        return got
    p, s = _box(case, seed)
    s = dict(s)
    if case["kind"] == "thermo":
        _exact_gas(p, s)
        return dict({k: s[k].reshape(-1) for k in KEYS}, subcycles=None)
    L = torch.as_tensor(p["L"], device=DEV)
    if case["kind"] == "train":
        if s["nH"].numel() > 20000:
            return None          # the whole graph of a large box does not fit in 20 seconds
        leaf = [s["nH"].requires_grad_(True), L.requires_grad_(True), s["T"].requires_grad_(True)]
    V = p["dx"] ** 3
    budget = torch.zeros((p["G"], 4), device=DEV, dtype=torch.float64)
    for _ in range(case["steps"]):
        out = _exact_photons(p, s, L)
        before = s["N"].reshape(p["G"], -1).sum(1)
        _exact_gas(p, s)
        budget[:, 0] = s["N"].reshape(p["G"], -1).sum(1).detach() * V
        budget[:, 1] += (before - s["N"].reshape(p["G"], -1).sum(1)).detach() * V
        budget[:, 2] += out
        budget[:, 3] += L.detach().sum(0) * p["dt"]
    got = {k: s[k].detach().reshape(-1) for k in KEYS}
    if case["kind"] == "train":
        loss = M_P * V * torch.sum(s["nH"] * (1.0 - s["xHII"]))
        g = torch.autograd.grad(loss, leaf)
        del got["nH"]
        return dict(got, loss=loss.detach(), g_nH=g[0], g_L=g[1], g_T=g[2])
    if case["budget"]:
        got["budget"] = budget
    return {k: v.cpu().numpy() for k, v in got.items()} if case["kind"] == "host" else got


def _exact_photons(p, s, L=None):
    """Injection and transport of every group, in place in `s`; the net
    outflow through the open faces [G]."""
    G, shape, dt = p["G"], p["shape"], p["dt"]
    nz, ny, nx = shape
    N, F = s["N"].reshape((G,) + shape), s["F"].reshape((G, 3) + shape)
    if len(p["src"]):
        L = torch.as_tensor(p["L"], device=DEV) if L is None else L
        cell = torch.as_tensor(((p["src"][:, 2].astype(np.int64) * ny + p["src"][:, 1]) * nx + p["src"][:, 0]),
                               device=DEV)
        N = N.reshape(G, -1).index_add(1, cell, L.t() * (dt / p["dx"] ** 3)).reshape((G,) + shape)
    newN, newF, out = [], [], torch.zeros(G, device=DEV, dtype=torch.float64)
    for g in range(G):
        U = torch.cat([N[g:g + 1], F[g]])
        acc = torch.zeros_like(U)
        for d in range(3):                      # x, y, z are the last, middle and first grid axes
            ax = 3 - d
            lo, hi = _ghost(p, U, g, d, 0), _ghost(p, U, g, d, 1)
            f = _face_flux(p, torch.cat([lo, U, hi], ax), d, ax)
            m = U.shape[ax]
            acc = acc + f.narrow(ax, 0, m) - f.narrow(ax, 1, m)
            area = p["dx"] ** 2 * dt
            for side, sgn, at in ((0, -1.0, 0), (1, 1.0, m)):
                if p["bc"][2 * d + side] != PER:
                    out[g] += sgn * area * f.detach().narrow(ax, at, 1)[0].sum()
        U = U + (dt / p["dx"]) * acc
        U = torch.where(U[:1] < 0, torch.zeros_like(U), U)
        # |F| <= c_r N (scaled, so that the squares of tiny states keep their digits)
        top = U.detach().abs().amax(0).clamp(min=1e-300)
        fs = U[1:] / top
        mag = torch.sqrt((fs * fs).sum(0).clamp(min=1e-300))
        cn = p["cr"] * U[0] / top
        over = mag > cn
        sc = torch.where(over, cn / torch.where(over, mag, torch.ones_like(mag)), torch.ones_like(cn))
        newN.append(U[0])
        newF.append(U[1:] * sc)
    s["N"] = torch.stack(newN).reshape(-1)
    s["F"] = torch.stack(newF).reshape(-1)
    return out


def _ghost(p, U, g, d, side):
    ax = 3 - d
    bc = p["bc"][2 * d + side]
    at = U.shape[ax] - 1 if (side == 1) != (bc == PER) else 0
    u = U.narrow(ax, at, 1)
    if bc == REF:
        sign = torch.ones((4, 1, 1, 1), device=DEV, dtype=torch.float64)
        sign[1 + d] = -1.0
        u = u * sign
    if bc == INF:
        fix = torch.as_tensor(p["inflow"][2 * d + side][g], device=DEV)
        u = fix.reshape(4, 1, 1, 1).expand_as(u)
    return u


def _closure(p, U, d):
    """f, mu = n_d and the flux [F_d, c^2 P_d.] of the M1 closure."""
    c, N = p["cr"], U[0]
    scale = U[1:].detach().abs().amax(0)
    lit = (N > 1e-30) & (scale > 0)
    scale = torch.where(lit, scale, torch.ones_like(scale))
    fs = torch.where(lit, U[1:] / scale, torch.full_like(U[1:], 1.0))
    mag = torch.sqrt((fs * fs).sum(0))
    n = torch.where(lit, fs / mag, torch.zeros_like(fs))
    f = torch.where(lit, mag * scale / (c * torch.where(lit, N, torch.ones_like(N))), torch.zeros_like(N))
    f = torch.where(f > 1.0, torch.ones_like(f), f)
    chi = (3 + 4 * f * f) / (5 + 2 * torch.sqrt(4 - 3 * f * f))
    a, b = 0.5 * (1 - chi), 0.5 * (3 * chi - 1)
    P = c * c * N * b * n[d] * n
    P = torch.stack([P[k] + (c * c * N * a if k == d else 0.0) for k in range(3)])
    return f, n[d], torch.cat([U[1 + d:2 + d], P])


_TABLE = {}


def _speed_table():
    """Extreme eigenvalues of the M1 flux Jacobian on f = k/256, mu = -1 +
    j/128, in the closed form of Skinner & Ostriker (2013)."""
    if not _TABLE:
        f = np.arange(257)[:, None] / 256.0
        mu = -1.0 + np.arange(257)[None, :] / 128.0
        q = np.sqrt(4 - 3 * f * f)
        # 2 - f^2 - q and q - 1 in forms without cancellation
        t = -f * f * (1 - f * f) / (2 - f * f + q)
        r = np.sqrt((2.0 / 3.0) * q * 3 * (1 - f * f) / (q + 1) + 2 * mu * mu * t)
        _TABLE["lo"] = torch.as_tensor((mu * f - r) / q, device=DEV).reshape(-1)
        _TABLE["hi"] = torch.as_tensor((mu * f + r) / q, device=DEV).reshape(-1)
    return _TABLE["lo"], _TABLE["hi"]


def _speeds(p, f, mu):
    out = []
    fx, mx = f * 256.0, (mu + 1.0) * 128.0
    k, j = fx.detach().floor().clamp(0, 255), mx.detach().floor().clamp(0, 255)
    wf, wm = fx - k, mx - j
    at = (k * 257 + j).long()
    for t in _speed_table():
        a = t[at] + wm * (t[at + 1] - t[at])
        b = t[at + 257] + wm * (t[at + 258] - t[at + 257])
        out.append((a + wf * (b - a)) * p["cr"])
    return out


def _face_flux(p, U, d, ax):
    f, mu, Fl = _closure(p, U, d)
    m = U.shape[ax] - 1
    uL, uR, fL, fR = U.narrow(ax, 0, m), U.narrow(ax, 1, m), Fl.narrow(ax, 0, m), Fl.narrow(ax, 1, m)
    if p["flux"] == "GLF":
        return 0.5 * (fL + fR) - 0.5 * p["cr"] * (uR - uL)
    lo, hi = _speeds(p, f, mu)
    b = ax - 1
    lp = torch.where(hi.narrow(b, 0, m) >= hi.narrow(b, 1, m), hi.narrow(b, 0, m), hi.narrow(b, 1, m)).clamp(min=0)
    lm = torch.where(lo.narrow(b, 0, m) <= lo.narrow(b, 1, m), lo.narrow(b, 0, m), lo.narrow(b, 1, m)).clamp(max=0)
    den = lp - lm
    ok = den > 0
    den = torch.where(ok, den, torch.ones_like(den))
    return torch.where(ok, (lp * fL - lm * fR + lp * lm * (uR - uL)) / den, 0.5 * (fL + fR))


def _exact_gas(p, s):
    """Thermochemistry of every cell over dt, in place in `s`."""
    G = p["G"]
    s["N"], s["F"] = s["N"].reshape(G, -1), s["F"].reshape(G, 3, -1)
    nc = s["nH"].numel()
    rows = torch.cat([torch.stack([s["nH"], s["xHII"], s["xHeII"], s["xHeIII"], s["T"]]), s["N"],
                      torch.ones_like(s["N"])])
    grad = rows.requires_grad
    parts, ids = [], []
    for at in range(0, nc, 1 << 21):   # bounded temporaries
        i, r = _subcycle(p, rows[:, at:at + (1 << 21)], grad)
        ids += [k + at for k in i]
        parts += r
    order = torch.argsort(torch.cat(ids))
    new = torch.cat(parts, 1)[:, order]
    s["xHII"], s["xHeII"], s["xHeIII"], s["T"] = new[1], new[2], new[3], new[4]
    s["N"], fs = new[5:5 + G].reshape(-1), new[5 + G:]
    s["F"] = (s["F"] * fs[:, None, :]).reshape(-1)


class _Np:
    """numpy under the torch names used below"""
    where, stack, log, exp, sqrt, minimum = np.where, np.stack, np.log, np.exp, np.sqrt, np.minimum

    @staticmethod
    def least(a, v):
        return np.maximum(a, v)

    @staticmethod
    def most(a, v):
        return np.minimum(a, v)


class _Th:
    where, stack, log, exp, sqrt, minimum = torch.where, torch.stack, torch.log, torch.exp, torch.sqrt, torch.minimum

    @staticmethod
    def least(a, v):
        return torch.clamp(a, min=v)

    @staticmethod
    def most(a, v):
        return torch.clamp(a, max=v)


def _subcycle(p, rows, grad):
    """Sub-cycles the cells of `rows` over dt under the 10% rule; (ids,
    rows) of the cells in the order in which they finish."""
    xp = _Th
    n = rows.shape[1]
    ids = torch.arange(n, device=DEV)
    left = torch.full((n,), p["dt"], device=DEV, dtype=torch.float64)
    step = left.clone()
    out_i, out_r = [], []
    while len(ids):
        if xp is _Th and not grad and len(ids) <= 3000:   # few cells: numpy has the shorter call
            xp, rows, left, step, ids = _Np, *(v.cpu().numpy() for v in (rows, left, step, ids))
        h = xp.minimum(step, left)
        ok, small, new = _attempt(xp, p, rows, h)
        rows = xp.where(ok, new, rows)
        left = xp.where(ok, xp.where(h == left, 0.0 * left, left - h), left)
        step = xp.where(ok, xp.where(small, 2.0 * h, h), 0.5 * h)
        fin = left <= 0
        if bool(fin.any()):
            keep = ~fin
            for v, to in ((ids, out_i), (rows, out_r)):
                v = v[..., fin]
                to.append(v if xp is _Th else torch.as_tensor(v, device=DEV))
            rows, left, step, ids = rows[:, keep], left[keep], step[keep], ids[keep]
    return out_i, out_r


def _rates(xp, T, case_b):
    """Rate fits of the paper's appendix and their T-derivatives."""
    r = {}
    lnT = xp.log(T)
    q = xp.sqrt(T / 1e5)
    u = 1.0 / (1.0 + q)
    du = -0.5 * q * u / T                       # d ln u / dT

    def cen(A, T0, T1=0.5):
        v = A * xp.exp(T1 * lnT - T0 / T) * u
        return v, v * (T1 / T + du + T0 / (T * T))

    def hg(A, T1, e, l0, b, s, tt=0):
        w = xp.exp(b * (math.log(T1 / l0) - lnT))
        v = A * xp.exp(e * (math.log(T1) - lnT) + tt * lnT) * (1.0 + w) ** (-s)
        return v, v * (tt - e + s * b * w / (1.0 + w)) / T

    def power(A, T1, e, tt=0):
        v = A * xp.exp(e * (math.log(T1) - lnT) + tt * lnT)
        return v, v * (tt - e) / T

    r["bHI"], r["bHeI"], r["bHeII"] = cen(5.85e-11, 157809.1), cen(2.38e-11, 285335.4), cen(5.68e-12, 631515.0)
    if case_b:
        r["aHII"] = hg(2.753e-14, 315614.0, 1.5, 2.74, 0.407, 2.242)
        r["aHeII"], r["eHeII"] = power(1.26e-14, 570670.0, 0.75), power(K_B * 1.26e-14, 570670.0, 0.75, 1)
        r["aHeIII"] = hg(5.506e-14, 1263030.0, 1.5, 2.74, 0.407, 2.242)
        r["eHII"] = hg(3.435e-30, 315614.0, 1.97, 2.25, 0.376, 3.72, 1)
        r["eHeIII"] = hg(8 * 3.435e-30, 1263030.0, 1.97, 2.25, 0.376, 3.72, 1)
    else:
        r["aHII"] = hg(1.269e-13, 315614.0, 1.503, 0.522, 0.47, 1.923)
        r["aHeII"], r["eHeII"] = power(3e-14, 570670.0, 0.654), power(K_B * 3e-14, 570670.0, 0.654, 1)
        r["aHeIII"] = hg(2.538e-13, 1263030.0, 1.503, 0.522, 0.47, 1.923)
        r["eHII"] = hg(1.778e-29, 315614.0, 1.965, 0.541, 0.502, 2.697, 1)
        r["eHeIII"] = hg(8 * 1.778e-29, 1263030.0, 1.965, 0.541, 0.502, 2.697, 1)
    r["zHI"], r["zHeI"], r["zHeII"] = cen(1.27e-21, 157809.1), cen(9.38e-22, 285335.4), cen(4.95e-22, 631515.0)
    r["pHI"], r["pHeII"] = cen(7.5e-19, 118348.0, 0.0), cen(5.54e-17, 473638.0, -0.397)
    r["ff"] = (1.42e-27 * xp.sqrt(T), 0.5 * 1.42e-27 * xp.sqrt(T) / T)
    e1, e2 = 1.24e-13 * xp.exp(-1.5 * lnT - 470000.0 / T), 0.3 * xp.exp(-94000.0 / T)
    r["diel"] = (e1 * (1.0 + e2), e1 * (1.0 + e2) * (-1.5 / T + 470000.0 / (T * T)) + e1 * e2 * 94000.0 / (T * T))
    return r


def _attempt(xp, p, rows, h):
    """One sub-step over h of every cell (App. A): (10% rule kept, all changes
    below 5%, new rows)."""
    G, X, cr = p["G"], p["X"], p["cr"]
    nH, x, y2, y3, T = rows[0], rows[1], rows[2], rows[3], rows[4]
    he = (1.0 - X) / (4.0 * X)
    nHe = he * nH
    nHI, nHII, nHeI, nHeII, nHeIII = nH * (1.0 - x), nH * x, nHe * (1.0 - y2 - y3), nHe * y2, nHe * y3
    ne = nHII + (y2 + 2.0 * y3) * nHe

    def mu_of(x, y2, y3):
        return 1.0 / (X * (1.0 + x) + 0.25 * (1.0 - X) * (1.0 + y2 + 2.0 * y3))

    changes, firsts = [], []
    crec = [0.0] * G
    if not p["otsa"]:
        ra, rb = _rates(xp, T, False), _rates(xp, T, True)
        for j, (k, n) in enumerate((("aHII", nHII), ("aHeII", nHeII), ("aHeIII", nHeIII))):
            crec[min(j, G - 1)] = crec[min(j, G - 1)] + (ra[k][0] - rb[k][0]) * n * ne
    Nn, Fs, gam, heat = [], [], [0.0, 0.0, 0.0], 0.0
    for i in range(G):
        N = rows[5 + i]
        sn, se = p["sigN"][i], p["sigE"][i]
        inv = 1.0 / (1.0 + h * (cr * (sn[0] * nHI + sn[1] * nHeI + sn[2] * nHeII)))
        n1 = (N + h * crec[i]) * inv
        changes.append(abs(n1 - N) / xp.least(N, 1e-30))
        Nn.append(n1)
        Fs.append(rows[5 + G + i] * inv)
        for j, n in enumerate((nHI, nHeI, nHeII)):
            gam[j] = gam[j] + sn[j] * cr * n1
            heat = heat + n * (cr * n1 * (p["egy"][i] * se[j] - EPS[j] * sn[j]))
    mu = mu_of(x, y2, y3)
    Tmu = T / mu
    case_b = p["otsa"]
    if p["isothermal"]:
        Tmu1 = Tmu
    else:
        r = _rates(xp, T, case_b)
        Tg = 2.727
        comp = 1.017e-37 * Tg ** 4

        def total(k):
            return ne * ((r["zHI"][k] + r["pHI"][k]) * nHI + r["zHeI"][k] * nHeI
                         + (r["zHeII"][k] + r["pHeII"][k] + r["eHeII"][k] + r["diel"][k]) * nHeII
                         + r["eHII"][k] * nHII + r["eHeIII"][k] * nHeIII
                         + r["ff"][k] * (nHII + nHeII + 4.0 * nHeIII) + (comp * (T - Tg) if k == 0 else comp))

        K = (2.0 / 3.0) * X / (nH * K_B)
        lam = heat - total(0)
        dT = lam * K * h / (1.0 + mu * total(1) * K * h)
        Tmu1 = Tmu + dT
        changes.append(abs(dT) / Tmu)
        firsts.append(abs(K * lam * h) / Tmu)
    T1 = T if p["isothermal"] else Tmu1 * mu
    r = _rates(xp, T1, case_b)
    b, db, a, da = r["bHI"][0], r["bHI"][1], r["aHII"][0], r["aHII"][1]
    C, D = b * ne + gam[0], a * ne
    dC, dD = nH * b, nH * a
    if not p["isothermal"]:
        f = ne * Tmu1 * mu * mu * X
        dC, dD = dC - f * db, dD - f * da
    J = dC - (C + D) - x * (dC + dD)
    xdot = C - x * (C + D)
    x1 = xp.most(xp.least(x + h * xdot / (1.0 - J * h), 1e-6), 1.0)
    changes.append(abs(x1 - x) / xp.least(x, 1e-6))
    firsts.append(abs(xdot) * h / xp.least(x, 1e-6))
    z2, z3 = y2, y3
    if X < 1.0:
        yI = 1.0 - y2 - y3
        ne2 = x1 * nH + (y2 + 2.0 * y3) * nHe
        r = _rates(xp, T if p["isothermal"] else Tmu1 * mu_of(x1, y2, y3), case_b)
        yI1 = (yI + y2 * r["aHeII"][0] * ne2 * h) / (1.0 + (r["bHeI"][0] * ne2 + gam[1]) * h)
        C2 = yI1 * (r["bHeI"][0] * ne2 + gam[1]) + y3 * r["aHeIII"][0] * ne2
        z2 = (y2 + C2 * h) / (1.0 + ((r["bHeII"][0] + r["aHeII"][0]) * ne2 + gam[2]) * h)
        ne3 = x1 * nH + (z2 + 2.0 * y3) * nHe
        r = _rates(xp, T if p["isothermal"] else Tmu1 * mu_of(x1, z2, y3), case_b)
        z3 = (y3 + z2 * (r["bHeII"][0] * ne3 + gam[2]) * h) / (1.0 + r["aHeIII"][0] * ne3 * h)
        two = (z2 >= yI1) & (z2 >= z3)
        three = ~two & (z3 >= yI1) & (z3 > z2)
        z2, z3 = xp.where(two, 1.0 - yI1 - z3, z2), xp.where(three, 1.0 - yI1 - z2, z3)
        z2, z3 = xp.most(xp.least(z2, 0.0), 1.0), xp.most(xp.least(z3, 0.0), 1.0)
    ne1 = x1 * nH + (z2 + 2.0 * z3) * nHe
    changes.append(abs(ne1 - ne) / xp.where(ne > 1e-6 * nH, ne, 1e-6 * nH))
    Tn = T if p["isothermal"] else xp.least(Tmu1 * mu_of(x1, z2, z3), 1.0)
    ok = changes[0] <= 0.1
    small = changes[0] < 0.05
    for v in changes[1:]:
        ok, small = ok & (v <= 0.1), small & (v < 0.05)
    for v in firsts:
        ok = ok & (v <= 0.1)
    return ok, small, xp.stack([nH, x1, z2, z3, Tn] + Nn + Fs)
