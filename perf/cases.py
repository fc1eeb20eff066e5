"""Measured workloads of the library, through its public Python entry points.

Each case is one unit of the work a user's program repeats: an RK step of a
patch (wave, MHD, CCZ4), of a batch of AMR patches, of a level of patches that
exchange ghosts, of a sub-cycled pair of levels, of a puncture box with
radiative boundaries, or the gradient of an observer misfit.  Sizes are those
of the repository's benchmark and tests, and ragged ones in between.

`exact` evaluates the same passes in 64 bits with torch alone: it shares no
code with the library, only the equations and the input fields.
"""
from __future__ import annotations

import math

import torch

from paper_1806_04182_gb300 import adjoint, amr, capi, inputs
from paper_1806_04182_gb300.state import PatchState

G = 3  # ghost points
PREC = {"fp64": capi.SF_FP64, "fp32": capi.SF_FP32_BULK, "fp32dw": capi.SF_FP32_BULK_DW}
SYS = {"wave": capi.SF_WAVE, "mhd": capi.SF_MHD, "z4": capi.SF_Z4}
NF = {"wave": 5, "mhd": 8, "z4": 25}
# add + mul + div per cell and right-hand side
FLOPS = {"wave": 160.0, "mhd": 5600.0, "z4": 7800.0}
Z4_ONE = (0, 1, 4, 6, 18)  # fields whose flat value is 1


def listed():
    return [
        # smallest patch of an AMR hierarchy (16^3 is the smallest patch of the batched
        # benchmark), stepped on its own: latency and launches
        dict(name="wave_16_fp32", kind="wave", nx=16, ny=16, nz=16, precision="fp32", steps=1),
        # the wave benchmark: 64^3 FP64
        dict(name="wave_64_fp64", kind="wave", nx=64, ny=64, nz=64, precision="fp64", steps=1),
        # the headline: CCZ4 96^3 robust-stability data, FP32 bulk, benchmark layout
        dict(name="ccz4_96_fp32dw", kind="z4", nx=96, ny=96, nz=96, precision="fp32dw",
             layout="benchmark", data="noise", lopsided=0, steps=1),
        # the same evolution in FP64
        dict(name="ccz4_96_fp64", kind="z4", nx=96, ny=96, nz=96, precision="fp64", layout="dense",
             data="noise", lopsided=0, steps=1),
        # a patch of odd size as PatchState lays it out when told nothing about rows
        dict(name="ccz4_61x47x53_fp32dw_dense", kind="z4", nx=61, ny=47, nz=53, precision="fp32dw",
             layout="dense", data="smooth", lopsided=0, steps=1),
        # the MHD benchmark: 128^3 blast, WENO5-JS, SSP-RK3, CFL 0.3, FP64 and FP32
        dict(name="mhd_128_fp64", kind="mhd", nx=128, ny=128, nz=128, precision="fp64", weno=0,
             split=0, steps=1),
        dict(name="mhd_128_fp32", kind="mhd", nx=128, ny=128, nz=128, precision="fp32", weno=0,
             split=0, steps=1),
        # one RK4 step of a batch of mixed wave and CCZ4 patches of uneven sizes, tuned, as a graph
        dict(name="amr_batch_96", kind="batch", npatch=96, lo=16, hi=64, table=0, precision="fp32dw"),
        # one RK4 step of a level: the 96^3 CCZ4 box as 2 x 2 x 2 patches with halo exchange, as a graph
        dict(name="level_8x48", kind="level", bx=2, by=2, bz=2, nx=48, ny=48, nz=48,
             precision="fp32dw"),
        # one coarse step of a two-level CCZ4 hierarchy, ratio 2, sub-cycled, as a graph
        dict(name="subcycled_64_64", kind="subcycled", nc=64, nf=64, at=16, ratio=2,
             precision="fp32dw"),
        # gradient of the observer misfit (forward, recomputation and adjoint steps): the adjoint
        # benchmark's box and observers over fewer steps
        dict(name="adjoint_128_fp32", kind="adjoint", nx=128, ny=128, nz=128, precision="fp32",
             nsteps=12, every=4, nobs=64),
        # a moving, spinning puncture with radiative boundaries and its constraint monitors
        dict(name="puncture_96_fp32dw", kind="puncture", nx=96, ny=96, nz=96, precision="fp32dw",
             layout="rows16"),
    ]


def draw(rng):
    """A case of the listed ranges: sizes uniform in the logarithm, odd ones among them."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):
        return dict(nx=size(lo, hi), ny=size(lo, hi), nz=size(lo, hi))

    kind = rng.choice(["wave", "wave", "z4", "z4", "z4", "mhd", "mhd", "mhd", "batch", "level",
                       "subcycled", "adjoint", "puncture"])
    if kind == "wave":
        return dict(kind=kind, **box(16, 128), precision=rng.choice(["fp64", "fp32"]), steps=rng.choice([1, 4]))
    if kind == "z4":
        precision = rng.choice(["fp32dw", "fp32dw", "fp32", "fp64"])
        layout = "dense" if precision == "fp64" else rng.choice(["dense", "rows16", "pairs", "benchmark"])
        lop = 1 if layout == "dense" and rng.random() < 0.25 else 0
        b = box(16, 96)
        return dict(kind=kind, **b, precision=precision, layout=layout,
                    data=rng.choice(["noise", "smooth"]), lopsided=lop, steps=1)
    if kind == "mhd":
        return dict(kind=kind, **box(16, 128), precision=rng.choice(["fp64", "fp32"]),
                    weno=rng.choice([0, 0, 1, 2]), split=rng.choice([0, 0, 0, 1]), steps=1)
    if kind == "batch":
        lo = rng.choice([16, 20, 24])
        precision = rng.choice(["fp32dw", "fp32dw", "fp64"])
        return dict(kind=kind, npatch=size(8, 32 if precision == "fp64" else 96), lo=lo,
                    hi=rng.randint(lo + 8, 64), table=rng.randrange(1000), precision=precision)
    if kind == "level":
        return dict(kind=kind, bx=rng.randint(1, 3), by=rng.randint(1, 2), bz=2, **box(16, 48),
                    precision="fp32dw")
    if kind == "subcycled":
        nc = rng.choice([32, 40, 48, 56, 64])
        nf = 2 * rng.randint(12, nc // 2 - 4)
        return dict(kind=kind, nc=nc, nf=nf, at=rng.randint(3, nc - nf // 2 - 3), ratio=2,
                    precision=rng.choice(["fp32dw", "fp32dw", "fp64"]))
    if kind == "adjoint":
        n = rng.randint(6, 12)
        return dict(kind=kind, **box(24, 128), precision=rng.choice(["fp32", "fp64"]), nsteps=n,
                    every=rng.randint(2, n), nobs=rng.choice([16, 64]))
    return dict(kind=kind, **box(32, 96), precision="fp32dw", layout=rng.choice(["rows16", "pairs", "dense"]))


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _axes(n, dx, x0=(0.0, 0.0, 0.0)):
    x, y, z = (x0[d] + dx[d] * torch.arange(n[d], device="cuda", dtype=torch.float64) for d in range(3))
    return x[None, None, :], y[None, :, None], z[:, None, None]


def _n(case):
    return case["nx"], case["ny"], case["nz"]


def _wave_data(n, length, seed):
    """A right-moving plane wave, integer wave vector in {1,2,3}^3 and phase from the seed."""
    g = _gen(seed)
    k = (1 + torch.floor(3 * _rand(g, 3))).tolist()
    p0 = _rand(g, 1).item()
    dx = tuple(length / v for v in n)
    x, y, z = _axes(n, dx)
    ph = 2 * math.pi * ((k[0] * x + k[1] * y + k[2] * z) / length + p0)
    c = torch.cos(ph) * (2 * math.pi / length)
    kn = math.sqrt(sum(v * v for v in k))
    return torch.stack([torch.sin(ph), kn * c, k[0] * c, k[1] * c, k[2] * c]), dx


def _z4_data(n, data, seed):
    """Flat space plus uniform noise of amplitude 1e-10 (robust stability), or plus three smooth
    Fourier modes of amplitude 0.01 in every field.  Deviations from flat space."""
    g = _gen(seed)
    if data == "noise":
        return 1e-10 * (2 * _rand(g, 25, n[2], n[1], n[0]) - 1)
    U = torch.zeros(25, n[2], n[1], n[0], device="cuda", dtype=torch.float64)
    x, y, z = _axes(n, tuple(1.0 / v for v in n))
    r = _rand(g, 25, 3, 4).tolist()
    for f in range(25):
        for m in r[f]:
            kx, ky, kz = (1 + int(2 * v) for v in m[:3])
            U[f] += 0.01 / 3 * torch.sin(2 * math.pi * (kx * x + ky * y + kz * z + m[3]))
    return U


def _ones(nf):
    one = torch.zeros(nf, 1, 1, 1, device="cuda", dtype=torch.float64)
    if nf == 25:
        one[list(Z4_ONE)] = 1.0
    return one


def _mhd_data(n, seed):
    """rho = 1, p = 0.1, B = (0.5, 0.5, 0), Gaussian velocities of rms 0.1, and a sphere of
    radius 0.1 at 10 times the pressure around a centre from the seed."""
    g = _gen(seed)
    dx = tuple(1.0 / v for v in n)
    v = torch.randn(3, n[2], n[1], n[0], generator=g, device="cuda", dtype=torch.float64) * (0.1 / math.sqrt(3))
    c = _rand(g, 3).tolist()
    d2 = 0.0
    for a, cc in zip(_axes(n, dx), c):
        d = (a - cc).abs()
        d2 = d2 + torch.minimum(d, 1 - d) ** 2
    p = torch.where(d2 < 0.01, 1.0, 0.1).to(torch.float64)
    one = torch.ones_like(p)
    E = 0.5 * (v * v).sum(0) + p / (GAMMA - 1) + 0.25
    return torch.stack([one, v[0], v[1], v[2], E, 0.5 * one, 0.5 * one, 0 * one]), dx


def _puncture_data(n, seed):
    """Brill-Lindquist conformal factor and Bowen-York curvature of one hole near the centre of a
    cell-centred box of side 16, its momentum and spin from the seed; ghost points included."""
    r_ = (2 * _rand(_gen(seed), 6) - 1).tolist()
    P, S = [0.1 * v for v in r_[:3]], [0.2 * v for v in r_[3:]]
    dx = tuple(16.0 / v for v in n)
    x0 = tuple(-8.0 + 0.5 * h for h in dx)
    x, y, z = _axes(tuple(v + 2 * G for v in n), dx, tuple(a - G * h for a, h in zip(x0, dx)))
    rel = (x - 0.05 + 0 * (y + z), y + 0.03 + 0 * (x + z), z - 0.02 + 0 * (x + y))
    r = torch.sqrt(rel[0] ** 2 + rel[1] ** 2 + rel[2] ** 2)
    nv = [c / r for c in rel]
    psi = 1 + 0.5 / r
    Pn = sum(P[d] * nv[d] for d in range(3))
    Sxn = [S[(d + 1) % 3] * nv[(d + 2) % 3] - S[(d + 2) % 3] * nv[(d + 1) % 3] for d in range(3)]
    U = torch.zeros((25,) + r.shape, device="cuda", dtype=torch.float64)
    U[0], U[18] = psi ** -4, psi ** -2
    U[1] = U[4] = U[6] = 1.0
    for q, (i, j) in enumerate(SYM):
        lin = P[i] * nv[j] + P[j] * nv[i] - ((1.0 if i == j else 0.0) - nv[i] * nv[j]) * Pn
        U[8 + q] = (1.5 / r ** 2 * lin + 3 / r ** 3 * (Sxn[i] * nv[j] + Sxn[j] * nv[i])) / psi ** 6
    return U, dx, x0


def _layout(name, nx):
    if name == "benchmark":
        return dict(x_pitch=104, x_offset=1, plane_rows=102)
    if name == "pairs":
        return dict(x_pitch=(nx + 7 + 3) // 4 * 4, x_offset=1)
    if name == "rows16":
        return dict(x_pitch=(nx + 6 + 3) // 4 * 4)
    return {}


# ------------------------------------------------------------------ prepare / run
class _Batch:
    """A batch handle that is given back with the state that holds it."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        capi.sf_batch_destroy(self.handle)


def _captured(handle, tune):
    """Tune and capture on a stream of its own (capture needs one)."""
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    if tune:
        capi.sf_batch_tune(handle, s.cuda_stream)
    capi.sf_batch_capture(handle, s.cuda_stream)
    torch.cuda.current_stream().wait_stream(s)


def _table(case):
    return inputs.amr_patch_table(case["npatch"], seed=case["table"], lo=case["lo"], hi=case["hi"])


def _table_data(t, seed):
    """(system name, field values, dx) of one entry of a batch table."""
    if t["system"] == "wave":
        U, dx = _wave_data(t["n"], 1.0, seed)
        h = t["dx"]  # same phases, the patch's own spacing
        return "wave", torch.cat([U[:1], U[1:] / (t["n"][0] * h)]), (h, h, h)
    return "z4", _z4_data(t["n"], "noise", seed) + _ones(25), (t["dx"],) * 3


def _adjoint_data(case, seed):
    """Initial phi and Pi of a plane wave, distinct observers, and what they recorded: the wave a
    little out of phase, sampled after each step."""
    n, g = _n(case), _gen(seed + 1)
    U, dx = _wave_data(n, 1.0, seed)
    dt, dtype = 0.25 * min(dx), torch.float64 if case["precision"] == "fp64" else torch.float32
    obs = torch.randperm(n[0] * n[1] * n[2], generator=g, device="cuda")[:case["nobs"]]
    phi, rate = U[0].reshape(-1)[obs], -U[1].reshape(-1)[obs]
    t = 0.05 + dt * torch.arange(1, case["nsteps"] + 1, device="cuda", dtype=torch.float64)[:, None]
    w = U[1].abs().max()  # angular frequency of unit amplitude
    ref = phi * torch.cos(w * t) + rate / w * torch.sin(w * t)
    return U[0].to(dtype), U[1].to(dtype), obs, ref.to(dtype), dx, dt


def _subcycled_states(case, seed):
    nc, nf, R = (case["nc"],) * 3, (case["nf"],) * 3, case["ratio"]
    dxc = (1.0 / case["nc"],) * 3
    return nc, nf, dxc, _z4_data(nc, "noise", seed), _z4_data(nf, "noise", seed + 77777), R


def prepare(case, seed):
    kind, prec = case["kind"], PREC[case["precision"]]
    if kind == "wave":
        U, dx = _wave_data(_n(case), 1.0, seed)
        st = PatchState(capi.SF_WAVE, _n(case), dx, 0.25 * min(dx), precision=prec)
        st.upload(U)
        return dict(kind=kind, st=st, steps=case["steps"])
    if kind == "z4":
        n = _n(case)
        dx = tuple(1.0 / v for v in n)
        st = PatchState(capi.SF_Z4, n, dx, 0.25 * min(dx), precision=prec,
                        prm=capi.params(lopsided=case["lopsided"]), **_layout(case["layout"], n[0]))
        st.upload(_z4_data(n, case["data"], seed) + _ones(25))
        return dict(kind=kind, st=st, steps=case["steps"])
    if kind == "mhd":
        U, dx = _mhd_data(_n(case), seed)
        st = PatchState(capi.SF_MHD, _n(case), dx, 1e-3, precision=prec,
                        prm=capi.params(rk=capi.SF_SSPRK3, weno_variant=case["weno"], flux_split=case["split"]))
        st.upload(U)
        return dict(kind=kind, st=st, steps=case["steps"])
    if kind == "batch":
        sts = []
        for q, t in enumerate(_table(case)):
            name, U, dx = _table_data(t, seed * 1000 + q)
            lay = _layout("pairs", t["n"][0]) if name == "z4" and prec != capi.SF_FP64 else {}
            sts.append(PatchState(SYS[name], t["n"], dx, t["dt"], precision=prec, **lay))
            sts[-1].upload(U)
        b = _Batch(capi.sf_batch_create(capi.params(), [s.patch(s.B, s.A, s.C) for s in sts]))
        _captured(b.handle, True)
        return dict(kind=kind, sts=sts, batch=b)
    if kind == "level":
        n, nb = _n(case), (case["bx"], case["by"], case["bz"])
        N = tuple(a * b for a, b in zip(n, nb))
        dx = tuple(1.0 / v for v in N)
        U = _z4_data(N, "noise", seed) + _ones(25)
        grid = {}
        for c in range(nb[2]):
            for b in range(nb[1]):
                for a in range(nb[0]):
                    st = PatchState(capi.SF_Z4, n, dx, 0.25 * min(dx), precision=prec,
                                    prm=capi.params(ghosts=capi.SF_GHOSTS_NONE), **_layout("pairs", n[0]))
                    st.upload(U[:, c * n[2]:(c + 1) * n[2], b * n[1]:(b + 1) * n[1], a * n[0]:(a + 1) * n[0]])
                    grid[(a, b, c)] = st
        batch = _Batch(amr.level_batch(grid))
        capi.sf_copy_boxes(amr.halo_boxes(grid, "A"), prec, torch.cuda.current_stream().cuda_stream)
        _captured(batch.handle, False)
        return dict(kind=kind, sts=list(grid.values()), batch=batch)
    if kind == "subcycled":
        nc, nf, dxc, Uc, Uf, R = _subcycled_states(case, seed)
        lay = _layout("benchmark", 0) if prec != capi.SF_FP64 else {}
        coarse = PatchState(capi.SF_Z4, nc, dxc, 0.25 * dxc[0], precision=prec, **lay)
        fine = PatchState(capi.SF_Z4, nf, tuple(v / R for v in dxc), 0.25 * dxc[0] / R, precision=prec,
                          prm=capi.params(ghosts=capi.SF_GHOSTS_NONE), **lay)
        pair = amr.SubcycledPair(coarse, fine, R, (case["at"],) * 3)
        for go in (lambda: pair.step(1), lambda: pair.capture(1), lambda: None):
            coarse.upload(Uc + _ones(25))
            fine.upload(Uf + _ones(25))
            go()
        return dict(kind=kind, pair=pair)
    if kind == "adjoint":
        phi, Pi, obs, ref, dx, dt = _adjoint_data(case, seed)
        return dict(kind=kind, phi=phi.requires_grad_(True), Pi=Pi.requires_grad_(True), obs=obs, ref=ref,
                    dx=dx, dt=dt, nsteps=case["nsteps"], prec=prec, every=case["every"])
    if kind == "puncture":
        U, dx, x0 = _puncture_data(_n(case), seed)
        st = PatchState(capi.SF_Z4, _n(case), dx, 0.25 * min(dx), precision=prec,
                        prm=capi.params(ghosts=capi.SF_GHOSTS_NONE), **_layout(case["layout"], case["nx"]))
        st.upload_ghosted(U)
        return dict(kind=kind, st=st, x0=x0, speed=[1.0] * 25)
    raise ValueError(kind)


def run(state):
    kind = state["kind"]
    if kind in ("wave", "z4"):
        state["st"].step(state["steps"])
        return {"u": state["st"].interior()}
    if kind == "mhd":
        rates = state["st"].step_cfl(state["steps"], cfl=0.3)
        return {"u": state["st"].interior(), "rates": rates}
    if kind in ("batch", "level"):
        capi.sf_batch_launch(state["batch"].handle, torch.cuda.current_stream().cuda_stream)
        sts = state["sts"]
        if kind == "level":
            return {"u": [s.interior() for s in sts]}
        # every patch's state, in at most 64 outputs
        groups = [sts[q::48] for q in range(min(48, len(sts)))]
        return {"u": [torch.cat([s.interior().reshape(-1) for s in g]) if len(g) > 1 else g[0].interior().reshape(-1)
                      for g in groups]}
    if kind == "subcycled":
        state["pair"].replay()
        return {"coarse": state["pair"].coarse.interior(), "fine": state["pair"].fine.interior()}
    if kind == "adjoint":
        phi, Pi = state["phi"], state["Pi"]
        phi.grad = Pi.grad = None
        J = adjoint.misfit(phi, Pi, state["obs"], state["ref"], state["dx"], state["dt"], state["nsteps"],
                           precision=state["prec"], checkpoint_every=state["every"])
        J.backward()
        return {"J": J, "dphi": phi.grad, "dPi": Pi.grad}
    st = state["st"]
    st.step_radiative(1, state["x0"], inputs.Z4_UINF, state["speed"])
    return {"u": st.A[:, :, :st.n[1] + 2 * G, st.xo:st.xo + st.n[0] + 2 * G], "monitors": st.diagnostics()[:4]}


def work(case):
    """State read once and written once per pass (with the compensation of FP32 RK4 steps), and the
    right-hand sides' operations."""
    kind, es = case["kind"], 8 if case["precision"] == "fp64" else 4

    def step(system, cells, stages=4):
        arrays = 4 if es == 4 and system != "mhd" else 2
        return cells * NF[system] * es * arrays, cells * stages * FLOPS[system]

    if kind in ("wave", "z4"):
        b, f = step(kind, case["nx"] * case["ny"] * case["nz"])
        return dict(bytes=b, flops=f * case["steps"])
    if kind == "mhd":
        b, f = step("mhd", case["nx"] * case["ny"] * case["nz"], 3)
        return dict(bytes=b, flops=f * case["steps"])
    if kind == "batch":
        parts = [step(t["system"], t["n"][0] * t["n"][1] * t["n"][2]) for t in _table(case)]
    elif kind == "level":
        parts = [step("z4", case["nx"] * case["ny"] * case["nz"] * case["bx"] * case["by"] * case["bz"])]
    elif kind == "subcycled":
        b, f = step("z4", case["nf"] ** 3)
        parts = [step("z4", case["nc"] ** 3), (b, case["ratio"] * f)]
    elif kind == "adjoint":
        cells = case["nx"] * case["ny"] * case["nz"]
        parts = [(4 * cells * es, cells * 4 * FLOPS["wave"] * 3 * case["nsteps"])]
    else:
        parts = [step("z4", (case["nx"] + 2 * G) * (case["ny"] + 2 * G) * (case["nz"] + 2 * G))]
    return dict(bytes=sum(p[0] for p in parts), flops=sum(p[1] for p in parts))


# ------------------------------------------------------------------ the same in 64 bits
GAMMA = 5.0 / 3.0
SIGMA = 0.1
SYM = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
SIDX = [[0, 1, 2], [1, 3, 4], [2, 4, 5]]


def _wrap(u):
    """Periodic ghost shell of (nf, nz, ny, nx)."""
    for d in (1, 2, 3):
        n = u.shape[d]
        u = u.index_select(d, torch.arange(-G, n + G, device=u.device) % n)
    return u


def _at(g, ox=0, oy=0, oz=0):
    """The interior of a ghosted array, shifted."""
    z, y, x = g.shape[-3:]
    return g[..., G + oz:z - G + oz, G + oy:y - G + oy, G + ox:x - G + ox]


def _sh(g, d, o):
    return _at(g, **{("ox", "oy", "oz")[d]: o})


def _D(g, d, h):
    return ((_sh(g, d, -2) - _sh(g, d, 2)) + 8 * (_sh(g, d, 1) - _sh(g, d, -1))) / (12 * h)


def _DD(g, d, h):
    return (16 * (_sh(g, d, -1) + _sh(g, d, 1)) - (_sh(g, d, -2) + _sh(g, d, 2)) - 30 * _at(g)) / (12 * h * h)


def _DX(g, a, b, ha, hb):
    w = {-2: 1.0, -1: -8.0, 1: 8.0, 2: -1.0}
    names = ("ox", "oy", "oz")
    return sum(wa * wb * _at(g, **{names[a]: oa, names[b]: ob})
               for oa, wa in w.items() for ob, wb in w.items()) / (144 * ha * hb)


def _KO(g, dx):
    return sum(SIGMA / (64 * dx[d]) * ((_sh(g, d, -3) + _sh(g, d, 3)) - 6 * (_sh(g, d, -2) + _sh(g, d, 2))
                                       + 15 * (_sh(g, d, -1) + _sh(g, d, 1)) - 20 * _at(g)) for d in range(3))


def _wave_rhs(g, dx):
    r = torch.stack([-_at(g)[1], -(_D(g[2], 0, dx[0]) + _D(g[3], 1, dx[1]) + _D(g[4], 2, dx[2])),
                     -_D(g[1], 0, dx[0]), -_D(g[1], 1, dx[1]), -_D(g[1], 2, dx[2])])
    return r + _KO(g, dx)


def _z4_rhs(g, dx, lop=0):
    """CCZ4 (Sec. V) from deviations `g` from flat space: 1+log slicing, Gamma-driver, kappa = 1,
    eta = 2, g = 3/4."""
    c = _at(g)
    one = _ones(25)
    v = c + one
    chi, Kh, Th, al = v[0], v[7], v[17], v[18]
    Gh, be, B = v[14:17], v[19:22], v[22:25]

    def mat(s):
        return torch.stack([torch.stack([s[SIDX[i][j]] for j in range(3)]) for i in range(3)])

    gt, At = mat(v[1:7]), mat(v[8:14])
    d1 = torch.stack([_D(g, d, dx[d]) for d in range(3)])  # [d, field]
    ko = _KO(g, dx)
    if lop:
        adv = 0.0
        for d in range(3):
            fwd = (_sh(g, d, 3) - 6 * _sh(g, d, 2) + 18 * _sh(g, d, 1) - 10 * c - 3 * _sh(g, d, -1)) / (12 * dx[d])
            bwd = (-_sh(g, d, -3) + 6 * _sh(g, d, -2) - 18 * _sh(g, d, -1) + 10 * c + 3 * _sh(g, d, 1)) / (12 * dx[d])
            adv = adv + be[d] * torch.where(be[d] > 0, fwd, torch.where(be[d] < 0, bwd, d1[d]))
    else:
        adv = (be[:, None] * d1).sum(0)

    def hess(f):
        h = [[None] * 3 for _ in range(3)]
        for a in range(3):
            h[a][a] = _DD(g[f], a, dx[a])
            for b in range(a + 1, 3):
                h[a][b] = h[b][a] = _DX(g[f], a, b, dx[a], dx[b])
        return torch.stack([torch.stack(r) for r in h])

    E = torch.einsum
    cof = torch.stack([torch.stack([gt[(i + 1) % 3, (j + 1) % 3] * gt[(i + 2) % 3, (j + 2) % 3]
                                    - gt[(i + 1) % 3, (j + 2) % 3] * gt[(i + 2) % 3, (j + 1) % 3]
                                    for j in range(3)]) for i in range(3)])
    det = (gt[0] * cof[0]).sum(0)
    ig = cof / det

    def tr(X):
        return E("ijzyx,ijzyx->zyx", ig, X)

    trA = tr(At)
    K = Kh + 2 * Th
    dbe = d1[:, 19:22].transpose(0, 1)  # [i, d] = d_d beta^i
    div = dbe[0, 0] + dbe[1, 1] + dbe[2, 2]
    dg = torch.stack([mat(d1[d, 1:7]) for d in range(3)])  # [d, i, j]
    lie = lambda X: E("ikzyx,kjzyx->ijzyx", X, dbe) + E("jkzyx,kizyx->ijzyx", X, dbe) - 2 / 3 * X * div  # noqa: E731
    rg = lie(gt) - 2 * al * (At - gt * trA / 3) - al * gt * torch.log(det) / 3
    Gl = 0.5 * (E("bpczyx->pbczyx", dg) + E("cpbzyx->pbczyx", dg) - dg)
    Gu = E("plzyx,lbczyx->pbczyx", ig, Gl)
    Gt = E("bczyx,pbczyx->pzyx", ig, Gu)
    Z = 0.5 * chi * (Gh - Gt)
    dchi, dal, dK, dTh = d1[:, 0], d1[:, 18], d1[:, 7], d1[:, 17]
    hchi, hal = hess(0), hess(18)
    dGh = d1[:, 14:17].transpose(0, 1)  # [c, d]
    R = torch.zeros_like(gt)
    for q, (i, j) in enumerate(SYM):
        R[i, j] = R[j, i] = -0.5 * tr(hess(1 + q))
    sGh = E("cazyx,cbzyx->abzyx", gt, dGh)
    R = R + 0.5 * (sGh + sGh.transpose(0, 1))
    GlG = E("czyx,abczyx->abzyx", Gh, Gl)
    R = R + 0.5 * (GlG + GlG.transpose(0, 1))
    Q = E("nmzyx,cmpzyx->cpnzyx", ig, Gu)
    t = E("cpnzyx,bcnzyx->pbzyx", Q, Gl)
    R = R + t + t.transpose(0, 1) + E("cpnzyx,cnbzyx->pbzyx", Q, Gl)
    trchi = tr(hchi) - 1.5 / chi * E("cmzyx,czyx,mzyx->zyx", ig, dchi, dchi) - (Gh * dchi).sum(0)
    Zl = E("cpzyx,czyx->pzyx", gt, Z)
    Zd = Zl[:, None] * dchi[None]
    R = R + 0.5 / chi * (hchi - E("cabzyx,czyx->abzyx", Gu, dchi)) - 0.25 / chi ** 2 * dchi[:, None] * dchi[None]
    R = R + (Zd + Zd.transpose(0, 1)) / chi ** 2 + 0.5 / chi * gt * trchi
    RZ = chi * tr(R)
    gda = E("cmzyx,czyx,mzyx->zyx", ig, dal, dchi)
    dadc = dal[:, None] * dchi[None]
    DDa = hal - E("cabzyx,czyx->abzyx", Gu, dal) + 0.5 / chi * (dadc + dadc.transpose(0, 1) - gt * gda)
    M = al * R - DDa
    Aud = E("aczyx,cbzyx->abzyx", ig, At)
    Auu = E("aczyx,bczyx->abzyx", Aud, ig)
    AAd = E("aczyx,cbzyx->abzyx", At, Aud)
    AA = tr(AAd)
    Zda = (Z * dal).sum(0)
    up = lambda X, w: E("abzyx,bzyx->azyx", X, w)  # noqa: E731
    hb = torch.stack([hess(19 + i) for i in range(3)])  # [i, m, n]
    rGh = (E("mnzyx,imnzyx->izyx", ig, hb) + up(ig, E("kmkzyx->mzyx", hb)) / 3
           - E("kzyx,ikzyx->izyx", Gh, dbe) + 2 / 3 * Gh * div - 2 * up(Auu, dal)
           + 2 * al * (E("pabzyx,abzyx->pzyx", Gu, Auu) - 1.5 / chi * up(Auu, dchi))
           - 2 * Th * up(ig, dal) - 4 / 3 * al * up(ig, dK) - 2 / 3 * al * up(ig, dTh)
           - 2 * al / chi * Z * (1 + 2 / 3 * K))
    rA = lie(At) - al * gt * trA / 3 + chi * (M - gt * tr(M) / 3) + al * (Kh * At - 2 * AAd)
    r = torch.empty_like(c)
    r[0] = 2 / 3 * chi * (al * K - div)
    for q, (i, j) in enumerate(SYM):
        r[1 + q], r[8 + q] = rg[i, j], rA[i, j]
    r[7] = -chi * tr(DDa) + al * (K * K / 3 + AA + Th) + 2 * Zda
    r[14:17] = rGh
    r[17] = -Zda + 0.5 * al * (RZ + 2 / 3 * Kh * Kh + 2 / 3 * Th * (Kh - 2 * Th) - AA) - 2 * al * Th
    r[18] = -2 * al * Kh
    r[19:22] = 0.75 * B
    r[22:25] = rGh - 2 * B
    return r + adv + ko


def _rk4(u, rhs, dt):
    """One RK4 step of interior `u`; also the stage inputs and increments."""
    k, s = [], [u]
    for c in (0.5, 0.5, 1.0):
        k.append(dt * rhs(s[-1]))
        s.append(u + c * k[-1])
    k.append(dt * rhs(s[-1]))
    return u + (k[0] + 2 * k[1] + 2 * k[2] + k[3]) / 6, s, k


def _stored(U, case):
    """Field deviations as the arrays of the case's precision hold them, in 64 bits."""
    return U if case["precision"] == "fp64" else U.float().double()


def _mhd_flux(q, d):
    rho, S, E, B = q[0], q[1:4], q[4], q[5:8]
    v = S / rho
    B2 = (B * B).sum(0)
    p = (GAMMA - 1) * (E - 0.5 * (S * v).sum(0) - 0.5 * B2)
    pt = p + 0.5 * B2
    F = torch.empty_like(q)
    F[0] = S[d]
    F[1:4] = S[d] * v - B[d] * B
    F[1 + d] += pt
    F[4] = (E + pt) * v[d] - (v * B).sum(0) * B[d]
    F[5:8] = v[d] * B - v * B[d]
    a2, b2, bd2 = GAMMA * p / rho, B2 / rho, B[d] ** 2 / rho
    s = a2 + b2
    return F, v[d].abs() + torch.sqrt(0.5 * (s + torch.sqrt(s * s - 4 * a2 * bd2)))


def _weno(w, eps, weno):
    """Left state at the right edge of the middle of five cells w[0..4]."""
    if weno == 2:
        c = [0.5 * w[2] + 0.5 * w[3], -0.5 * w[1] + 1.5 * w[2]]
        b = [(w[3] - w[2]) ** 2, (w[2] - w[1]) ** 2]
        a = [gk / (eps + bk) ** 2 for gk, bk in zip((2 / 3, 1 / 3), b)]
    else:
        c = [(2 * w[2] + 5 * w[3] - w[4]) / 6, (-w[1] + 5 * w[2] + 2 * w[3]) / 6, (2 * w[0] - 7 * w[1] + 11 * w[2]) / 6]
        b = [13 / 12 * (w[2] - 2 * w[3] + w[4]) ** 2 + 0.25 * (3 * w[2] - 4 * w[3] + w[4]) ** 2,
             13 / 12 * (w[1] - 2 * w[2] + w[3]) ** 2 + 0.25 * (w[1] - w[3]) ** 2,
             13 / 12 * (w[0] - 2 * w[1] + w[2]) ** 2 + 0.25 * (w[0] - 4 * w[1] + 3 * w[2]) ** 2]
        gk = (0.3, 0.6, 0.1)
        if weno == 1:
            tau = (b[0] - b[2]).abs()
            a = [g_ * (1 + (tau / (eps + bk)) ** 2) for g_, bk in zip(gk, b)]
        else:
            a = [g_ / (eps + bk) ** 2 for g_, bk in zip(gk, b)]
    return sum(x * y for x, y in zip(a, c)) / sum(a)


def _mhd_rhs(u, dx, weno, split):
    """Interfaces i - 1/2, i = 0..n, of every direction from the periodic array (nf, nz, ny, nx)."""
    r = torch.zeros_like(u)
    for d in range(3):
        ax = 3 - d
        eps = dx[d] ** (2 if weno == 2 else 4)
        w = [torch.roll(u, 3 - q, ax) for q in range(6)]  # cells i - 3 .. i + 2
        if split:
            f, s = zip(*[_mhd_flux(q, d) for q in w])
            S = torch.stack(s).amax(0)
            F = (_weno([0.5 * (a + S * b) for a, b in zip(f, w)][:5], eps, weno)
                 + _weno([0.5 * (a - S * b) for a, b in zip(f, w)][:0:-1], eps, weno))
        else:
            L, Rr = _weno(w[:5], eps, weno), _weno(w[:0:-1], eps, weno)
            (fl, sl), (fr, sr) = _mhd_flux(L, d), _mhd_flux(Rr, d)
            F = 0.5 * (fl + fr - torch.maximum(sl, sr) * (Rr - L))
        r -= (torch.roll(F, -1, ax) - F) / dx[d]
    return r


def _mhd_rate(u, dx):
    return max((_mhd_flux(u, d)[1] / dx[d]).max().item() for d in range(3))


def _prolong_matrix(nf, nc, at, R):
    """Ghosted fine points (from -G) by ghosted coarse points: 6-point Lagrange interpolation."""
    M = torch.zeros(nf + 2 * G, nc + 2 * G, dtype=torch.float64)
    for i in range(-G, nf + G):
        F = R * at + i
        b, t = F // R, (F % R) / R
        for j in range(-2, 4):
            l = 1.0
            for m in range(-2, 4):
                if m != j:
                    l *= (t - m) / (j - m)
            M[i + G, b + j + G] = l
    return M.cuda()


def _bor_value(u, k, R, r, stage):
    """App. C dense output and App. D: fine stage input `stage` of fine step r from the coarse
    increments k_1..k_4 of one step from u."""
    th, q = r / R, 1.0 / R
    P = [[0, 1, -1.5, 2 / 3], [0, 0, 1, -2 / 3], [0, 0, 1, -2 / 3], [0, 0, -0.5, 2 / 3]]

    def dense(m):  # m-th theta-derivative of sum_j b_j k_j
        return sum(kj * sum(p[e] * math.perm(e, m) * th ** (e - m) for e in range(m, 4)) for p, kj in zip(P, k))

    d0, d1, d2, d3 = (dense(m) for m in range(4))
    vf = 4 * (k[2] - k[1])
    f = [q * d1, q * d1 + q * q / 2 * d2 + q ** 3 / 8 * (d3 - vf), q * d1 + q * q / 2 * d2 + q ** 3 / 8 * (d3 + vf)]
    return u + d0 + (0.0, 0.5 * f[0], 0.5 * f[1], f[2])[stage]


def _rad_rhs(g, dx, x0):
    """-(x^i/r d_i U + (U - U_inf)/r) at every point of a ghosted array of deviations
    from U_inf, one-sided at its edges."""
    z, y, x = g.shape[-3:]
    X, Y, Z = _axes((x, y, z), dx, tuple(a - G * h for a, h in zip(x0, dx)))
    r = torch.sqrt(X * X + Y * Y + Z * Z)
    tot = g / r
    for d, pos in enumerate((X, Y, Z)):
        ax = 3 - d
        n = g.shape[ax]
        at = lambda lo, hi: g.narrow(ax, lo, hi - lo)  # noqa: E731
        mid = ((at(0, n - 4) - at(4, n)) + 8 * (at(3, n - 1) - at(1, n - 3))) / (12 * dx[d])
        p = [at(q, q + 1) for q in range(5)]
        m = [at(n - 1 - q, n - q) for q in range(5)]
        one = lambda s: (-25 * s[0] + 48 * s[1] - 36 * s[2] + 16 * s[3] - 3 * s[4]) / (12 * dx[d])  # noqa: E731
        two = lambda s: (-3 * s[0] - 10 * s[1] + 18 * s[2] - 6 * s[3] + s[4]) / (12 * dx[d])  # noqa: E731
        tot = tot + pos / r * torch.cat([one(p), two(p), mid, -two(m), -one(m)], ax)
    return -tot


def _monitors(g, dx):
    """Sums of Theta^2, |Z|^2, (ln det)^2 and (tr A)^2 of a ghosted array of deviations."""
    v = _at(g) + _ones(25)
    gt = torch.stack([torch.stack([v[1 + SIDX[i][j]] for j in range(3)]) for i in range(3)])
    At = torch.stack([torch.stack([v[8 + SIDX[i][j]] for j in range(3)]) for i in range(3)])
    m = gt.permute(2, 3, 4, 0, 1)
    ig = torch.linalg.inv(m).permute(3, 4, 0, 1, 2)
    dg = torch.stack([torch.stack([torch.stack([_D(g[1 + SIDX[i][j]], d, dx[d]) for j in range(3)])
                                   for i in range(3)]) for d in range(3)])
    E = torch.einsum
    Gl = 0.5 * (E("bpczyx->pbczyx", dg) + E("cpbzyx->pbczyx", dg) - dg)
    Z = 0.5 * v[0] * (v[14:17] - E("bczyx,plzyx,lbczyx->pzyx", ig, ig, Gl))
    ld = torch.log(torch.linalg.det(m))
    trA = E("ijzyx,ijzyx->zyx", ig, At)
    return torch.stack([(v[17] ** 2).sum(), (Z * Z).sum(), (ld * ld).sum(), (trA ** 2).sum()])


def exact(case, seed):
    kind = case["kind"]
    with torch.no_grad() if kind != "adjoint" else torch.enable_grad():
        if kind == "wave":
            u, dx = _wave_data(_n(case), 1.0, seed)
            u = _stored(u, case)
            for _ in range(case["steps"]):
                u = _rk4(u, lambda s: _wave_rhs(_wrap(s), dx), 0.25 * min(dx))[0]
            return {"u": u}
        if kind == "z4":
            n = _n(case)
            dx = tuple(1.0 / v for v in n)
            u = _z4_data(n, case["data"], seed)
            one = _ones(25)
            if case["precision"] == "fp64":
                u = (u + one) - one
            u = _stored(u, case)
            for _ in range(case["steps"]):
                u = _rk4(u, lambda s: _z4_rhs(_wrap(s), dx, case["lopsided"]), 0.25 * min(dx))[0]
            return {"u": u + one if case["precision"] == "fp64" else u}
        if kind == "mhd":
            u, dx = _mhd_data(_n(case), seed)
            u, rates = _stored(u, case), []
            for _ in range(case["steps"]):
                rates.append(_mhd_rate(u, dx))
                dt = 0.3 / rates[-1]
                f = lambda s: s + dt * _mhd_rhs(s, dx, case["weno"], case["split"])  # noqa: E731
                s2 = 0.75 * u + 0.25 * f(f(u))
                u = u / 3 + 2 / 3 * f(s2)
            return {"u": u, "rates": rates}
        if kind == "batch":
            outs = []
            for q, t in enumerate(_table(case)):
                name, U, dx = _table_data(t, seed * 1000 + q)
                if name == "z4":
                    one = _ones(25)
                    u = _stored(U - one, case)
                    u = _rk4(u, lambda s: _z4_rhs(_wrap(s), dx), t["dt"])[0]
                    u = u + one if case["precision"] == "fp64" else u
                else:
                    u = _rk4(_stored(U, case), lambda s: _wave_rhs(_wrap(s), dx), t["dt"])[0]
                outs.append(u.reshape(-1))
            return {"u": [torch.cat(outs[q::48]) for q in range(min(48, len(outs)))]}
        if kind == "level":
            n, nb = _n(case), (case["bx"], case["by"], case["bz"])
            N = tuple(a * b for a, b in zip(n, nb))
            dx = tuple(1.0 / v for v in N)
            u = _stored(_z4_data(N, "noise", seed), case)
            u = _rk4(u, lambda s: _z4_rhs(_wrap(s), dx), 0.25 * min(dx))[0]
            return {"u": [u[:, c * n[2]:(c + 1) * n[2], b * n[1]:(b + 1) * n[1], a * n[0]:(a + 1) * n[0]]
                          for c in range(nb[2]) for b in range(nb[1]) for a in range(nb[0])]}
        if kind == "subcycled":
            nc, nf, dxc, uc, uf, R = _subcycled_states(case, seed)
            one = _ones(25)
            if case["precision"] == "fp64":
                uc, uf = (uc + one) - one, (uf + one) - one
            uc, uf = _stored(uc, case), _stored(uf, case)
            dxf, dt = tuple(v / R for v in dxc), 0.25 * dxc[0]
            new, _, k = _rk4(uc, lambda s: _z4_rhs(_wrap(s), dxc), dt)
            M = _prolong_matrix(nf[0], nc[0], case["at"], R)

            def filled(interior, r, stage):
                c = _wrap(_bor_value(uc, k, R, r, stage))
                f = torch.einsum("kc,jb,ia,fcba->fkji", M, M, M, c)
                f[:, G:-G, G:-G, G:-G] = interior
                return f

            for r in range(R):
                stage = iter(range(4))
                uf = _rk4(uf, lambda s: _z4_rhs(filled(s, r, next(stage)), dxf), dt / R)[0]
            a, e = case["at"], case["nf"] // R
            new[:, a:a + e, a:a + e, a:a + e] = uf[:, ::R, ::R, ::R]
            off = one if case["precision"] == "fp64" else 0.0
            return {"coarse": new + off, "fine": uf + off}
        if kind == "adjoint":
            phi, Pi, obs, ref, dx, dt = _adjoint_data(case, seed)
            phi, Pi = (v.double().requires_grad_(True) for v in (phi, Pi))
            w = _wrap(phi[None])
            u = torch.stack([phi, Pi] + [_D(w[0], d, dx[d]) for d in range(3)])
            J = 0.0
            for q in range(case["nsteps"]):
                u = _rk4(u, lambda v: _wave_rhs(_wrap(v), dx), dt)[0]
                J = J + 0.5 * ((u[0].reshape(-1)[obs] - ref[q].double()) ** 2).sum()
            J.backward()
            return {"J": J.detach(), "dphi": phi.grad, "dPi": Pi.grad}
        U, dx, x0 = _puncture_data(_n(case), seed)
        one = _ones(25)
        g = _stored(U - one, case)
        inner = (slice(None),) + (slice(G, -G),) * 3

        def rhs(s):
            r = _rad_rhs(s, dx, x0)
            r[inner] = _z4_rhs(s, dx)
            return r

        g = _rk4(g, rhs, 0.25 * min(dx))[0]
        return {"u": g, "monitors": _monitors(g, dx)}
