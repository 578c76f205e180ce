"""Performance cases of the coupled electrohydrodynamic lattice step.

Each case is a run that a user of the library makes through its public binding
(``paper_1712_08494_gb300.lbeh``): load a state, advance it, read the fields
back.  ``listed()`` names the ones that stand for the workloads of this
repository (its tests and its benchmark); ``draw()`` gives others of the same
ranges.  Inputs are made on the GPU from the seed alone.  ``exact()`` is the
model of arXiv:1712.08494, Sec. II, written in plain torch in 64 bits.

A case is a dict of plain values:
  kind    "drop", "slab", "flat", "suspension", "coated", "batch", "adjoint",
          "restart"
  nx,ny,nz (or n)  box;  prec  "fp64" | "fp32" | "bf16" | "fp16" (population storage)
  steps   coupled timesteps of one pass
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_1712_08494_gb300 as pkg

DEV = "cuda"
NXYZ = ("nx", "ny", "nz")


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the plain method at its own size (a validation run): 32^3 in FP64, two slabs, one fixed charged
        # sphere; tens of thousands of sites, so launches, barriers and latency are all there is
        dict(name="slab32_fp64", kind="slab", n=32, prec="fp64", steps=10),
        # flat interfaces of the paper's Sec. III.A: quasi one-dimensional, FP64, selective solvation
        dict(name="flat512x4x4_fp64", kind="flat", nx=512, ny=4, nz=4, prec="fp64", dmu=1.0, chi=0.5, steps=10),
        # one small droplet by itself (the reduced copy of the droplet workload the tests run)
        dict(name="drop64_fp32", kind="drop", nx=64, ny=64, nz=64, prec="fp32", dmu=0.0, steps=10),
        # a box whose axes are no power of two and differ, one of them odd: what a user picks by geometry
        dict(name="drop120x105x90_fp32", kind="drop", nx=120, ny=105, nz=90, prec="fp32", dmu=0.0, steps=10),
        # the benchmark's droplet
        dict(name="drop128_fp32", kind="drop", nx=128, ny=128, nz=128, prec="fp32", dmu=0.0, steps=10),
        # the same with BF16 population storage
        dict(name="drop128_bf16", kind="drop", nx=128, ny=128, nz=128, prec="bf16", dmu=0.0, steps=10),
        # the largest run: a charged drop of the paper's Sec. III.D with selective solvation
        dict(name="drop384_fp32", kind="drop", nx=384, ny=384, nz=384, prec="fp32", dmu=4.0, steps=5),
        # electrophoresis: 200 moving charged spheres in one fluid
        dict(name="suspension256_fp32", kind="suspension", n=256, ncoll=200, r=6.0, prec="fp32", steps=4),
        # a drop coated by 80 moving spheres, two fluids (Sec. III.G)
        dict(name="coated128_fp32", kind="coated", n=128, ncoll=80, r=5.0, prec="fp32", steps=5),
        # a parameter sweep: 96 independent charged drops of uneven size in one launch
        dict(name="batch96_fp32", kind="batch", nbox=96, emin=32, emax=64, prec="fp32", steps=20),
        # gradients of the drop's deformation through the coupled steps
        dict(name="adjoint96_fp32", kind="adjoint", n=96, prec="fp32", steps=20, every=10),
        # a run taken up from a checkpoint in pinned host memory, advanced, observed and written back
        dict(name="restart128_fp32", kind="restart", n=128, prec="fp32", steps=4),
    ]


def _smooth(lo, hi):
    """Lengths of the range whose factors are 2, 3, 5 and 7, odd ones among them."""
    out = []
    for v in range(lo, hi + 1):
        m = v
        for f in (2, 3, 5, 7):
            while m % f == 0:
                m //= f
        if m == 1:
            out.append(v)
    return out


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["drop", "drop", "drop", "drop", "suspension", "suspension", "coated", "flat", "batch", "adjoint", "restart"])
    if kind == "drop":
        axes = _smooth(24, 320)
        while True:
            at = [_log_int(rng, 24, 320) for _ in range(3)]
            nx, ny, nz = (min(axes, key=lambda v: abs(v - t)) for t in at)
            if nx * ny * nz <= 300 ** 3 and max(nx, ny, nz) <= 6 * min(nx, ny, nz):
                break
        prec = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16", "fp64"])
        if prec == "fp64" and (max(nx, ny, nz) > 256 or nx * ny * nz > 128 ** 3):
            prec = "fp32"
        dmu = rng.choice([0.0, 0.0, 1.0, 4.0])
        steps = 10 if nx * ny * nz < 160 ** 3 else 5
        return dict(kind="drop", nx=nx, ny=ny, nz=nz, prec=prec, dmu=dmu, steps=steps)
    if kind == "suspension":
        n = 8 * _log_int(rng, 6, 26)
        r = rng.choice([4.0, 5.0, 6.0])
        share = rng.uniform(0.005, 0.04)  # of the volume
        ncoll = max(1, int(share * n ** 3 / (4.0 / 3.0 * math.pi * r ** 3)))
        return dict(kind="suspension", n=n, ncoll=min(ncoll, 400), r=r, prec=rng.choice(["fp32", "fp32", "bf16"]), steps=4)
    if kind == "coated":
        n = 8 * rng.randint(8, 18)
        return dict(kind="coated", n=n, ncoll=rng.randint(8, max(9, n * n // 260)), r=5.0, prec="fp32", steps=5)
    if kind == "flat":
        return dict(kind="flat", nx=32 * rng.randint(4, 16), ny=4, nz=rng.choice([4, 6, 8]), prec=rng.choice(["fp64", "fp32"]),
                    dmu=rng.choice([1.0, 2.0, 3.0]), chi=rng.choice([0.0, 0.5]), steps=10)
    if kind == "batch":
        return dict(kind="batch", nbox=_log_int(rng, 6, 80), emin=32, emax=8 * rng.randint(5, 8), prec="fp32", steps=10)
    if kind == "adjoint":
        n = 8 * rng.randint(4, 12)
        return dict(kind="adjoint", n=n, prec="fp32", steps=rng.randint(4, 16), every=rng.choice([4, 8]))
    return dict(kind="restart", n=8 * rng.randint(5, 18), prec="fp32", steps=rng.randint(1, 6))


# ---------------------------------------------------------------- parameters and inputs
def _params(case, nx, ny, nz, **kw):
    p = dict(nx=nx, ny=ny, nz=nz, ncomp=2, nions=2, prec=case["prec"], tau=1.0, G=4.0, rho0_shift=(0.04, 0.04), D=0.05,
             bjerrum=0.4, eps_r=(1.0, 0.5), eps_r_colloid=0.125, dmu=(0.0, 0.0), drho_a=0.66, E_ext=(0.0, 0.0, 1e-3),
             poisson_tol=1e-6, poisson_max_iter=50, ncolloid_max=0, rho_p=5.0, k_hertz=1.0, psi_subdiv=3, colloids_move=0,
             poisson_solver="auto")
    p.update(kw)
    return SimpleNamespace(**p)


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _noise(shape, gen):
    return 1.0 + 0.01 * (2.0 * torch.rand(shape, generator=gen, device=DEV, dtype=torch.float64) - 1.0)


def _grid(p):
    return torch.meshgrid(*(torch.arange(k, device=DEV, dtype=torch.float64) for k in (p.nz, p.ny, p.nx)), indexing="ij")


def _two_fluids(inside, gen):
    """Fluid a (0.7) outside, fluid b (0.7) inside, 0.04 of the other, 1% noise."""
    red = torch.where(inside, 0.04, 0.7) * _noise(inside.shape, gen)
    blue = torch.where(inside, 0.7, 0.04) * _noise(inside.shape, gen)
    return torch.stack([red, blue])


def _drop_inputs(p, gen, r, salt=1e-3, charge=0.0):
    z, y, x = _grid(p)
    inside = (x - p.nx / 2.0) ** 2 + (y - p.ny / 2.0) ** 2 + (z - p.nz / 2.0) ** 2 < r * r
    del x, y, z
    rho = _two_fluids(inside, gen)
    n = torch.full((2,) + tuple(inside.shape), salt, device=DEV, dtype=torch.float64)
    if charge:  # Q / V extra cations inside, as many extra anions outside
        n[0][inside] += charge / int(inside.sum())
        n[1][~inside] += charge / int((~inside).sum())
    return rho, n, inside


def _far(p, cx, cr, margin):
    z, y, x = _grid(p)
    far = torch.ones((p.nz, p.ny, p.nx), dtype=torch.bool, device=DEV)
    ax, ay, az = x[0, 0], y[0, :, 0], z[:, 0, 0]

    def d2(v, c, n):
        d = (v - c).abs()
        d = torch.minimum(d, n - d)
        return d * d
    for c, r in zip(cx, cr):
        far &= (d2(az, c[2], p.nz)[:, None, None] + d2(ay, c[1], p.ny)[None, :, None] + d2(ax, c[0], p.nx)) > (r + margin) ** 2
    return far


def _place(rng, n, count, gap):
    """Centres at least `gap` apart (periodic), as many as fit in a bounded number of tries."""
    got = np.zeros((0, 3))
    for _ in range(200 * count):
        c = rng.uniform(0.0, float(n), size=3)
        d = np.abs(got - c)
        d = np.minimum(d, n - d)
        if len(got) == 0 or (d * d).sum(1).min() >= gap * gap:
            got = np.vstack([got, c])
            if len(got) == count:
                break
    return got


def _inputs(case, seed):
    """(params, fields in 64 bits, what else the kind needs)."""
    gen, rng, k = _gen(seed), np.random.default_rng(int(seed)), case["kind"]
    if k == "drop":
        nx, ny, nz = (case[a] for a in NXYZ)
        eps = (1.0, 1.0) if case["dmu"] else (1.0, 0.5)
        p = _params(case, nx, ny, nz, dmu=(case["dmu"], -case["dmu"]), eps_r=eps,
                    poisson_tol=1e-10 if case["prec"] == "fp64" else 1e-6)
        rho, n, _ = _drop_inputs(p, gen, 0.1875 * min(nx, ny, nz))
        return p, dict(rho=rho, n=n), {}
    if k == "slab":
        m = case["n"]
        p = _params(case, m, m, m, E_ext=(0.0, 0.0, 0.0), poisson_tol=1e-10, poisson_max_iter=200, ncolloid_max=1)
        z, _, _ = _grid(p)
        rho = _two_fluids(z >= m // 2, gen)
        n = torch.full((2, m, m, m), 0.01, device=DEV, dtype=torch.float64)
        cx, cr = np.array([[m / 2.0, m / 2.0, m / 2.0 - 0.5]]), np.array([4.0])
        far = _far(p, cx, cr, 2.0)
        n[0][far] += 20.0 / int(far.sum())
        return p, dict(rho=rho, n=n), dict(x=cx, v=np.zeros_like(cx), q=np.array([-20.0]), r=cr)
    if k == "flat":
        nx, ny, nz = (case[a] for a in NXYZ)
        dmu, chi = case["dmu"], case["chi"]
        p = _params(case, nx, ny, nz, dmu=(dmu, -dmu), eps_r=(1.0, (1.0 - chi) / (1.0 + chi)), E_ext=(0.0, 0.0, 0.0),
                    poisson_tol=1e-7, poisson_max_iter=200)
        _, _, x = _grid(p)
        noise = 1.0 + 0.001 * torch.rand((nx,), generator=gen, device=DEV, dtype=torch.float64)  # a function of x alone
        red = torch.where(x < nx // 2, 0.7, 0.04) * noise
        blue = torch.where(x < nx // 2, 0.04, 0.7) * noise
        n = torch.full((2, nz, ny, nx), 1e-3, device=DEV, dtype=torch.float64)
        return p, dict(rho=torch.stack([red, blue]), n=n), {}
    if k == "suspension":
        m, r = case["n"], case["r"]
        cx = _place(rng, m, case["ncoll"], 2 * r + 2.0)
        nc = len(cx)
        cq, cr = rng.uniform(-40.0, -10.0, size=nc), np.full(nc, r)
        p = _params(case, m, m, m, ncomp=1, G=0.0, eps_r=(1.0, 1.0), E_ext=(1e-3, 0.0, 0.0), ncolloid_max=nc, colloids_move=1,
                    rho0_shift=(1.0, 0.0))
        n = torch.full((2, m, m, m), 1e-3, device=DEV, dtype=torch.float64)
        far = _far(p, cx, cr, 2.0)
        n[0][far] += float(-cq.sum()) / int(far.sum())
        rho = torch.ones((1, m, m, m), device=DEV, dtype=torch.float64)
        return p, dict(rho=rho, n=n), dict(x=cx, v=np.zeros_like(cx), q=cq, r=cr)
    if k == "coated":
        m, nc, r = case["n"], case["ncoll"], case["r"]
        p = _params(case, m, m, m, eps_r=(1.0, 1.0), dmu=(4.0, -4.0), ncolloid_max=nc, colloids_move=1)
        rd = m / 4.0
        rho, n, _ = _drop_inputs(p, gen, rd)
        t = np.arange(nc) + 0.5  # a Fibonacci lattice on the drop's surface
        polar, azim = np.arccos(1.0 - 2.0 * t / nc), math.pi * (1.0 + math.sqrt(5.0)) * t
        cx = m / 2.0 + rd * np.stack([np.cos(azim) * np.sin(polar), np.sin(azim) * np.sin(polar), np.cos(polar)], axis=1)
        return p, dict(rho=rho, n=n), dict(x=cx, v=np.zeros_like(cx), q=np.zeros(nc), r=np.full(nc, r))
    if k == "adjoint":
        m = case["n"]
        p = _params(case, m, m, m, E_ext=(0.0, 0.0, 1.5e-3))
        rho, n, inside = _drop_inputs(p, gen, 0.1875 * m, charge=50.0)
        dn = torch.stack([inside / inside.sum(), ~inside / (~inside).sum()]).to(torch.float64)
        return p, dict(rho=rho, n=n), dict(dn=dn)
    # restart: a smooth drop, its ions and the potential that goes with them
    m = case["n"]
    p = _params(case, m, m, m)
    z, y, x = _grid(p)
    c = m / 2.0
    s = 0.5 * (1.0 + torch.tanh((torch.sqrt((x - c) ** 2 + (y - c) ** 2 + (z - c) ** 2) - 0.1875 * m) / 2.0))
    rho = torch.stack([0.04 + 0.66 * s, 0.7 - 0.66 * s]) * _noise((2, m, m, m), gen)
    n = 1e-3 * _noise((2, m, m, m), gen)
    rho, n = rho.float().double(), n.float().double()  # a checkpoint in 32 bits
    phi = _poisson(n[0] - n[1], _eps(p, rho), p.E_ext, 1e-6).float().double()
    return p, dict(rho=rho, n=n, phi=phi), {}


def _batch(case, seed):
    rng, out = np.random.default_rng(int(seed)), []
    for b in range(case["nbox"]):
        # every edge of the range appears equally often, so that another seed is other drops and not another amount of work
        edges = list(range(case["emin"], case["emax"] + 1, 8))
        e = edges[b % len(edges)]
        p = _params(case, e, e, e, E_ext=(0.0, 0.0, float(rng.uniform(0.0, 2e-3))))
        rho, n, _ = _drop_inputs(p, _gen(1000 * int(seed) + b), 0.3 * e, charge=float(rng.uniform(0.0, 200.0)))
        out.append((p, rho, n))
    return out


# ---------------------------------------------------------------- prepare / run
def _read(lbeh, keep, handle, rho, n, phi, u=None, host=False):
    """The fields a run hands on, into the caller's buffers."""
    fl = lbeh.lbeh_fields()
    fl.dtype, fl.on_device = (lbeh.LBEH_F64 if phi.dtype == torch.float64 else lbeh.LBEH_F32), 0 if host else 1
    for s in range(rho.shape[0]):
        fl.rho[s] = rho[s].data_ptr()
    for s in range(2):
        fl.n[s] = n[s].data_ptr()
    fl.phi = phi.data_ptr()
    if u is not None:
        fl.u = u.data_ptr()
    if keep:  # colloid tables are host arrays
        for k in ("cx", "cv"):
            setattr(fl, k, keep[k].ctypes.data_as(lbeh.C.POINTER(lbeh.C.c_double)))
    lbeh.lbeh_get_fields(handle, fl)


def _reads_u(case):
    # velocities are read where the storage resolves them: not from 16-bit populations, and not from a
    # suspension at rest, where the run's results are its spheres' positions and velocities
    return case["kind"] not in ("suspension", "adjoint", "batch") and case["prec"] in ("fp32", "fp64")


def prepare(case, seed):
    lbeh = pkg.load()
    st = SimpleNamespace(case=case, lbeh=lbeh)
    dt = _dtype(case)
    if case["kind"] == "batch":
        boxes = _batch(case, seed)
        st.batch = lbeh.Batch([p for p, _, _ in boxes])
        total = sum(p.nx * p.ny * p.nz for p, _, _ in boxes)
        st.rho, st.n, st.phi = (torch.empty((k * total,), device=DEV, dtype=dt) for k in (2, 2, 1))
        st.views, at = [], 0
        for box, (p, rho, n) in zip(st.batch.boxes, boxes):
            box.set_fields(rho=list(rho.to(dt)), n=list(n.to(dt)))
            m = p.nx * p.ny * p.nz
            st.views.append((st.rho[2 * at:2 * (at + m)].view(2, m), st.n[2 * at:2 * (at + m)].view(2, m), st.phi[at:at + m]))
            at += m
        return st
    p, f, more = _inputs(case, seed)
    shape = (p.nz, p.ny, p.nx)
    st.sys = lbeh.System(p)
    st.keep = {}
    col = {}
    if "x" in more:
        col = dict(colloid_x=more["x"], colloid_v=more["v"], colloid_q=more["q"], colloid_r=more["r"])
        st.keep = dict(cx=np.zeros_like(more["x"]), cv=np.zeros_like(more["x"]))
    if case["kind"] == "restart":
        st.host = {k: v.to(dt).cpu().pin_memory() for k, v in f.items()}
        st.out = {k: torch.empty(s, dtype=dt).pin_memory() for k, s in
                  dict(rho=(2,) + shape, n=(2,) + shape, phi=shape, u=(3,) + shape).items()}
        return st
    st.sys.set_fields(rho=list(f["rho"].to(dt)), n=list(f["n"].to(dt)), **col)
    if case["kind"] == "adjoint":
        st.dn = more["dn"].contiguous()
        st.f0 = torch.empty((2, 19) + shape, device=DEV, dtype=torch.float64)
        st.n0 = torch.empty((2,) + shape, device=DEV, dtype=torch.float64)
        return st
    st.out = dict(rho=torch.empty((p.ncomp,) + shape, device=DEV, dtype=dt), n=torch.empty((2,) + shape, device=DEV, dtype=dt),
                  phi=torch.empty(shape, device=DEV, dtype=dt))
    if _reads_u(case):
        st.out["u"] = torch.empty((3,) + shape, device=DEV, dtype=dt)
    return st


def run(st):
    case, lbeh = st.case, st.lbeh
    kind = case["kind"]
    if kind == "batch":
        st.batch.step(case["steps"])
        for box, (rho, n, phi) in zip(st.batch.boxes, st.views):
            _read(lbeh, None, box.h, rho, n, phi)
        return dict(rho=st.rho, n=st.n, phi=st.phi)
    if kind == "adjoint":
        seed, g = lbeh.lbeh_obs_seed(), lbeh.lbeh_grads()
        seed.d_deformation = 1.0
        g.on_device = 1
        g.dn0_dQ, g.f0_bar, g.n0_bar = st.dn.data_ptr(), st.f0.data_ptr(), st.n0.data_ptr()
        lbeh.lbeh_step_adjoint(st.sys.h, case["steps"], case["every"], seed, g)
        # the state's gradients in the precision they are computed in; the value and its parameter gradients as one vector
        return dict(f0=st.f0.float(), n0=st.n0.float(),
                    value_and_grad=np.array([g.deformation, *g.dE_ext[:], g.dG, g.dQ], dtype=np.float32))
    if kind == "restart":
        h = st.host
        st.sys.set_fields(rho=list(h["rho"]), n=list(h["n"]), phi=h["phi"])
        st.sys.step(case["steps"])
        o = st.sys.observables()
        _read(lbeh, None, st.sys.h, host=True, **st.out)
        return dict(st.out, sums=np.array([*o.mass[:], *o.ions[:]], dtype=np.float32))
    st.sys.step(case["steps"])
    _read(lbeh, st.keep, st.sys.h, **st.out)
    if st.keep:
        return dict(st.out, **{k: v.astype(np.float64 if case["prec"] == "fp64" else np.float32) for k, v in st.keep.items()})
    return st.out


# ---------------------------------------------------------------- work
def work(case):
    """One pass: every step reads and writes the populations, the ions and the potential once (a step is a global
    dependence: the potential of all sites enters every site), the read-out writes its fields once."""
    if case["kind"] == "batch":
        edges = list(range(case["emin"], case["emax"] + 1, 8))
        N = sum(edges[b % len(edges)] ** 3 for b in range(case["nbox"]))
    elif "n" in case:
        N = case["n"] ** 3
    else:
        N = case["nx"] * case["ny"] * case["nz"]
    e = 8 if case["prec"] == "fp64" else 4
    s = {"fp64": 8, "fp32": 4}.get(case["prec"], 2)
    nc = 1 if case["kind"] == "suspension" else 2
    state = 2 * (19 * nc * s + 2 * e + e)
    out = (nc + 2 + 1 + (3 if _reads_u(case) else 0)) * e
    # per site and step: 19 equilibria of ~20 operations a component, ~400 for fields, forces and fluxes, and a
    # potential solve of a few dozen seven-point stencils
    flops = 19 * 20 * nc + 400 + 30 * 20
    if case["kind"] == "adjoint":  # forward, recompute and reverse; the gradients once
        return dict(bytes=N * (4 * case["steps"] * state + (38 + 2) * 8), flops=N * case["steps"] * 5 * flops)
    extra = 5 * e if case["kind"] == "restart" else 0
    return dict(bytes=N * (case["steps"] * state + out + extra), flops=N * case["steps"] * flops)


# ---------------------------------------------------------------- the model in 64 bits
_C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
      (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
_AX = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]


def _at(a, c):
    """a(x + c) at x, periodic."""
    return torch.roll(a, shifts=(-c[2], -c[1], -c[0]), dims=(-3, -2, -1))


def _back(a, c):
    return torch.roll(a, shifts=(c[2], c[1], c[0]), dims=(-3, -2, -1))


def _eps(p, rho, psi_s=None):
    ref = 1.0 / (4.0 * math.pi * p.bjerrum)
    a, b = rho[0], rho[1] if len(rho) > 1 else torch.zeros_like(rho[0])
    tot = a + b
    c = torch.where(tot > 0, (b - a) / torch.where(tot > 0, tot, 1.0), 0.0)
    f = 0.5 * ref * (p.eps_r[0] * (1.0 - c) + p.eps_r[1] * (1.0 + c))
    return f if psi_s is None else psi_s * p.eps_r_colloid * ref + (1.0 - psi_s) * f


def _poisson(q, eps, E_ext, tol, phi=None):
    """sum_d eps_{i+d/2} (phi_{i+d} - phi_i) = -(q - mean q) + div_h(eps E_ext), mean-free, by conjugate gradients with
    the constant-coefficient Fourier inverse as preconditioner."""
    k = [0.5 * (eps + _at(eps, a)) for a in _AX]

    def A(v):
        out = torch.zeros_like(v)
        for a, ka in zip(_AX, k):
            fl = ka * (_at(v, a) - v)
            out += fl - _back(fl, a)
        return out
    nz, ny, nx = q.shape
    sym = [2.0 - 2.0 * torch.cos(2.0 * math.pi * torch.arange(n, device=q.device, dtype=torch.float64) / n) for n in (nz, ny, nx)]
    lam = -(sym[0][:, None, None] + sym[1][None, :, None] + sym[2][None, None, :nx // 2 + 1]) * float(eps.mean())
    lam[0, 0, 0] = 1.0

    def M(v):
        t = torch.fft.rfftn(v) / lam
        t[0, 0, 0] = 0.0
        return torch.fft.irfftn(t, s=v.shape)
    b = -(q - q.mean())
    for a, ka, e in zip(_AX, k, E_ext):
        if e:
            b = b + e * (ka - _back(ka, a))
    phi = torch.zeros_like(q) if phi is None else phi - phi.mean()
    r = b - A(phi)
    stop = tol * float(b.norm())
    d = rz = None
    for _ in range(200):
        if float(r.norm()) <= stop:
            break
        z = M(r)
        rz, old = float((r * z).sum()), rz
        d = z if d is None else z + (rz / old) * d
        w = A(d)
        al = rz / float((d * w).sum())
        phi = phi + al * d
        r = r - al * w
    return phi - phi.mean()


def _sphere(p, cx, cr, cq):
    """Solid mask, solid fraction, surface nodes and surface charge of one sphere away from the box's faces."""
    z, y, x = _grid(p)

    def d2(ox, oy, oz):
        return (x + ox - cx[0]) ** 2 + (y + oy - cx[1]) ** 2 + (z + oz - cx[2]) ** 2
    solid = d2(0.0, 0.0, 0.0) < cr * cr
    h = p.psi_subdiv + 1
    off = [(i + 0.5) / h - 0.5 for i in range(h)]
    frac = sum((d2(a, b, c) < cr * cr).double() for a in off for b in off for c in off) / h ** 3
    near = torch.zeros_like(solid)
    for c in _C[1:]:
        near |= ~_at(solid, c)
    surf = solid & near
    return solid, frac, surf, surf.double() * (cq / int(surf.sum()))


def _model(p, f64, steps, sphere=None, rounded=None):
    """`steps` coupled timesteps of Sec. II from rest; a sphere, where there is one, is fixed."""
    rnd = (lambda v: v) if rounded is None else (lambda v: v.to(rounded).double())
    rho0, n, phi = rnd(f64["rho"]), rnd(f64["n"]), f64.get("phi")
    ns = len(rho0)
    fluid = psi_s = None
    qc = 0.0
    if sphere is not None:
        solid, psi_s, surf, qc = sphere
        fluid = (~solid).double()
        rho0, n = rho0 * fluid, n * fluid
    f = [[_W[q] * rho0[s] for q in range(19)] for s in range(ns)]
    ref = 1.0 / (4.0 * math.pi * p.bjerrum)
    bar = 0.5 * (p.eps_r[0] + p.eps_r[1]) * ref
    dmd = [d / p.drho_a for d in p.dmu]
    one = 1.0 if fluid is None else fluid
    for _ in range(steps):
        rho = [sum(f[s][1:], f[s][0]) for s in range(ns)]
        J = []
        for a in range(3):
            J.append(sum(c[a] * sum(f[s][q] for s in range(ns)) for q, c in enumerate(_C) if c[a]))
        rv = rho
        if fluid is not None:  # interface solid nodes carry the mean of their fluid neighbours
            cnt = sum(_at(fluid, c) for c in _C[1:])
            rv = [torch.where(surf, sum(_at(r, c) for c in _C[1:]) / cnt.clamp(min=1.0), r) for r in rho]
        eps = _eps(p, rv, psi_s)
        phi = _poisson(n[0] - n[1] + qc, eps, p.E_ext, 1e-13, phi)
        E = [0.5 * (_back(phi, a) - _at(phi, a)) + e for a, e in zip(_AX, p.E_ext)]
        # ion fluxes through the faces i + a/2, and their friction on the fluid
        pf = None if psi_s is None else torch.where(solid, 0.0, 1.0 - psi_s)
        nt = n if pf is None else torch.where(pf > 0, n / torch.where(pf > 0, pf, 1.0), 0.0)
        F = []
        for s, zs in ((0, 1.0), (1, -1.0)):
            F.append([])
            for a, ax in enumerate(_AX):
                nj = _at(nt[s], ax)
                nb = 0.5 * (nt[s] + nj)
                g = (nj - nt[s]) - zs * nb * 0.5 * (E[a] + _at(E[a], ax))
                if dmd[s]:
                    g = g - dmd[s] * nb * (_at(rho[0], ax) - rho[0])
                F[s].append(p.D * g if pf is None else p.D * pf * _at(pf, ax) * g)
        E2 = E[0] ** 2 + E[1] ** 2 + E[2] ** 2
        tot = sum(rho)
        inv = torch.where(tot > 0, 1.0 / torch.where(tot > 0, tot, 1.0), 0.0)
        Phi = [[None] * 3 for _ in range(ns)]
        psi = [-torch.expm1(-r) for r in rv]

        def gsum(v, a):
            return sum(_W[q] * c[a] * _at(v, c) for q, c in enumerate(_C) if c[a])
        for a, ax in enumerate(_AX):
            fel = 0.25 * (eps - bar) * (_at(E2, ax) - _back(E2, ax))
            fel = fel - sum(F[s][a] + _back(F[s][a], ax) for s in range(2)) / (2.0 * p.D)
            for s in range(ns):
                Phi[s][a] = rho[s] * inv * fel
                if ns == 2 and p.G:
                    Phi[s][a] = Phi[s][a] - p.G * psi[s] * gsum(psi[1 - s], a)
            for s in range(2):
                if dmd[s]:
                    Phi[0][a] = Phi[0][a] - 3.0 * dmd[s] * psi[0] * gsum(n[s], a)
            for s in range(ns):
                Phi[s][a] = Phi[s][a] * one
        u = [(J[a] + 0.5 * sum(Phi[s][a] for s in range(ns))) * inv * one for a in range(3)]
        new = []
        for s in range(2):
            v = n[s].clone()
            for a, ax in enumerate(_AX):
                v += F[s][a] - _back(F[s][a], ax)
                for sg in (1, -1):
                    c = tuple(sg * k for k in ax)
                    amt = torch.clamp(sg * u[a], min=0.0) * n[s]
                    if fluid is not None:
                        amt = amt * fluid * _at(fluid, c)
                    v += _back(amt, c) - amt
            new.append(v * one)
        n = torch.stack(new)
        del new, F, E, E2, psi
        for s in range(ns):
            ue = [J[a] * inv + torch.where(rho[s] > 0, p.tau * Phi[s][a] / torch.where(rho[s] > 0, rho[s], 1.0), 0.0) for a in range(3)]
            usq = ue[0] ** 2 + ue[1] ** 2 + ue[2] ** 2
            out = [None] * 19
            back = [0.0] * 19
            for q, c in enumerate(_C):
                cu = sum(c[a] * ue[a] for a in range(3) if c[a]) if q else 0.0
                feq = _W[q] * rho[s] * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
                post = f[s][q] + (feq - f[s][q]) / p.tau
                if fluid is None:
                    out[q] = _back(post, c)
                else:
                    to = _at(fluid, c)
                    out[q] = _back(post * fluid * to, c)
                    if q:  # half-way bounce-back off the fixed sphere
                        back[_C.index((-c[0], -c[1], -c[2]))] = post * fluid * (1.0 - to)
            f[s] = [(out[q] + back[q]) * one for q in range(19)]
    rho = torch.stack([sum(f[s][1:], f[s][0]) for s in range(ns)])
    return dict(rho=rho, n=n, phi=phi, u=torch.stack(u))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("suspension", "coated", "adjoint"):
        # spheres that move and are projected anew each step, and the reverse sweep through all steps: in plain torch these
        # take minutes
        return None
    if kind == "batch":
        got = [_model(p, dict(rho=rho, n=n), case["steps"], rounded=torch.float32) for p, rho, n in _batch(case, seed)]
        return {k: torch.cat([g[k].reshape(-1) for g in got]) for k in ("rho", "n", "phi")}
    p, f, more = _inputs(case, seed)
    sphere = _sphere(p, more["x"][0], float(more["r"][0]), float(more["q"][0])) if "x" in more else None
    got = _model(p, f, case["steps"], sphere, rounded=None if case["prec"] == "fp64" else torch.float32)
    if not _reads_u(case):
        del got["u"]
    if kind == "slab":
        got.update(cx=more["x"], cv=more["v"])
    if kind == "restart":
        got["sums"] = torch.cat([got["rho"].sum((1, 2, 3)), got["n"].sum((1, 2, 3))])
    return got
