"""The work a user of this package has it do, as measurable cases.

Every case goes through the public entry points (``Solver``, ``Batch``, the
closure and its trainer) the way a program that owns a simulation calls them: a
handle set up once, a call that advances it some steps, the fields, J and
delta f read back on the device.  The initial state is a field in mid-run (smooth, about ten
cells a feature, 1 V/m unless the velocity-space advection is on), so the plasma
is driven everywhere from the first step.  Inputs come from the seed alone and
are made on the GPU; ``exact`` repeats the same steps in plain 64-bit torch.
"""
from __future__ import annotations

import json
import math
import os

import numpy as np
import torch

import paper_2211_05647_gb300 as P
from paper_2211_05647_gb300.fdtd_plasma import QUANTITY, Batch, MlpTrainer, Solver

C0 = 299792458.0
QE = 1.602176634e-19
ME = 9.1093837015e-31
EPS0 = 8.8541878128e-12
ETA0 = 376.730313668
LAM0 = 0.03
F0 = C0 / LAM0
W0 = 2 * math.pi * F0
NC = EPS0 * ME * W0 * W0 / (QE * QE)          # critical density at W0
TAU = 0.96 / F0
SOURCE = dict(kind="gauss_sine", amp=1.0, fc=F0, tau=TAU, t0=4.52 * TAU)
CLOSURE_FILE = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "data", "closure_2d_tmz_cylinder.npz")
VMAX = 6.0


# ------------------------------------------------------------------- the cases
def listed():
    return [
        # A co-simulation that takes one step and looks at the field: launch latency and nothing else.
        dict(name="slab1d_one_step", kind="slab1d", nz=1000, s0=400, s1=700, nv=64, precision="f32", steps=1),
        # The 1-D slab of the benchmark, FP64: a short line stepped many times.
        dict(name="slab1d_f64", kind="slab1d", nz=2000, s0=1000, s1=1500, nv=64, precision="f64", steps=128),
        # A parameter scan: 256 independent lines of 1k to 64k cells, BF16 distributions.
        dict(name="batch1d_256_bf16", kind="batch1d", runs=256, nz_min=1024, nz_max=65536, nv=64, f_dtype="bf16",
             steps=200),
        # A small 2-D study on a desk-top grid: every launch is short.
        dict(name="tmz_192", kind="tmz2d", nx=192, ny=160, r=40, nv=32, nvp=32, f_dtype="f32", nonlinear=0, steps=40),
        # The benchmark's 2-D grid: 823 k plasma cells of 1024 velocity nodes.
        dict(name="tmz_4096", kind="tmz2d", nx=4096, ny=4096, r=512, nv=32, nvp=32, f_dtype="f32", nonlinear=0,
             steps=32),
        # Odd grid and odd velocity grid, BF16 rows: what a convergence study has between the powers of two.
        dict(name="tmz_odd_bf16", kind="tmz2d", nx=1531, ny=1187, r=150, nv=31, nvp=16, f_dtype="bf16", nonlinear=0,
             steps=50),
        # Strong fields: the flux-form velocity-space advection is on.
        dict(name="tmz_nonlinear", kind="tmz2d", nx=512, ny=512, r=128, nv=32, nvp=32, f_dtype="f32", nonlinear=1,
             steps=20),
        # The benchmark's 3-D slab, BF16 rows of 32 nodes.
        dict(name="yee_512_bf16", kind="yee3d", nx=512, ny=512, nz=512, s0=192, s1=320, nv=32, f_dtype="bf16",
             evolve=0, steps=16),
        # Odd 3-D grid with the paper's 31 velocity nodes, FP32 rows.
        dict(name="yee_odd", kind="yee3d", nx=203, ny=117, nz=131, s0=40, s1=90, nv=31, f_dtype="f32", evolve=0,
             steps=25),
        # The isotropic part evolves (heating and elastic collisions) on the speed grid.
        dict(name="yee_256_evolve", kind="yee3d", nx=256, ny=256, nz=256, s0=96, s1=160, nv=32, f_dtype="f32",
             evolve=1, steps=16),
        # The learned closure in place of the velocity-space solve on the largest 2-D grid.
        dict(name="closure_8192", kind="closure", nx=8192, ny=8192, r=1024, steps=20),
        # Training the closure: one epoch of 4096-sample minibatches.
        dict(name="train_epoch", kind="train", n=131072, batch=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["slab1d", "batch1d", "tmz2d", "tmz2d", "yee3d", "yee3d", "closure", "train"])
    if kind == "slab1d":
        nz = _log(rng, 500, 8000)
        s0 = int(nz * rng.uniform(0.2, 0.5))
        return dict(kind=kind, nz=nz, s0=s0, s1=s0 + max(8, int(nz * rng.uniform(0.1, 0.4))),
                    nv=rng.choice([31, 32, 48, 64]), precision=rng.choice(["f32", "f64"]), steps=_log(rng, 1, 200))
    if kind == "batch1d":
        hi = _log(rng, 4096, 65536)
        return dict(kind=kind, runs=_log(rng, 8, 256), nz_min=1024, nz_max=hi, nv=rng.choice([32, 63, 64]),
                    f_dtype=rng.choice(["f32", "bf16"]), steps=_log(rng, 20, 110))
    if kind == "tmz2d":
        nx, ny = _log(rng, 128, 3000), _log(rng, 128, 3000)
        if rng.random() < 0.5:
            nx = (nx + 3) // 4 * 4
        nl = int(rng.random() < 0.25)
        r = min(int(min(nx, ny) * rng.uniform(0.08, 0.3)), 130 if nl else 400)
        return dict(kind=kind, nx=nx, ny=ny, r=r, nv=rng.choice([24, 31, 32]),
                    nvp=rng.choice([16, 20, 32]), f_dtype="f32" if nl else rng.choice(["f32", "bf16"]), nonlinear=nl,
                    steps=_log(rng, 10, 50))
    if kind == "yee3d":
        nx, ny, nz = _log(rng, 64, 300), _log(rng, 64, 300), _log(rng, 64, 300)
        if rng.random() < 0.5:
            nx = (nx + 3) // 4 * 4
        s0 = int(nz * rng.uniform(0.25, 0.4))
        ev = int(rng.random() < 0.3)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, s0=s0, s1=s0 + int(nz * rng.uniform(0.15, 0.35)),
                    nv=rng.choice([31, 32, 64]), f_dtype="f32" if ev else rng.choice(["f32", "bf16"]), evolve=ev,
                    steps=_log(rng, 8, 20))
    if kind == "closure":
        nx, ny = _log(rng, 256, 6000) // 4 * 4, _log(rng, 256, 6000)
        return dict(kind=kind, nx=nx, ny=ny, r=int(min(nx, ny) * rng.uniform(0.1, 0.25)), steps=_log(rng, 10, 20))
    batch = rng.choice([512, 1000, 2048, 4096, 8192])
    return dict(kind=kind, n=batch * _log(rng, 4, 40) + rng.randrange(batch), batch=batch)


# ---------------------------------------------------------------------- inputs
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed, salt):
    return torch.Generator(device=_dev()).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _smooth(shape, seed, salt, scale, cells=10):
    """FP32 field of unit-variance coarse noise, interpolated linearly: features of about `cells` cells."""
    coarse = [max(2, n // cells + 2) for n in shape]
    x = torch.randn([1, 1] + coarse, generator=_gen(seed, salt), device=_dev())
    mode = {1: "linear", 2: "bilinear", 3: "trilinear"}[len(shape)]
    return torch.nn.functional.interpolate(x, size=list(shape), mode=mode, align_corners=True)[0, 0] * scale


def _vgrid(case):
    return {"slab1d": "signed1d", "batch1d": "signed1d", "tmz2d": "cart2d", "closure": "cart2d",
            "yee3d": "speed3d" if case.get("evolve") else "signed1d"}[case["kind"]]


def _dx(case):
    return LAM0 / (40 if case["kind"] in ("slab1d", "batch1d") else 20)


def _cpml(case):
    return 10 if case["kind"] in ("tmz2d", "closure") else 8


def _nu0(case):
    return (0.005 if case["kind"] == "yee3d" else 0.01) * W0


def _cylinder(case, seed, wp):
    """Gaussian column of radius r with a rippled profile, peak (wp W0)^2 (FP64, zero outside r)."""
    nx, ny, r = case["nx"], case["ny"], case["r"]
    j, i = torch.meshgrid(torch.arange(ny, device=_dev(), dtype=torch.float64),
                          torch.arange(nx, device=_dev(), dtype=torch.float64), indexing="ij")
    r2 = (i - nx / 2) ** 2 + (j - ny / 2) ** 2
    d = torch.exp(-r2 / (0.5 * r * r)) * (1.0 + 0.2 * _smooth((ny, nx), seed, 7, 1.0, 24).double()).clamp_min(0.05)
    d = torch.where(r2 <= r * r, d, torch.zeros_like(d))
    return d * (wp * wp * NC / d.max())


def _inputs(case, seed):
    """Initial fields (FP32, or the grid's precision) and density (FP64) of a single-grid case."""
    k = case["kind"]
    if k == "slab1d":
        nz = case["nz"]
        dens = torch.zeros(nz + 1, dtype=torch.float64, device=_dev())
        dens[case["s0"]:case["s1"]] = 0.25 * NC
        f = dict(ex=_smooth((nz + 1,), seed, 1, 1.0), hy=_smooth((nz,), seed, 2, 1 / ETA0))
        return f, dens
    if k in ("tmz2d", "closure"):
        sh = (case["ny"], case["nx"])
        amp = 5e3 if case.get("nonlinear") else 1.0
        f = dict(ez=_smooth(sh, seed, 1, amp), hx=_smooth(sh, seed, 2, amp / ETA0), hy=_smooth(sh, seed, 3, amp / ETA0))
        f["ez"][0, :] = 0
        f["ez"][:, 0] = 0
        return f, _cylinder(case, seed, 0.9 if k == "closure" else 0.8)
    sh = (case["nz"], case["ny"], case["nx"])
    amp = 1e3 if case["evolve"] else 1.0
    f = {n: _smooth(sh, seed, q, amp / (ETA0 if n[0] == "h" else 1.0))
         for q, n in enumerate(("ex", "ey", "ez", "hx", "hy", "hz"))}
    for n, axes in (("ex", (0, 1)), ("ey", (0, 2)), ("ez", (1, 2))):   # PEC walls
        for ax in axes:
            f[n].select(ax, 0).zero_()
    prof = torch.zeros(case["nz"], dtype=torch.float64, device=_dev())
    s0, s1 = case["s0"], case["s1"]
    prof[s0:s1] = 1.44 * NC * torch.arange(1, s1 - s0 + 1, device=_dev(), dtype=torch.float64) / (s1 - s0)
    return f, prof[:, None, None].expand(sh).contiguous()


def _batch_inputs(case, seed):
    """Per run: nz and slab [a, b) (the case's), density, mean collision frequency, initial E and H (host, FP32)."""
    lengths, rng = np.random.default_rng(20221114), np.random.default_rng(int(seed) + 17)
    runs = []
    for _ in range(case["runs"]):
        nz = int(lengths.integers(case["nz_min"], case["nz_max"] + 1))
        half = int(lengths.uniform(0.2, 0.6) * nz / 2)
        wp, nu = rng.uniform(0.1, 1.5), 10.0 ** rng.uniform(-3.0, -1.0)
        m = nz // 10 + 2
        x, xc = np.arange(nz + 1) / 10.0, np.arange(m + 1)
        e = np.interp(x, xc, rng.standard_normal(m + 1)).astype(np.float32)
        h = np.interp(x[:nz], xc, rng.standard_normal(m + 1) / ETA0).astype(np.float32)
        runs.append(dict(nz=nz, a=nz // 2 - half, b=nz // 2 + half, n=wp * wp * NC, nu0=nu * W0, e=e, h=h))
    return runs


def _train_inputs(case, seed):
    """Sixteen samples of a modulated carrier and the density ratio; a smooth unit-variance target; He-style weights."""
    n, g = case["n"], _gen(seed, 5)

    def u(*s):
        return torch.rand(*s, generator=g, device=_dev())
    amp, ph, gr = torch.exp(0.5 * torch.randn(n, 1, generator=g, device=_dev())), 2 * math.pi * u(n, 1), 0.1 * u(n, 1) - 0.05
    k = torch.arange(16, device=_dev(), dtype=torch.float32)
    e = amp * torch.exp(gr * k) * torch.sin(2 * math.pi / 40 * k + ph)
    d = 0.64 * u(n, 1)
    x = torch.cat([e, d], 1).contiguous()
    t = d[:, 0] * (e[:, 15] - 1.5 * e[:, 9] + 0.7 * e[:, 2] * torch.cos(3 * d[:, 0])) * 4.0

    def w(rows, cols, sd):
        return (torch.randn(rows * cols, generator=g, device=_dev()) * sd)
    z = torch.zeros
    p = torch.cat([w(17, 128, math.sqrt(2 / 17)), z(128, device=_dev()), w(128, 128, math.sqrt(2 / 128)),
                   z(128, device=_dev()), w(128, 1, math.sqrt(1 / 128)), z(1, device=_dev())])
    return x, t.contiguous(), p


def _closure_desc():
    z = np.load(CLOSURE_FILE)
    d = json.loads(str(z["meta"]))
    return z["params"].astype(np.float32), {k: d[k] for k in ("e_scale", "j_scale", "n_scale", "rho", "n_train_max", "beta")}


def _source(case):
    k = case["kind"]
    if k in ("slab1d", "batch1d"):
        return dict(location="point", k=min(100, case.get("nz", 400) // 4), **SOURCE)
    if k in ("tmz2d", "closure"):
        return dict(location="point", i=case["nx"] // 4, j=case["ny"] // 2, **SOURCE)
    c = _cpml(case)
    return dict(location="sheet", k=max(c + 2, case["nz"] // 20), i0=c, i1=case["nx"] - c, j0=c, j1=case["ny"] - c,
                **SOURCE)


def _plasma(case):
    k = case["kind"]
    p = dict(vgrid=_vgrid(case), nv=case.get("nv", 32), nv_perp=case.get("nvp", 32 if k == "closure" else 1), te_ev=1.0,
             vmax_vth=VMAX, nu0=_nu0(case), nu_model="nsv", seed=20221112,
             f_dtype="f64" if case.get("precision") == "f64" else case.get("f_dtype", "f32"))
    if case.get("nonlinear"):
        p["nonlinear"] = 1
    if case.get("evolve"):
        p.update(evolve_f0=1, mass_ratio=1.37e-5, tg_ev=0.026)
    return p


# ---------------------------------------------------------------- the measured call
def prepare(case, seed):
    k = case["kind"]
    if k == "train":
        x, t, p = _train_inputs(case, seed)
        total = 8 * (case["n"] // case["batch"])
        return dict(kind=k, tr=MlpTrainer(p, case["batch"], lr=2e-3), x=x, t=t, seed=int(seed) % 1000, total=total)
    if k == "batch1d":
        specs, runs = [], _batch_inputs(case, seed)
        for r in runs:
            dens = np.zeros(r["nz"] + 1)
            dens[r["a"]:r["b"]] = r["n"]
            specs.append(dict(grid=dict(ndim=1, nx=1, ny=1, nz=r["nz"], dx=_dx(case), courant=0.5, mur=1, precision="f32"),
                              source=_source(case), plasma=dict(_plasma(case), density=dens, nu0=r["nu0"])))
        b = Batch(specs)
        for i, r in enumerate(runs):
            b.write(i, "ex", r["e"])
            b.write(i, "hy", r["h"])
        dtype = dict(ex=torch.float32, hy=torch.float32, j=torch.float32,
                     df=torch.bfloat16 if case["f_dtype"] == "bf16" else torch.float32)
        parts, out = {}, {}
        for q, dt in dtype.items():   # one device buffer per quantity, the runs laid end to end
            size = [b.lib.fdtd_batch_quantity_bytes(b.h, i, QUANTITY[q]) for i in range(len(runs))]
            parts[q] = [(i, int(o), int(s)) for i, (o, s) in enumerate(zip(np.cumsum([0] + size[:-1]), size)) if s]
            out[q] = torch.empty(sum(size) // (2 if dt == torch.bfloat16 else 4), dtype=dt, device=_dev())
        return dict(kind=k, b=b, parts=parts, out=out, steps=case["steps"])
    f, dens = _inputs(case, seed)
    grid = dict(ndim={"slab1d": 1, "yee3d": 3}.get(k, 2), nx=case.get("nx", 1), ny=case.get("ny", 1),
                nz=case.get("nz", 1), dx=_dx(case), courant=0.5, mur=int(k == "slab1d"),
                cpml_cells=0 if k == "slab1d" else _cpml(case), precision=case.get("precision", "f32"))
    s = Solver(grid)
    s.set_source(**_source(case))
    s.set_plasma(dens, **_plasma(case))
    if k == "closure":
        w, d = _closure_desc()
        s.set_closure(w, engine="tcgen05", **d)
    for n, v in f.items():
        s.write(n, v.reshape(-1))
    names = list(f) + ["j"] + ([] if k == "closure" else ["df"]) + (["f0"] if case.get("evolve") else [])
    return dict(kind=k, s=s, steps=case["steps"], names=names)


def run(state):
    k = state["kind"]
    if k == "train":
        tr = state["tr"]
        loss = tr.epoch(state["x"], state["t"], state["seed"], 0, 0, state["total"])
        return dict(loss=loss, params=tr.p, m=tr.m, v=tr.v)
    if k == "batch1d":
        b = state["b"]
        b.step(state["steps"])
        for q, o in state["out"].items():
            base = o.data_ptr()
            for i, off, size in state["parts"][q]:
                b._check(b.lib.fdtd_batch_read(b.h, i, QUANTITY[q], base + off, size, 1))
        return state["out"]
    s = state["s"]
    s.step(state["steps"])
    return {n: s.read(n) for n in state["names"]}


# ------------------------------------------------------------------------ work
def _rows(case):
    """Plasma cells and velocity nodes of a cell."""
    k = case["kind"]
    if k == "slab1d":
        return case["s1"] - case["s0"], case["nv"]
    if k == "batch1d":
        return int(0.4 * case["runs"] * (case["nz_min"] + case["nz_max"]) / 2), case["nv"]
    if k == "yee3d":
        return case["nx"] * (case["ny"] - 1) * (case["s1"] - case["s0"]), case["nv"]
    return int(math.pi * case["r"] ** 2), case.get("nv", 32) * case.get("nvp", 32)


def work(case):
    """Fields, distribution rows and closure histories read and written once a step; the arithmetic of the updates."""
    k = case["kind"]
    if k == "train":
        n = case["n"] // case["batch"] * case["batch"]
        mac = 17 * 128 + 128 * 128 + 128
        return {"bytes": n * 18 * 4 + case["n"] // case["batch"] * 18945 * 4 * 6, "flops": n * mac * 6}
    rows, nn = _rows(case)
    esz = 8 if case.get("precision") == "f64" else 4
    fb = 2 if case.get("f_dtype") == "bf16" else esz
    if k == "batch1d":
        cells, comp = case["runs"] * (case["nz_min"] + case["nz_max"]) / 2, 2
    else:
        cells = case.get("nx", 1) * case.get("ny", 1) * case.get("nz", 1)
        comp = {"slab1d": 2, "yee3d": 6}.get(k, 3)
    b, fl = 2 * esz * comp * cells, 6 * comp * cells
    if k == "closure":      # per cell: the history ring, density and J; the network
        b += rows * (32 + 2 + 4 + 8)
        fl += rows * 2 * (17 * 128 + 128 * 128 + 128)
    else:
        b += 2 * fb * rows * nn * (2 if case.get("evolve") else 1)
        fl += rows * nn * (30 if case.get("evolve") or case.get("nonlinear") else 6)
    return {"bytes": b * case["steps"], "flops": fl * case["steps"]}


# ---------------------------------------------------- the same steps in 64 bits
def _tables(case, dt, nu0):
    """Velocity nodes of the grid: alpha, beta, w' = -e w, and the F0 pieces of the speed grid (FP64)."""
    vth = math.sqrt(QE * 1.0 / ME)
    nv, grid = case.get("nv", 32), _vgrid(case)
    vm = VMAX * vth
    if grid == "speed3d":
        gam = vm / nv
        v = (torch.arange(nv, device=_dev(), dtype=torch.float64) + 0.5) * gam
        speed, dV, w = v, 4 * math.pi * v * v * gam, 4 * math.pi / 3 * v ** 3 * gam
        f0 = torch.exp(-v * v / (2 * vth * vth)) / (2 * math.pi * vth * vth) ** 1.5
    else:
        dv = 2 * vm / nv
        v = (torch.arange(nv, device=_dev(), dtype=torch.float64) + 0.5 - 0.5 * nv) * dv
        if grid == "cart2d":
            nq = case.get("nvp", 32)
            dq = 2 * vm / nq
            q = (torch.arange(nq, device=_dev(), dtype=torch.float64) + 0.5 - 0.5 * nq) * dq
            v, q = (t.reshape(-1) for t in torch.meshgrid(v, q, indexing="ij"))
            speed, dV = torch.sqrt(v * v + q * q), torch.full_like(v, dv * dq)
            f0 = torch.exp(-(v * v + q * q) / (2 * vth * vth)) / (2 * math.pi * vth * vth)
        else:
            speed, dV = v.abs(), torch.full_like(v, dv)
            f0 = torch.exp(-v * v / (2 * vth * vth)) / math.sqrt(2 * math.pi * vth * vth)
        w, gam = v * dV, dv
    nu = nu0 * speed / ((speed * f0 * dV).sum() / (f0 * dV).sum())
    f0p = -v / (vth * vth) * f0
    return dict(v=v, nu=nu, f0=f0, f0p=f0p, gam=gam, al=(2 - dt * nu) / (2 + dt * nu),
                be=2 * dt * (QE / ME) * f0p / (2 + dt * nu), w=-QE * w)


def _pulse(t):
    u = (t - SOURCE["t0"]) / TAU
    return math.sin(2 * math.pi * F0 * (t - SOURCE["t0"])) * math.exp(-u * u)


def _cpml_axis(n, L, dx, dt, half):
    """b, a and 1/kappa of one axis at integer or half-integer positions (polynomial grading of order 3)."""
    x = (np.arange(n) + (0.5 if half else 0.0)) * dx
    delta = L * dx
    rho = np.where(x < delta, delta - x, np.where(x > (n - L) * dx, x - (n - L) * dx, 0.0)) / delta
    inside = (x < delta) | (x > (n - L) * dx)
    sig, kap, alp = 1.3 * 4.0 / (150 * math.pi * dx) * rho ** 3, 1 + 6.0 * rho ** 3, 0.05 * (1 - rho)
    b = np.where(inside, np.exp(-(sig / kap + alp) * dt / EPS0), 0.0)
    a = np.where(inside & (sig > 0), sig * (b - 1) / (dx * (sig * kap + alp * kap * kap)), 0.0)
    return [torch.as_tensor(t, device=_dev()) for t in (b, a, np.where(inside, 1 / kap, 1.0))]


class _Cpml:
    """psi <- b psi + a d and d / kappa + dx-scaled psi for one derivative along one axis of an ndim array."""

    def __init__(self, case, ndim, dt):
        self.dx, self.nd = _dx(case), ndim
        n = [case["nx"], case["ny"], case.get("nz", 1)][:ndim]
        self.t = [[_cpml_axis(n[a], _cpml(case), self.dx, dt, h) for h in (0, 1)] for a in range(ndim)]
        self.psi = {}

    def __call__(self, key, d, axis, half):
        b, a, ik = (t.reshape([-1] + [1] * axis) for t in self.t[axis][half])
        p = self.psi.get(key)
        p = a * d if p is None else p.mul_(b).add_(a * d)
        self.psi[key] = p
        return (d * ik).add_(p, alpha=self.dx)


def _up(f, ax):
    """f at the next node along tensor axis ax minus f (a zero ghost past the end)."""
    d = -f
    n = f.shape[ax]
    d.narrow(ax, 0, n - 1).add_(f.narrow(ax, 1, n - 1))
    return d


def _down(f, ax):
    """f minus f at the previous node along tensor axis ax (zero at the first node)."""
    d = torch.zeros_like(f)
    n = f.shape[ax]
    torch.sub(f.narrow(ax, 1, n - 1), f.narrow(ax, 0, n - 1), out=d.narrow(ax, 1, n - 1))
    return d


class _Rows:
    """The distribution rows of a plasma: linear, with velocity-space advection, or with an evolving F0."""

    def __init__(self, case, dt, n, nu0=None):
        self.case, self.dt, self.n = case, dt, n
        self.t = _tables(case, dt, _nu0(case) if nu0 is None else nu0)
        nn = self.t["al"].numel()
        self.df = torch.zeros(n.numel(), nn, dtype=torch.float64, device=_dev())
        self.g = torch.zeros_like(self.df) if case.get("evolve") else None

    def step(self, E):
        t, dt = self.t, self.dt
        if self.case.get("nonlinear"):
            self.df = self._advect(E)
        elif self.g is not None:
            self._evolve(E)
        else:
            self.df.mul_(t["al"])
            for a in range(0, E.numel(), 1 << 18):
                self.df[a:a + (1 << 18)].addmm_((self.n * E)[a:a + (1 << 18), None], t["be"][None, :])
        return self.df @ t["w"]

    def _advect(self, E):
        t, dt, out = self.t, self.dt, torch.empty_like(self.df)
        npar, nperp = self.case["nv"], self.case["nvp"]
        for s in range(0, E.numel(), 1 << 14):
            x = self.df[s:s + (1 << 14)].reshape(-1, npar, nperp)
            acc = (-(QE / ME) * E[s:s + (1 << 14)])[:, None, None]
            flux = torch.zeros(x.shape[0], npar + 1, nperp, dtype=x.dtype, device=x.device)
            flux[:, 1:-1] = acc * torch.where(acc > 0, x[:, :-1], x[:, 1:])
            A = -(flux[:, 1:] - flux[:, :-1]) / t["gam"]
            odd, even = 0.5 * (x - x.flip(1)), 0.5 * (x + x.flip(1))
            ao, ae = 0.5 * (A - A.flip(1)), 0.5 * (A + A.flip(1))
            al, be = t["al"].reshape(1, npar, nperp), t["be"].reshape(1, npar, nperp)
            nE = (self.n * E)[s:s + (1 << 14)][:, None, None]
            y = even + dt * ae + al * odd + be * nE + dt * (1 + al) * 0.5 * ao
            out[s:s + (1 << 14)] = y.reshape(x.shape[0], -1)
        return out

    def _evolve(self, E):
        t, dt, g, n = self.t, self.dt, self.g, self.n[:, None]
        gam, v, nv = t["gam"], t["v"], t["v"].numel()
        gp = torch.zeros_like(g)
        gp[:, :-1] = g[:, 1:]
        gm = torch.cat([g[:, :1], g[:, :-1]], 1)
        bq = 2 * dt * (QE / ME) / (2 + dt * t["nu"])
        new = t["al"] * self.df + bq * (t["f0p"] + (gp - gm) / (2 * gam)) * (n * E[:, None])
        a = v ** 3 * 0.5 * (self.df + new) / n
        ve = torch.arange(1, nv, device=_dev(), dtype=torch.float64) * gam
        F = t["f0"] + g
        flux = torch.zeros(g.shape[0], nv + 1, dtype=g.dtype, device=g.device)
        flux[:, 1:-1] = (QE / ME / 3) * E[:, None] * (a[:, :-1] + a[:, 1:]) / (2 * ve)
        c1 = 1.37e-5 * ve ** 3 * 0.5 * (t["nu"][:-1] + t["nu"][1:])
        flux[:, 1:-1] += c1 * (0.5 * (F[:, :-1] + F[:, 1:]) + QE * 0.026 / ME / (ve * gam) * (F[:, 1:] - F[:, :-1]))
        self.g = g + dt * (flux[:, 1:] - flux[:, :-1]) / (v * v * gam)
        self.df = new


def _exact_line(case, seed):
    """One line, or a batch of lines laid end to end (each with its own tables), with Mur ends."""
    if case["kind"] == "slab1d":
        f, dens = _inputs(case, seed)
        lines = [dict(nz=case["nz"], a=case["s0"], b=case["s1"], n=0.25 * NC, nu0=_nu0(case), e=f["ex"].cpu().numpy(),
                      h=f["hy"].cpu().numpy())]
    else:
        lines = _batch_inputs(case, seed)
    dx = _dx(case)
    dt = 0.5 * dx / C0
    ch, ce = dt * C0 * C0 * EPS0 / dx, dt / (EPS0 * dx)
    m = (C0 * dt - dx) / (C0 * dt + dx)
    off = np.cumsum([0] + [r["nz"] + 1 for r in lines])
    i64 = dict(device=_dev(), dtype=torch.int64)
    E = torch.as_tensor(np.concatenate([r["e"] for r in lines]), device=_dev()).double()
    H = torch.as_tensor(np.concatenate([np.append(r["h"], 0.0) for r in lines]), device=_dev()).double()
    first, last = torch.as_tensor(off[:-1], **i64), torch.as_tensor(off[1:] - 1, **i64)
    src = first + _source(case)["k"]
    cells = torch.cat([torch.arange(o + r["a"], o + r["b"], **i64) for o, r in zip(off, lines)])
    rows = [r["b"] - r["a"] for r in lines]
    n = torch.cat([torch.full((c,), r["n"], dtype=torch.float64, device=_dev()) for c, r in zip(rows, lines)])
    tabs = [_tables(case, dt, r["nu0"]) for r in lines]
    w, nn = tabs[0]["w"], tabs[0]["w"].numel()
    df = torch.zeros(int(sum(rows)), nn, dtype=torch.float64, device=_dev())
    line = torch.repeat_interleave(torch.arange(len(lines), device=_dev()), torch.as_tensor(rows, device=_dev()))
    al, be = torch.stack([t["al"] for t in tabs]), torch.stack([t["be"] for t in tabs])
    inner = torch.ones(E.numel(), dtype=torch.bool, device=_dev())
    inner[first] = False
    inner[last] = False
    J = torch.zeros_like(n)
    for s in range(case["steps"]):
        d = torch.zeros_like(H)
        d[:-1] = E[1:] - E[:-1]
        d[last] = 0
        H -= ch * d
        e1, e2, b1, b2 = E[first + 1], E[last - 1], E[first], E[last]
        nE = n * E[cells]
        for a in range(0, n.numel(), 1 << 18):
            q = slice(a, a + (1 << 18))
            df[q] = al[line[q]] * df[q] + be[line[q]] * nE[q, None]
        J = df @ w
        E[cells] -= dt / EPS0 * J
        d = torch.zeros_like(E)
        d[1:] = H[1:] - H[:-1]
        E = torch.where(inner, E - ce * d, E)
        E[src] += _pulse((s + 1) * dt)
        E[first] = e1 + m * (E[first + 1] - b1)
        E[last] = e2 + m * (E[last - 1] - b2)
    keep = torch.ones(H.numel(), dtype=torch.bool, device=_dev())
    keep[last] = False
    if case["kind"] == "batch1d":
        return dict(ex=E, hy=H[keep], j=J, df=df.reshape(-1))
    return dict(ex=E, hy=H[keep], j=J, df=df)


def _gelu(z):
    return 0.5 * z * (1 + torch.tanh(math.sqrt(2 / math.pi) * (z + 0.044715 * z ** 3)))


def _split(p):
    o = np.cumsum([0, 17 * 128, 128, 128 * 128, 128, 128, 1])
    w1, b1, w2, b2, w3, b3 = (p[a:b] for a, b in zip(o[:-1], o[1:]))
    return w1.reshape(17, 128), b1, w2.reshape(128, 128), b2, w3, b3


class _Closure:
    """Rows above the training density keep the velocity-space update; the others take the network."""

    def __init__(self, case, dt, n, cells):
        p, self.d = _closure_desc()
        self.p = [t.double() for t in _split(torch.as_tensor(p, device=_dev()))]
        dense = n > self.d["n_train_max"]
        self.cells, order = torch.cat([cells[dense], cells[~dense]]), torch.cat([n[dense], n[~dense]])
        self.nk = int(dense.sum())
        self.rows, self.n = _Rows(case, dt, order[:self.nk]), order[self.nk:]
        self.hist = torch.zeros(16, self.n.numel(), dtype=torch.float64, device=_dev())
        self.J = torch.zeros_like(self.n)

    def step(self, E):
        d, (w1, b1, w2, b2, w3, b3) = self.d, self.p
        jk, Ec = self.rows.step(E[:self.nk]), E[self.nk:]
        self.hist = torch.cat([self.hist[1:], Ec[None]])
        y = torch.empty_like(Ec)
        for a in range(0, Ec.numel(), 1 << 19):
            q = slice(a, a + (1 << 19))
            x = torch.cat([self.hist[:, q].t() / d["e_scale"], (self.n[q] / d["n_scale"])[:, None]], 1)
            y[q] = _gelu(_gelu(x @ w1 + b1) @ w2 + b2) @ w3 + b3
        self.J = d["rho"] * self.J + d["beta"] * self.n * Ec + d["j_scale"] * y
        return torch.cat([jk, self.J])


def _exact_grid(case, seed):
    nd = 3 if case["kind"] == "yee3d" else 2
    f, dens = _inputs(case, seed)
    f = {n: v.double() for n, v in f.items()}
    dx = _dx(case)
    dt = 0.5 * dx / C0
    ch, ce = dt * C0 * C0 * EPS0 / dx, dt / (EPS0 * dx)
    pol = "ex" if nd == 3 else "ez"
    live = dens > 0
    live.select(0, 0).zero_()
    live.select(1, 0).zero_()
    cells = live.reshape(-1).nonzero()[:, 0]
    n = dens.reshape(-1)[cells]
    n = n.float().double() if case["kind"] != "closure" else n   # the solver's rows hold FP32 densities
    del dens, live
    if case["kind"] == "closure":
        plasma = _Closure(case, dt, n, cells)
        cells = plasma.cells
    else:
        plasma = _Rows(case, dt, n)
    c = _Cpml(case, nd, dt)
    src = _source(case)
    J = None
    for s in range(case["steps"]):
        if nd == 2:
            f["hx"].sub_(c("hx", _up(f["ez"], 0), 1, 1), alpha=ch)
            f["hy"].add_(c("hy", _up(f["ez"], 1), 0, 1), alpha=ch)
        else:   # tensor axes are (z, y, x); CPML axes (x, y, z)
            for h, (p, ap), (q, aq) in (("hx", ("ez", 1), ("ey", 2)), ("hy", ("ex", 2), ("ez", 0)),
                                        ("hz", ("ey", 0), ("ex", 1))):
                f[h].sub_(c(h + "p", _up(f[p], 2 - ap), ap, 1), alpha=ch)
                f[h].add_(c(h + "q", _up(f[q], 2 - aq), aq, 1), alpha=ch)
        flat = f[pol].view(-1)
        E = flat[cells]
        J = plasma.step(E)
        flat[cells] = E - dt / EPS0 * J
        if nd == 2:
            u = c("ezx", _down(f["hy"], 1), 0, 0) - c("ezy", _down(f["hx"], 0), 1, 0)
            f["ez"][1:, 1:].add_(u[1:, 1:], alpha=ce)
            f["ez"][src["j"], src["i"]] += _pulse((s + 1) * dt)
        else:
            for e, (p, ap), (q, aq) in (("ex", ("hz", 1), ("hy", 2)), ("ey", ("hx", 2), ("hz", 0)),
                                        ("ez", ("hy", 0), ("hx", 1))):
                u = c(e + "p", _down(f[p], 2 - ap), ap, 0) - c(e + "q", _down(f[q], 2 - aq), aq, 0)
                wall = [slice(0 if "zyx"[a] == e[1] else 1, None) for a in range(3)]
                f[e][tuple(wall)].add_(u[tuple(wall)], alpha=ce)
            f["ex"][src["k"], src["j0"]:src["j1"], src["i0"]:src["i1"]] += _pulse((s + 1) * dt)
    out = {k: v.reshape(-1) for k, v in f.items()}
    out["j"] = J
    if case["kind"] != "closure":
        out["df"] = plasma.df
    if case.get("evolve"):
        out["f0"] = plasma.g
    return out


def _philox7(c, k):
    """Philox4x32 with seven rounds on uint64 arrays holding 32-bit words."""
    m32 = np.uint64(0xFFFFFFFF)
    for _ in range(7):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [((p1 >> np.uint64(32)) ^ c[1] ^ k[0]) & m32, p1 & m32, ((p0 >> np.uint64(32)) ^ c[3] ^ k[1]) & m32, p0 & m32]
        k = [(k[0] + np.uint64(0x9E3779B9)) & m32, (k[1] + np.uint64(0xBB67AE85)) & m32]
    return c


def _shuffle(n, seed, epoch):
    """The trainer's seeded order of n samples: a four-round Feistel network, walked until it lands below n."""
    bits = max(2, (n - 1).bit_length())
    half = np.uint64((bits + bits % 2) // 2)
    mask = np.uint64((1 << int(half)) - 1)
    key = [np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)]
    out = np.arange(n, dtype=np.uint64)
    todo = np.ones(n, dtype=bool)
    while todo.any():
        x = out[todo]
        L, R = x >> half, x & mask
        for r in range(4):
            z = np.zeros_like(R)
            h = _philox7([R, z + np.uint64(r), z + np.uint64(epoch & 0xFFFFFFFF), z + np.uint64(epoch >> 32)], key)[0]
            L, R = R, (L ^ h) & mask
        x = (L << half) | R
        out[todo] = x
        todo[todo] = x >= np.uint64(n)
    return torch.as_tensor(out.astype(np.int64), device=_dev())


def _exact_train(case, seed):
    x, t, p = _train_inputs(case, seed)
    x, t, p = x.double(), t.double(), p.double()
    n, B = case["n"], case["batch"]
    order = _shuffle(n, int(seed) % 1000, 0)
    m, v, total, loss, nb = torch.zeros_like(p), torch.zeros_like(p), 8 * (n // B), 0.0, n // B
    for b in range(nb):
        q = order[b * B:(b + 1) * B]
        w = p.clone().requires_grad_(True)
        w1, b1, w2, b2, w3, b3 = _split(w)
        y = _gelu(_gelu(x[q] @ w1 + b1) @ w2 + b2) @ w3 + b3
        L = ((y - t[q]) ** 2).mean()
        g, = torch.autograd.grad(L, w)
        loss += float(L.detach()) / nb
        lr = 2e-3 * 0.5 * (1 + math.cos(math.pi * min(b, total) / total))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        p = p - lr * (m / (1 - 0.9 ** (b + 1))) / (torch.sqrt(v / (1 - 0.999 ** (b + 1))) + 1e-8)
    return dict(loss=torch.tensor([loss], dtype=torch.float64), params=p, m=m, v=v)


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] in ("slab1d", "batch1d"):
        return _exact_line(case, seed)
    return _exact_grid(case, seed)
