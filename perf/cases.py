"""The work a user of this library has it do, as timed cases.

A case is one pass of a user's program through the public binding
(``paper_1806_06917_gb300.pd`` and ``autograd``): a run of explicit steps from a
state the program holds on the device, the same with host arrays every step, a
static solve, a force with its gradient, the setup of a simulation, or a batch of
requests to the server. ``kind`` names which; the other fields are sizes and options.

``exact`` evaluates the same physics in plain 64-bit torch: bonds gathered from
lattice coordinates, no code of the package.
"""
import math

import numpy as np
import torch

from paper_1806_06917_gb300 import pd
from paper_1806_06917_gb300 import workloads as wk
from paper_1806_06917_gb300.autograd import internal_force

MODELS = {"pmb": wk.PMB, "lps": wk.LPS, "np": wk.NP, "lp": wk.LP}
# 64-bit or 32-bit operations one directed bond needs per evaluation of each law
BOND_FLOPS = {"pmb": 30, "lps": 24 + 38, "np": 14, "lp": 11}


def _steps(name, model, n, m, steps, **kw):
    c = dict(name=name, kind="steps", model=model, nx=n[0], ny=n[1], nz=n[2] if len(n) == 3 else 1, m=m, steps=steps,
             precision="fp32c", state="f64", integrator="verlet", vol_corr=False, breaking=False, collar="none",
             energy=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest simulation of the repository's workloads: the 50 x 50 plate pulled at two
        # collars, its whole 200-step run; eight tiles, every step bound by latency
        _steps("plate50_run", "pmb", (50, 50), 3, 200, collar="velocity"),
        # a crack-growth run: the notched 64^3 block, bonds breaking under the pulse, read back
        # every 20 steps
        _steps("block64_break", "pmb", (64, 64, 64), 3, 20, breaking=True),
        # the large production block: 16.8 million points, 2e9 bonds, two steps and a read-back
        _steps("block256", "pmb", (256, 256, 256), 3, 2),
        # the state-based headline workload: the 128^3 LPS block
        _steps("lps128", "lps", (128, 128, 128), 3, 8),
        # an ordinary request's size, ragged against the tiles, with the energies monitored
        _steps("lps_ragged", "lps", (45, 37, 52), 3, 40, energy=True),
        # the paper's explicit benchmark: 443^2 lattice at the wide horizon m = 20, NP law
        _steps("np443_m20", "np", (443, 443), 20, 10, collar="clamp"),
        # a reference run in full FP64, as used to check an FP32C production run
        _steps("block64_fp64", "pmb", (64, 64, 64), 3, 2, precision="fp64"),
        # a program that pushes states from host memory through one step each (two upload buffers
        # in turn) and takes the displacements back, pipelined
        dict(name="lps96_host", kind="host", model="lps", nx=96, ny=96, nz=96, m=3, steps=6),
        # one load step of the 200 x 200 clamped plate's quasi-static path, GMRES(50), FP64
        dict(name="static200", kind="static", nx=200, ny=200, m=3, krylov="gmres", precond=False, precision="fp64"),
        # force and its gradient through the torch bridge (an inverse problem's inner call)
        dict(name="grad200", kind="grad", nx=200, ny=200, nz=1, m=3, precision="fp64"),
        # setting up a simulation: create, neighbour build, neighbour lists read out
        dict(name="setup64", kind="setup", model="pmb", nx=64, ny=64, nz=64, m=3),
        # a batch of small mixed requests to a running server, waited for
        dict(name="serve12", kind="serve", count=12, median=24, lo=10, hi=48, steps_lo=50, steps_hi=150),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps"] * 6 + ["host", "static", "grad", "setup", "serve"])
    if kind == "steps":
        model = rng.choice(["pmb", "pmb", "lps", "lps", "np", "lp"])
        dim = 3 if model == "lps" else 2 if model in ("np", "lp") else rng.choice([2, 3, 3])
        precision = rng.choice(["fp32c", "fp32c", "fp32c", "fp64"])
        if dim == 2:
            n = (_log(rng, 25, 440), _log(rng, 25, 440))
            wide = [k for k in (2, 3, 4, 8, 20) if 6 * k <= min(n) and (k <= 8 or precision == "fp32c")]
            m = rng.choice(wide if model in ("np", "lp") else [2, 3, 4])
        else:
            hi = 64 if precision == "fp64" else 128
            n = tuple(_log(rng, 20, hi) for _ in range(3))
            m = rng.choice([2, 3, 3, 4])
        bonds = _bonds_about(n, m)
        per_step = bonds * BOND_FLOPS[model] * (64 if precision == "fp64" else 1)
        steps = max(1, min(_log(rng, 2, 200), int(4e10 / per_step)))
        breaking = model == "pmb" and dim == 3 and precision == "fp32c" and rng.random() < 0.5
        c = _steps("", model, n, m, steps, precision=precision, breaking=breaking,
                   state=rng.choice(["f64", "f64", "f64", "df"]) if precision == "fp32c" else "f64",
                   integrator=rng.choice(["verlet", "verlet", "verlet", "cd"]),
                   vol_corr=rng.random() < 0.2, energy=rng.random() < 0.3,
                   collar="clamp" if model in ("np", "lp") else "velocity" if dim == 2 else "none")
        del c["name"]
        return c
    if kind == "host":
        n = [_log(rng, 24, 96) for _ in range(3)]
        return dict(kind="host", model=rng.choice(["pmb", "lps"]), nx=n[0], ny=n[1], nz=n[2], m=rng.choice([2, 3]),
                    steps=rng.randint(2, 8))
    if kind == "static":
        return dict(kind="static", nx=_log(rng, 30, 160), ny=_log(rng, 30, 160), m=rng.choice([2, 3]),
                    krylov=rng.choice(["gmres", "cg"]), precond=rng.random() < 0.3, precision="fp64")
    if kind == "grad":
        d3 = rng.random() < 0.4
        n = [_log(rng, 16, 48) for _ in range(3)] if d3 else [_log(rng, 30, 300), _log(rng, 30, 300), 1]
        return dict(kind="grad", nx=n[0], ny=n[1], nz=n[2], m=rng.choice([2, 3]),
                    precision=rng.choice(["fp64", "fp32c"]))
    if kind == "setup":
        d3 = rng.random() < 0.7
        n = [_log(rng, 16, 128) for _ in range(3)] if d3 else [_log(rng, 30, 800), _log(rng, 30, 800), 1]
        return dict(kind="setup", model=rng.choice(["pmb", "lps"]) if d3 else "pmb", nx=n[0], ny=n[1], nz=n[2],
                    m=rng.choice([2, 3, 4]))
    lo = rng.randint(8, 14)
    return dict(kind="serve", count=rng.randint(4, 14), median=rng.randint(16, 28), lo=lo, hi=rng.randint(30, 50),
                steps_lo=20, steps_hi=rng.randint(40, 150))


# ----------------------------------------------------------------- descriptions

def _dim(c):
    return 3 if c.get("nz", 1) > 1 else 2


def _offsets(dim, m):
    r = range(-m, m + 1)
    return [(x, y, z) for z in (r if dim == 3 else (0,)) for y in r for x in r if 0 < x * x + y * y + z * z <= m * m]


def _bonds_about(n, m):
    total = 0
    for d in _offsets(len(n), m):
        k = 1
        for a in range(len(n)):
            k *= max(0, n[a] - abs(d[a]))
        total += k
    return total


def _bonds(c):
    return _bonds_about((c["nx"], c["ny"], c["nz"])[:_dim(c)], c["m"])


def _grid(c):
    dim = _dim(c)
    if c.get("model") in ("np", "lp"):      # the study's horizon: h = 0.05 / 20 at m = 20, 0.1 / m below
        h = (0.05 if c["m"] >= 20 else 0.1) / c["m"]
        return wk.Grid(dim=2, n=(c["nx"], c["ny"], 1), h=h, m=c["m"], origin=(-c["m"] * h, -c["m"] * h, 0.0))
    return wk.Grid(dim=dim, n=(c["nx"], c["ny"], c.get("nz", 1)), h=1.0 / c["nx"], m=c["m"])


def _material(c):
    model = MODELS[c.get("model", "pmb")]
    v = int(c.get("vol_corr", False))
    if model == wk.LPS:
        return wk.Material(model=model, E=72e9, rho=2440.0, K=40e9, mu=30e9, vol_corr=v)
    if model in (wk.NP, wk.LP):
        return wk.Material(model=model, E=0.0, rho=1.0, psi_c=1.0, psi_beta=1.0, vol_corr=v)
    return wk.Material(model=model, E=72e9, rho=2440.0, s_c=1e-3 if c.get("breaking") else 0.0, vol_corr=v)


def _run(c):
    return dict(precision=pd.PD_FP64 if c.get("precision") == "fp64" else pd.PD_FP32C,
                dt=1e-5 if c.get("model") in ("np", "lp") else 0.0,
                integrator=pd.PD_INTEGRATOR_CD if c.get("integrator") == "cd" else pd.PD_INTEGRATOR_VERLET,
                state=pd.PD_STATE_DF if c.get("state") == "df" else pd.PD_STATE_F64)


def _coords(g):
    i = torch.arange(g.npoints, device="cuda")
    nx, ny = g.n[0], g.n[1]
    return torch.stack([i % nx, (i // nx) % ny, i // (nx * ny)], 1)[:, :g.dim]


def _notch(c):
    return dict(axis=2, pos=c["nz"] // 2 - 0.5, lo=(-0.5, -0.5, 0.0), hi=(0.1 * c["nx"], c["ny"] - 0.5, 0.0))


def _initial(c, g, seed):
    """u0, v0 and the collar (kind, value; None for a free lattice) of a run, FP64 on the device."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rnd = np.random.default_rng(seed)
    xyz = _coords(g)
    X = xyz.double() * g.h + torch.tensor(g.origin[:g.dim], dtype=torch.float64, device="cuda")
    v0 = torch.zeros_like(X)
    kind = val = None
    model = c.get("model", "pmb")
    if model in ("np", "lp"):
        ext = [g.h * (k - 1 - 2 * g.m) for k in g.n[:2]]       # the material domain inside the collar
        ctr = torch.tensor([e * rnd.uniform(0.4, 0.6) for e in ext], dtype=torch.float64, device="cuda")
        a = torch.tensor([1e-3, rnd.uniform(0.0, 5e-4)], dtype=torch.float64, device="cuda")
        u0 = torch.exp(-((X - ctr) ** 2).sum(1, keepdim=True) / rnd.uniform(0.003, 0.01)) * a
    elif model == "lps":
        u0 = (1e-4 / 3.0) * X + torch.randn(X.shape, generator=gen, device="cuda", dtype=torch.float64) * (1e-5 * g.h)
    elif c.get("breaking"):
        # a pulse that has stretched its flank to about the critical stretch, still moving outwards
        ctr = 0.5 * g.h * (torch.tensor(g.n, dtype=torch.float64, device="cuda") - 1)
        p = torch.exp(-((X - ctr) ** 2).sum(1, keepdim=True) / (8.0 * g.h) ** 2)
        ex = torch.tensor([1.0, 0.0, 0.0], dtype=torch.float64, device="cuda")
        u0 = p * ex * (rnd.uniform(0.0115, 0.0125) * g.h)
        u0 = u0 + torch.randn(X.shape, generator=gen, device="cuda", dtype=torch.float64) * (1e-5 * g.h)
        v0 = p * ex
    else:
        u0 = torch.randn(X.shape, generator=gen, device="cuda", dtype=torch.float64) * (1e-4 * g.h)
    collar = c.get("collar", "none")
    if collar != "none":
        kind = torch.zeros(X.shape, dtype=torch.uint8, device="cuda")
        val = torch.zeros_like(X)
        left, right = xyz[:, 0] < g.m, xyz[:, 0] >= g.n[0] - g.m
        if collar == "velocity":
            kind[left | right, 0] = pd.PD_BC_VELOCITY
            val[left, 0], val[right, 0] = -0.1, 0.1
            v0 = val.clone()
        else:
            out = left | right | (xyz[:, 1] < g.m) | (xyz[:, 1] >= g.n[1] - g.m)
            kind[out] = pd.PD_BC_DISPLACEMENT
            u0[out] = 0.0
    return u0.contiguous(), v0.contiguous(), kind, val


def _clamped(c, g, strain):
    """The clamped plate's collar: left held, right pulled by strain x width."""
    xyz = _coords(g)
    kind = torch.zeros((g.npoints, 2), dtype=torch.uint8, device="cuda")
    val = torch.zeros((g.npoints, 2), dtype=torch.float64, device="cuda")
    left, right = xyz[:, 0] < g.m, xyz[:, 0] >= g.n[0] - g.m
    kind[left] = pd.PD_BC_DISPLACEMENT
    kind[right, 0] = pd.PD_BC_DISPLACEMENT
    val[right, 0] = strain * (g.n[0] - 1) * g.h
    return kind, val


def _strain(seed):
    return 1e-5 * np.random.default_rng(seed).uniform(0.8, 1.2)


def _grad_inputs(c, g, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    shape = (g.npoints, g.dim)
    u = torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64) * (1e-4 * g.h)
    return u, torch.randn(shape, generator=gen, device="cuda", dtype=torch.float64)


def _requests(c, seed):
    # the mix itself (sizes, laws, steps) belongs to the case, the initial data to the seed
    mix = wk.serving_mix(count=c["count"], seed=5, side_median=c["median"], side_lo=c["lo"], side_hi=c["hi"],
                         steps_lo=c["steps_lo"], steps_hi=c["steps_hi"], m_choices=(2, 3))
    rng = np.random.default_rng(seed)
    return [(r, rng.normal(0.0, 1e-4 * r.grid.h, size=(r.grid.npoints, r.grid.dim))) for r in mix]


# ------------------------------------------------------------------ prepare, run

def _sim(c, g):
    sim = pd.pd_create(*pd.describe(g, _material(c), **_run(c)))
    pd.pd_build_neighbors(sim, stream=torch.cuda.current_stream())
    return sim


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        reqs = _requests(c, seed)
        out = [(np.empty_like(u0), np.empty_like(u0)) for _, u0 in reqs]
        return dict(kind=kind, server=pd.Server(), reqs=[(pd.describe(r.grid, r.mat), r.steps, u0) for r, u0 in reqs],
                    out=out)
    if kind == "setup":
        # the random origin does not enter the lists; the material sets the time step
        g, mat = _grid(c), _material(c)
        mat.rho *= np.random.default_rng(seed).uniform(0.9, 1.1)
        n, nb = g.npoints, _bonds(c)
        return dict(kind=kind, desc=pd.describe(g, mat), row_ptr=torch.empty(n + 1, dtype=torch.int64, device="cuda"),
                    col=torch.empty(nb, dtype=torch.int32, device="cuda"),
                    perm=torch.empty(n, dtype=torch.int64, device="cuda"))
    g = _grid(c)
    sim = _sim(c, g)
    st = torch.cuda.current_stream()
    if kind == "grad":
        u, w = _grad_inputs(c, g, seed)
        return dict(kind=kind, sim=sim, u=u, w=w)
    if kind == "static":
        k, v = _clamped(c, g, _strain(seed))
        pd.pd_set_bc(sim, k, v, stream=st)
        opts = pd.newton_opts(krylov=pd.PD_KRYLOV_GMRES if c["krylov"] == "gmres" else pd.PD_KRYLOV_CG,
                              precond=pd.PD_PRECOND_BLOCK_JACOBI if c["precond"] else pd.PD_PRECOND_NONE)
        zero = torch.zeros((g.npoints, 2), dtype=torch.float64, device="cuda")
        return dict(kind=kind, sim=sim, opts=opts, zero=zero, u=torch.empty_like(zero))
    u0, v0, k, v = _initial(c, g, seed)
    if c.get("breaking"):
        q = _notch(c)
        pd.pd_break_bonds(sim, q["axis"], q["pos"], q["lo"], q["hi"], stream=st)
    if k is not None:
        pd.pd_set_bc(sim, k, v, stream=st)
    s = dict(kind=kind, sim=sim, steps=c["steps"], energy=c.get("energy", False))
    if kind == "host":
        u1, v1 = _initial(c, g, seed + 7919)[:2]
        s.update(src=[(a.cpu().pin_memory(), b.cpu().pin_memory()) for a, b in ((u0, v0), (u1, v1))],
                 out=[torch.empty(u0.shape, dtype=torch.float64).pin_memory() for _ in range(c["steps"])])
        return s
    return s | dict(u0=u0, v0=v0, u=torch.empty_like(u0), v=torch.empty_like(u0))


def run(s):
    kind, st = s["kind"], torch.cuda.current_stream()
    if kind == "steps":
        sim = s["sim"]
        pd.pd_set_state(sim, s["u0"], s["v0"], stream=st)
        pd.pd_step_explicit(sim, s["steps"], stream=st)
        out = {}
        if s["energy"]:
            out["kinetic"], out["strain"] = pd.pd_energy(sim, stream=st)
        out["u"], out["v"] = pd.pd_get_state(sim, s["u"], s["v"], stream=st)
        return out
    if kind == "host":
        sim = s["sim"]
        for k in range(s["steps"]):
            pd.pd_set_state_async(sim, *s["src"][k % 2], stream=st)
            pd.pd_step_explicit(sim, 1, stream=st)
            pd.pd_get_state_async(sim, s["out"][k], stream=st)
        pd.pd_io_sync(sim)
        return s["out"]
    if kind == "static":
        pd.pd_set_state(s["sim"], s["zero"], s["zero"], stream=st)
        r = pd.pd_solve_static(s["sim"], s["opts"], stream=st)
        pd.pd_get_state(s["sim"], s["u"], stream=st, want_v=False)
        return {"u": s["u"], "converged": r["converged"]}
    if kind == "grad":
        u = s["u"].detach().requires_grad_(True)
        f = internal_force(s["sim"], u)
        (gu,) = torch.autograd.grad(f, u, s["w"])
        return {"f": f.detach(), "grad": gu}
    if kind == "setup":
        sim = pd.pd_create(*s["desc"])
        pd.pd_build_neighbors(sim, stream=st)
        pd.pd_get_neighbors(sim, s["row_ptr"], s["col"], s["perm"], stream=st)
        dt = pd.pd_get_dt(sim)
        pd.pd_destroy(sim)
        return {"row_ptr": s["row_ptr"], "col": s["col"], "perm": s["perm"], "dt": dt}
    srv = s["server"]
    tickets = [pd.pd_submit(srv, *d, n, u0=u0, u_out=uo, v_out=vo) for (d, n, u0), (uo, vo) in zip(s["reqs"], s["out"])]
    for t in tickets:
        pd.pd_wait(srv, t, 60.0)
    return s["out"]


def work(case):
    """Every input read and every output written once, and the operations of every bond."""
    c, kind = case, case["kind"]
    if kind == "serve":
        rs = _requests(c, 0)
        return {"bytes": sum(3.0 * u0.nbytes for _, u0 in rs),
                "flops": float(sum(_bonds_about(r.grid.n[:r.grid.dim], r.grid.m) * r.steps
                                   * BOND_FLOPS["lps" if r.mat.model == wk.LPS else "pmb"] for r, _ in rs))}
    n, bonds, dim = c["nx"] * c["ny"] * c.get("nz", 1), _bonds(dict(c, nz=c.get("nz", 1))), _dim(c)
    if kind == "setup":
        return {"bytes": 4.0 * bonds + 16.0 * n, "flops": float(bonds)}
    if kind == "grad":
        return {"bytes": 4.0 * 8 * dim * n, "flops": 30.0 * bonds + 45.0 * bonds}
    if kind == "static":
        # about 8 products a lattice side of the Krylov solve, 2D products of 8 operations a bond
        it = 8 * max(c["nx"], c["ny"])
        return {"bytes": 2.0 * 8 * dim * n, "flops": 8.0 * bonds * it}
    if kind == "host":
        return {"bytes": 3.0 * 8 * dim * n * c["steps"], "flops": float(BOND_FLOPS[c["model"]] * bonds * c["steps"])}
    return {"bytes": 4.0 * 8 * dim * n, "flops": float(BOND_FLOPS[c["model"]] * bonds * c["steps"])}


# ------------------------------------------------------------------------- exact

class _Lattice:
    """Bond sums in 64 bits over chunks of points: the neighbour of point i at offset d is i + d."""

    def __init__(self, g, mat, notch=None):
        self.g, self.mat, self.dim = g, mat, g.dim
        off = _offsets(g.dim, g.m)
        self.d = torch.tensor(off, dtype=torch.int64, device="cuda")[:, :g.dim]
        nx, ny = g.n[0], g.n[1]
        self.lin = torch.tensor([x + nx * (y + ny * z) for x, y, z in off], device="cuda")
        self.xi = self.d.double() * g.h
        self.r0 = torch.sqrt((self.d * self.d).sum(1).double()) * g.h
        delta, q = g.m * g.h, self.r0
        self.vij = torch.where(q > delta - g.h / 2, (delta + g.h / 2 - q) / g.h, torch.ones_like(q)) \
            if mat.vol_corr else torch.ones_like(q)
        E = 9 * mat.K * mat.mu / (3 * mat.K + mat.mu) if mat.model == wk.LPS else mat.E
        self.V = g.h ** 3 if g.dim == 3 else g.h ** 2 * mat.thickness
        if mat.model in (wk.NP, wk.LP):
            ball = math.pi * delta ** 2 if g.dim == 2 else 4 * math.pi * delta ** 3 / 3
            self.c = 4 * mat.psi_c * mat.psi_beta / (delta * ball)
        else:
            self.c = 18 * E / 1.5 / (math.pi * delta ** 4) if g.dim == 3 \
                else 9 * E / (math.pi * mat.thickness * delta ** 3)
        self.chunk = max(1024, (1 << 23) // len(off))
        self.xyz = _coords(g)
        self.intact = None
        if mat.s_c > 0:
            self.intact = torch.cat([self._inside(lo, hi) for lo, hi in self._chunks()])
        if notch is not None:
            self._cut(notch)
        if mat.model == wk.LPS:
            self.mw = self._sum(lambda lo, hi, ok, j: (ok * (self.r0 ** 2 * self.V * self.vij)).sum(1))

    def _chunks(self):
        n = self.g.npoints
        return [(lo, min(n, lo + self.chunk)) for lo in range(0, n, self.chunk)]

    def _inside(self, lo, hi):
        p = self.xyz[lo:hi, None, :] + self.d
        top = torch.tensor(self.g.n[:self.dim], device="cuda")
        return ((p >= 0) & (p < top)).all(2)

    def _cut(self, q):
        a = q["axis"]
        others = [b for b in range(self.dim) if b != a]
        for lo, hi in self._chunks():
            x = self.xyz[lo:hi, None, :].double()
            sa = x[..., a] - q["pos"]
            sb = sa + self.d[:, a]
            cross = sa * sb < 0
            t = -sa / torch.where(self.d[:, a] == 0, torch.ones_like(self.r0), self.d[:, a].double())
            for b in others:
                p = x[..., b] + t * self.d[:, b]
                cross &= (p >= q["lo"][b]) & (p <= q["hi"][b])
            self.intact[lo:hi] &= ~cross

    def _sum(self, fn):
        out = []
        for lo, hi in self._chunks():
            ok = self.intact[lo:hi] if self.intact is not None else self._inside(lo, hi)
            i = torch.arange(lo, hi, device="cuda")[:, None]
            out.append(fn(lo, hi, ok, torch.where(ok, i + self.lin, i)))
        return torch.cat(out)

    def dt_crit(self):
        top = self._sum(lambda lo, hi, ok, j: (ok * (self.c * self.V * self.vij / self.r0)).sum(1)).max()
        return math.sqrt(2 * self.mat.rho / float(top))

    def _bond(self, u, lo, hi, j):
        """eta, y and |y|^2 - |xi|^2 (without cancellation) of the bonds of points lo..hi."""
        e = u[j] - u[lo:hi, None, :]
        y = self.xi + e
        return e, y, (e * (y + self.xi)).sum(2)

    def _stretch(self, u, lo, hi, j):
        e, y, num = self._bond(u, lo, hi, j)
        r = torch.sqrt(num + self.r0 ** 2)
        return y, r, num / (self.r0 * (r + self.r0))

    def theta(self, u):
        def one(lo, hi, ok, j):
            y, r, s = self._stretch(u, lo, hi, j)
            return 3 / self.mw[lo:hi] * (ok * (s * self.r0 ** 2 * self.V * self.vij)).sum(1)
        return self._sum(one)

    def force(self, u, breaking=True):
        mat = self.mat
        th = self.theta(u) if mat.model == wk.LPS else None
        inner = (self.d * self.d).sum(1) < self.g.m ** 2

        def one(lo, hi, ok, j):
            if mat.model in (wk.NP, wk.LP):
                S = ((u[j] - u[lo:hi, None, :]) * self.xi).sum(2) / self.r0 ** 2
                w = self.c * self.V * self.vij * inner * ok * S / self.r0
                if mat.model == wk.NP:
                    w = w * torch.exp(-mat.psi_beta * self.r0 * S * S)
                return (w[..., None] * self.xi).sum(1)
            y, r, s = self._stretch(u, lo, hi, j)
            if mat.model == wk.LPS:
                m = self.mw
                t = ((3 * mat.K - 5 * mat.mu) * self.r0 * (th / m)[lo:hi, None]
                     + 15 * mat.mu * (s * self.r0) / m[lo:hi, None]
                     + (3 * mat.K - 5 * mat.mu) * self.r0 * (th / m)[j] + 15 * mat.mu * (s * self.r0) / m[j])
                w = t * self.V * self.vij / r
            else:
                if self.intact is not None and breaking:
                    ok = ok & ~(s > mat.s_c)
                    self.intact[lo:hi] = ok
                w = self.c * self.V * self.vij * s / r
            return ((w * ok)[..., None] * y).sum(1)
        return self._sum(one)

    def tangent(self, u, w):
        def one(lo, hi, ok, j):
            y, r, s = self._stretch(u, lo, hi, j)
            n = y / r[..., None]
            dw = w[j] - w[lo:hi, None, :]
            nd = (n * dw).sum(2)
            k = ok * (self.c * self.V * self.vij)
            return ((k * nd * (1 / self.r0 - s / r))[..., None] * n + (k * s / r)[..., None] * dw).sum(1)
        return self._sum(one)

    def energy(self, u, v):
        mat = self.mat
        th = self.theta(u) if mat.model == wk.LPS else None
        inner = (self.d * self.d).sum(1) < self.g.m ** 2

        def one(lo, hi, ok, j):
            k = ok * (self.V * self.vij)
            if mat.model in (wk.NP, wk.LP):
                S = ((u[j] - u[lo:hi, None, :]) * self.xi).sum(2) / self.r0 ** 2
                x = self.r0 * S * S
                psi = -torch.expm1(-mat.psi_beta * x) / mat.psi_beta if mat.model == wk.NP else x
                return (k * inner * psi).sum(1) * self.c / 4
            y, r, s = self._stretch(u, lo, hi, j)
            if mat.model == wk.LPS:
                ed = s * self.r0 - th[lo:hi, None] * self.r0 / 3
                return mat.K * th[lo:hi] ** 2 / 2 + 15 * mat.mu / (2 * self.mw[lo:hi]) * (k * ed * ed).sum(1)
            return (k * s * s * self.r0).sum(1) * self.c / 4
        return float(mat.rho * (v * v).sum() * self.V / 2), float(self._sum(one).sum() * self.V)


def _explicit(lat, u, v, steps, dt, kind=None, val=None):
    """Velocity-Verlet with collars: the states after each step, v at the last one."""
    rho = lat.mat.rho
    vel = kind == pd.PD_BC_VELOCITY if kind is not None else None
    dis = kind == pd.PD_BC_DISPLACEMENT if kind is not None else None

    def held(v):
        return v if kind is None else torch.where(vel, val, torch.where(dis, torch.zeros_like(v), v))

    us = []
    for k in range(steps):
        v = held(v + (dt if k else dt / 2) * lat.force(u) / rho)
        u = u + dt * v
        if kind is not None:
            u = torch.where(dis, val, u)
        us.append(u)
    return us, held(v + dt / 2 * lat.force(u) / rho)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "serve":
        out = []
        for r, u0 in _requests(c, seed):
            lat = _Lattice(r.grid, r.mat)
            u = torch.from_numpy(u0).cuda()
            us, v = _explicit(lat, u, torch.zeros_like(u), r.steps, 0.5 * lat.dt_crit())
            out.append((us[-1].cpu().numpy(), v.cpu().numpy()))
        return out
    g, mat = _grid(c), _material(c)
    if kind == "setup":
        mat.rho *= np.random.default_rng(seed).uniform(0.9, 1.1)
        return {"row_ptr": None, "col": None, "perm": None, "dt": 0.5 * _Lattice(g, mat).dt_crit()}
    lat = _Lattice(g, mat, _notch(c) if c.get("breaking") else None)
    if kind == "grad":
        u, w = _grad_inputs(c, g, seed)
        return {"f": lat.force(u), "grad": lat.tangent(u, w)}
    if kind == "static":
        return {"u": _static(lat, *_clamped(c, g, _strain(seed))), "converged": None}
    u0, v0, k, v = _initial(c, g, seed)
    if kind == "host":
        u1, v1 = _initial(c, g, seed + 7919)[:2]
        dt = 0.5 * lat.dt_crit()
        us = [_explicit(lat, a, b, 1, dt)[0][0].cpu() for a, b in ((u0, v0), (u1, v1))]
        return [us[k % 2] for k in range(c["steps"])]
    dt = _run(c)["dt"] or 0.5 * lat.dt_crit()
    us, vel = _explicit(lat, u0, v0, c["steps"], dt, k, v)
    out = {"u": us[-1], "v": vel}
    if c["energy"]:
        out["kinetic"], out["strain"] = lat.energy(us[-1], vel)
    return out


def _static(lat, kind, val):
    """Newton on f(u) = 0 with the prescribed displacements held, each step by conjugate gradients."""
    free = (kind == 0).double()
    u = val.clone()
    r = lat.force(u) * free
    stop = 1e-13 * float(r.norm())
    for _ in range(6):
        if float(r.norm()) <= stop:
            break
        x, q, p = torch.zeros_like(u), r.clone(), r.clone()
        rr = (q * q).sum()
        goal = float(rr) * 1e-26
        for it in range(4000):
            Ap = -lat.tangent(u, p) * free
            a = rr / (p * Ap).sum()
            x = x + a * p
            q = q - a * Ap
            new = (q * q).sum()
            if it % 20 == 0 and float(new) < goal:
                break
            p = q + (new / rr) * p
            rr = new
        u = u + x
        r = lat.force(u) * free
    return u
