"""What a program that uses this framework has it do, as cases to be timed.

Kinds of case:

- ``run``      one grid: some steps, then the state and its moments read back (the solver's own loop,
               in both storage types, with the optional terms and time schemes);
- ``batch``    many grids stepped together (a parameter sweep, the surrogate's training runs), then
               every grid's moments and distribution;
- ``restart``  one grid set to a new point of a scan from host arrays (fields, SEE, source, f, surface
               charge), its moments and f read back: what every point pays before its first step;
- ``moment``   the density moment of a distribution that the caller holds in device memory;
- ``forward``  the surrogate's predictions for a list of points;
- ``train``    epochs of the surrogate's training on a data set of host arrays.

``exact`` gives the same results by plain torch in 64 bits, from the equations of Sun et al.
(arXiv 2303.14119, Sec. 2): nothing of this framework's code is used there.
"""
import math
import random

import numpy as np
import torch

from paper_2303_14119_gb300 import fk

QE, ME, EPS0 = 1.602176634e-19, 9.1093837015e-31, 8.8541878128e-12
H_MAX, V1, V2, CFL = 20e-6, 6e7, 3e7, 0.4  # the gap, the velocity spans and the time step of every workload
K_S, X_LO, X_HI, T_FE = 1.0, 10e-6, 15e-6, 4.0
T_E, LN_LAMBDA = 2.0, 10.0  # the collision term's defaults
MOST_CELL_STEPS = 1024 * 256 * 256 * 200  # of the largest listed run


def listed():
    point = dict(Ey=-1e6, delta_max=3.0, A_max=400.0, T_se=2.0, J=1.0)
    plain = dict(kind="run", scheme="unsplit", collisions=False, reflection=0.0)
    return [
        # the plain single-instance configuration: 64 x 48 x 48 in FP64; every step is short, so its
        # launches and its chain of reductions count
        dict(plain, name="run_small_f64", nx=64, nv1=48, nv2=48, f64=True, steps=500, **point),
        # one point of the parameter sweep stepped alone, of odd sizes (rows that need padding)
        dict(plain, name="run_sweep_point_f32", nx=321, nv1=117, nv2=117, f64=False, steps=300,
             Ey=-2.3e6, delta_max=2.6, A_max=310.0, T_se=3.1, J=1.0),
        # the full-scale configuration in both storage types
        dict(plain, name="run_full_f32", nx=1024, nv1=256, nv2=256, f64=False, steps=200, **point),
        dict(plain, name="run_full_f64", nx=1024, nv1=256, nv2=256, f64=True, steps=40, **point),
        # every term of the model on: collisions and reflection at the wall (512 x 128 x 128 is the grid
        # of the surrogate's fine runs)
        dict(plain, name="run_collisions_f32", nx=512, nv1=128, nv2=128, f64=False, steps=300,
             **dict(point, collisions=True, reflection=0.2, J=1e5)),
        # the split time scheme on the same grid
        dict(plain, name="run_strang_f32", nx=512, nv1=128, nv2=128, f64=False, steps=150,
             **dict(point, scheme="strang", J=1e5)),
        # a parameter sweep: 16 grids of uneven sizes (nx 128-512, nv 64-192) as one batch
        dict(kind="batch", name="batch_sweep_f32", grids=16, nx_lo=128, nx_hi=512, nv_lo=64, nv_hi=192,
             draws=2023, J=1.0, f64=False, steps=200),
        # training runs of the surrogate: many small equal grids as one batch
        dict(kind="batch", name="batch_surrogate_f32", grids=384, nx_lo=64, nx_hi=64, nv_lo=48, nv_hi=48,
             draws=11, J=1e6, f64=False, steps=500),
        # the next point of a scan on a grid that exists: fields, yield, source, f and surface charge set
        dict(kind="restart", name="restart_f32", nx=512, nv1=128, nv2=128, f64=False,
             **dict(point, J=1e5)),
        # the density of the full-scale distribution held by the caller
        dict(kind="moment", name="moment_full_f64", nx=1024, nv1=256, nv2=256),
        # the surrogate network: triage of a sweep's worth of points, and training on 4096 runs
        dict(kind="forward", name="surrogate_forward", n_in=6, width=256, depth=3, n_out=65, n=4096,
             max_batch=512),
        dict(kind="train", name="surrogate_train", n_in=6, width=256, depth=3, n_out=65, n=4096, batch=256,
             max_batch=512, epochs=4),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _point(rng):
    """The parameters of a scan: the sweep's ranges."""
    return dict(Ey=-math.exp(rng.uniform(math.log(3e5), math.log(5e6))), delta_max=rng.uniform(2.0, 4.0),
                A_max=rng.uniform(250.0, 600.0), T_se=rng.uniform(1.0, 5.0),
                J=math.exp(rng.uniform(0.0, math.log(1e6))))


def _sizes(rng, most):
    nx, nv1, nv2 = _log(rng, 64, 1024), _log(rng, 48, 256), _log(rng, 48, 256)
    while nx * nv1 * nv2 > most:
        nx = nx // 2 + 1
    return dict(nx=nx, nv1=nv1, nv2=nv2)


def draw(rng):
    kind = rng.choice(("run", "run", "run", "run", "batch", "batch", "restart", "moment", "forward", "train"))
    if kind == "run":
        f64 = rng.random() < 0.4
        c = dict(kind=kind, f64=f64, scheme=rng.choice(("unsplit", "unsplit", "unsplit", "lie", "strang")),
                 collisions=rng.random() < 0.3, reflection=0.0, **_point(rng), **_sizes(rng, 1 << 25))
        if rng.random() < 0.3:
            c["reflection"] = rng.uniform(0.05, 0.5)
        # as many steps as keep a pass below the largest listed one's work (an FP64 step costs about six
        # FP32 ones, a split step two or three)
        cost = c["nx"] * c["nv1"] * c["nv2"] * (6 if f64 else 1) * (1 if c["scheme"] == "unsplit" else 3)
        c["steps"] = max(20, min(_log(rng, 100, 500), MOST_CELL_STEPS // (2 * cost)))
        return c
    if kind == "batch":
        small = rng.random() < 0.5
        lo = dict(nx_lo=48, nx_hi=96, nv_lo=32, nv_hi=56) if small else dict(nx_lo=128, nx_hi=512, nv_lo=64, nv_hi=160)
        return dict(kind=kind, grids=_log(rng, 32, 128) if small else _log(rng, 4, 12), draws=rng.randrange(1 << 20),
                    J=math.exp(rng.uniform(0.0, math.log(1e6))), f64=rng.random() < 0.25,
                    steps=_log(rng, 60, 200), **lo)
    if kind == "restart":
        return dict(kind=kind, f64=rng.random() < 0.5, **_point(rng), **_sizes(rng, 1 << 23))
    if kind == "moment":
        return dict(kind=kind, **_sizes(rng, 1 << 26))
    c = dict(kind=kind, n_in=rng.randint(4, 12), width=16 * rng.randint(4, 16), depth=rng.randint(1, 4),
             n_out=rng.randint(16, 128), n=_log(rng, 300, 4096), max_batch=512)
    if kind == "train":
        c.update(batch=rng.choice((64, 96, 128, 256, 500)), epochs=rng.randint(1, 3))
    return c


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _f0(shape, J, seed, dtype):
    """A distribution as a run holds one: of the injected beam's density scale, falling off with speed and
    leaning toward the anode, with seeded noise cell by cell (made on the device)."""
    nx, nv1, nv2 = shape
    scale = 1e-3 * (J / QE) / (T_FE * QE / ME) ** 1.5
    c1 = (torch.arange(nv1, device="cuda", dtype=torch.float64) + 0.5) / nv1 * 2 - 1
    c2 = (torch.arange(nv2, device="cuda", dtype=torch.float64) + 0.5) / nv2 * 2 - 1
    shape_v = torch.exp(-4 * c1[:, None] ** 2 - 2 * (c2[None, :] - 0.2) ** 2).to(dtype)
    f = torch.rand(nx, nv1, nv2, generator=_gen(seed), device="cuda", dtype=dtype)
    return f.add_(0.2).mul_(shape_v).mul_(scale)


def _pinned(shape, dtype):
    return torch.empty(shape, dtype=dtype, pin_memory=True)


def _host(t):
    h = _pinned(t.shape, t.dtype)
    h.copy_(t)
    return h


def _case_points(c):
    """The grids of a batch: sizes and parameters from the case alone."""
    rng = random.Random(c["draws"])
    out = []
    for _ in range(c["grids"]):
        nv = rng.randint(c["nv_lo"], c["nv_hi"])
        out.append(dict(_point(rng), J=c["J"], nx=rng.randint(c["nx_lo"], c["nx_hi"]), nv1=nv, nv2=nv))
    return out


def _shape(c):
    return c["nx"], c["nv1"], c["nv2"]


def _sigma0(seed):
    return 1e-9 * (1.0 + (seed % 7) / 7.0)  # C/m^2: the wall has begun to charge


def _grid(c, f64, history=4096):
    return fk.Grid(c["nx"], c["nv1"], c["nv2"], H_MAX, -V1, V1, -V2, V2, cfl=CFL,
                   precision=fk.FK_F64 if f64 else fk.FK_F32, history_capacity=history)


def _set_point(g, c):
    g.set_fields(c["Ey"])
    g.set_see(c["delta_max"], c["A_max"], K_S, c["T_se"])
    g.set_source(c["J"], X_LO, X_HI, T_FE)


def _set_f(g, host, f64):
    (g.set_f if f64 else g.set_f32)(host)


def prepare(case, seed):
    c = case
    if c["kind"] == "run":
        dtype = torch.float64 if c["f64"] else torch.float32
        g = _grid(c, c["f64"])
        _set_point(g, c)
        if c["collisions"]:
            g.set_collisions(T_E, LN_LAMBDA, True)
        if c["reflection"]:
            g.set_reflection(c["reflection"])
        if c["scheme"] != "unsplit":
            g.set_scheme(dict(lie=fk.FK_SCHEME_LIE, strang=fk.FK_SCHEME_STRANG)[c["scheme"]])
        host = _host(_f0(_shape(c), c["J"], seed, dtype))
        _set_f(g, host.numpy(), c["f64"])
        g.set_surface_charge(_sigma0(seed))
        return dict(case=c, grid=g, out=host.numpy(), keep=host)  # f is read back into the same host array
    if c["kind"] == "batch":
        dtype = torch.float64 if c["f64"] else torch.float32
        points = _case_points(c)
        grids = []
        for p in points:
            g = _grid(p, c["f64"])
            _set_point(g, p)
            grids.append(g)
        with fk.Batch(grids) as b:  # the schedule, found on these grids before their runs begin
            b.autotune(2)
            b.sync()
            chunks = b.chunks()
        f = _pinned((sum(p["nx"] * p["nv1"] * p["nv2"] for p in points),), dtype)  # all the grids' cells
        parts, at = [], 0
        for i, (g, p) in enumerate(zip(grids, points)):
            h = f[at:at + p["nx"] * p["nv1"] * p["nv2"]].view(_shape(p))
            at += h.numel()
            h.copy_(_f0(_shape(p), p["J"], seed * 1009 + i, dtype))
            _set_f(g, h.numpy(), c["f64"])
            g.set_surface_charge(_sigma0(seed + i))
            parts.append(h.numpy())
        b = fk.Batch(grids)
        b.set_chunks(chunks)
        nx = sum(p["nx"] for p in points)
        return dict(case=c, batch=b, f=f, parts=parts, n_e=np.empty(nx), Ex=np.empty(nx))
    if c["kind"] == "restart":
        dtype = torch.float64 if c["f64"] else torch.float32
        f = _host(_f0(_shape(c), c["J"], seed, dtype).double())
        out = _pinned(f.shape, torch.float64)
        return dict(case=c, grid=_grid(c, c["f64"]), f=f.numpy(), out=out.numpy(), keep=(f, out),
                    sigma=_sigma0(seed))
    if c["kind"] == "moment":
        f = _f0(_shape(c), 1.0, seed, torch.float64)
        return dict(case=c, f=f, n_e=torch.empty(c["nx"], dtype=torch.float64, device="cuda"))
    X, T, w, params = _net_inputs(c, seed)
    net = fk.Mlp(c["n_in"], c["width"], c["depth"], c["n_out"], c["max_batch"])
    net.set_params(params)
    return dict(case=c, net=net, X=X, T=T, w=w)


def _net_inputs(c, seed):
    """Normalised features and targets (smooth in the features, as the charge histories are) and a
    network's initial weights, on the host."""
    rng = np.random.default_rng(seed)
    X = rng.uniform(-1.7, 1.7, (c["n"], c["n_in"])).astype(np.float32)
    A = rng.normal(0.0, 0.7, (c["n_in"], c["n_out"])).astype(np.float32)
    T = np.tanh(X @ A).astype(np.float32)
    w = np.ones(c["n_out"], dtype=np.float32)
    w[-1] = 16.0
    dims = [c["n_in"]] + [c["width"]] * c["depth"] + [c["n_out"]]
    parts = []
    for q in range(len(dims) - 1):
        parts.append(rng.normal(0.0, math.sqrt(2.0 / dims[q]), dims[q + 1] * dims[q]))
        parts.append(np.zeros(dims[q + 1]))
    return X, T, w, np.concatenate(parts).astype(np.float32)


# ------------------------------------------------------------------ one pass
def _profile(a, f64):
    """n_e and E_x of an FP32 grid are kept beside its f in the same storage type."""
    return a if f64 else a.astype(np.float32)


def run(state):
    c = state["case"]
    if c["kind"] == "run":
        g = state["grid"]
        g.step(c["steps"])
        n_e, Ex, gpe, gsee = g.moments()
        sigma = g.surface_charge()
        f = (g.get_f if c["f64"] else g.get_f32)(state["out"])
        return dict(f=f, n_e=_profile(n_e, c["f64"]), Ex=_profile(Ex, c["f64"]), gamma_pe=gpe, gamma_see=gsee,
                    sigma=sigma)
    if c["kind"] == "batch":
        b = state["batch"]
        b.step(c["steps"])
        sigma, gpe, gsee, n_e, Ex = b.moments(state["n_e"], state["Ex"])
        for g, part in zip(b.grids, state["parts"]):
            (g.get_f if c["f64"] else g.get_f32)(part)
        return dict(f=state["f"], n_e=_profile(n_e, c["f64"]), Ex=_profile(Ex, c["f64"]),
                    gamma_pe=_profile(gpe, c["f64"]), gamma_see=_profile(gsee, c["f64"]), sigma=_profile(sigma, c["f64"]))
    if c["kind"] == "restart":
        g = state["grid"]
        _set_point(g, c)
        g.set_f(state["f"])
        g.set_surface_charge(state["sigma"])
        n_e, Ex, gpe, gsee = g.moments()
        return dict(f=g.get_f(state["out"]), n_e=n_e, Ex=Ex, gamma_pe=gpe, gamma_see=gsee)
    if c["kind"] == "moment":
        fk.fk_density_moment_noalloc(state["f"].data_ptr(), c["nx"], c["nv1"], c["nv2"], 2 * V1 / c["nv1"],
                                     2 * V2 / c["nv2"], state["n_e"].data_ptr(),
                                     torch.cuda.current_stream().cuda_stream or None)
        return state["n_e"]
    if c["kind"] == "forward":
        return state["net"].forward(state["X"])
    losses = state["net"].train(state["X"], state["T"], state["w"], batch=c["batch"], epochs=c["epochs"], lr=1e-3,
                                seed=5)
    return dict(params=state["net"].get_params(), losses=[float(v) for v in losses])


# ------------------------------------------------------------------ what it cannot do without
def _net_params(c):
    dims = [c["n_in"]] + [c["width"]] * c["depth"] + [c["n_out"]]
    return sum(a * b + b for a, b in zip(dims, dims[1:]))


def work(case):
    """Bytes: for steps, one read and one write of f for each, and the state once to the host at the end.
    Operations: eight for the upwind update of a cell, four more for the collision term."""
    c = case
    if c["kind"] in ("run", "batch"):
        esize = 8 if c["f64"] else 4
        points = [c] if c["kind"] == "run" else _case_points(c)
        cells = sum(p["nx"] * p["nv1"] * p["nv2"] for p in points)
        planes = sum(p["nx"] for p in points)
        return dict(bytes=c["steps"] * cells * 2 * esize + cells * esize + 2 * planes * 8,
                    flops=c["steps"] * cells * (12 if c.get("collisions") else 8))
    cells = c["nx"] * c["nv1"] * c["nv2"] if "nx" in c else 0
    if c["kind"] == "restart":  # f in from the host, read once for its moments, and out to the host
        return dict(bytes=cells * (8 + 8 + (8 if c["f64"] else 4)), flops=cells)
    if c["kind"] == "moment":
        return dict(bytes=cells * 8 + c["nx"] * 8, flops=cells)
    p = _net_params(c)
    if c["kind"] == "forward":
        return dict(bytes=4 * c["n"] * (c["n_in"] + c["n_out"]) + 4 * p, flops=2 * p * c["n"])
    return dict(bytes=4 * c["epochs"] * c["n"] * (c["n_in"] + c["n_out"]) + 8 * p, flops=6 * p * c["n"] * c["epochs"])


# ------------------------------------------------------------------ the same in 64 bits, by plain torch
class _Model:
    """Grids of one shape, all the arrays with one leading axis for the grids (Sec. 2 of the paper)."""

    def __init__(self, points, shape, collisions=False, reflection=0.0):
        G, (nx, nv1, nv2) = len(points), shape
        par = lambda k: torch.tensor([p[k] for p in points], device="cuda", dtype=torch.float64).view(G, 1, 1)  # noqa: E731
        self.dx, self.dv1, self.dv2 = H_MAX / nx, 2 * V1 / nv1, 2 * V2 / nv2
        self.dt, self.dvv, self.refl = CFL * self.dx / V1, self.dv1 * self.dv2, reflection
        v1 = (-V1 + (torch.arange(nv1, device="cuda", dtype=torch.float64) + 0.5) * self.dv1).view(1, nv1, 1)
        v2 = (-V2 + (torch.arange(nv2, device="cuda", dtype=torch.float64) + 0.5) * self.dv2).view(1, 1, nv2)
        self.v1, self.i0 = v1, int((v1 <= 0).sum())
        self.cx = (v1 * self.dt / self.dx).view(1, 1, nv1, 1)
        vv = v1 ** 2 + v2 ** 2
        al2 = torch.atan((v2 / v1).abs()) ** 2
        z = 1.284 * (0.5 * ME * vv / QE) / (par("A_max") * (1 + K_S * al2 / math.pi))
        delta = 1.526 * par("delta_max") * (1 + K_S * al2 / (2 * math.pi)) * (1 - torch.exp(-z ** 1.725)) / z ** 0.725
        self.delta = torch.where(v1 < 0, delta, torch.zeros_like(delta))
        g = torch.exp(-ME * vv / (2 * par("T_se") * QE)) * (v1 > 0)
        self.gse = g / ((v1 * g).sum((1, 2), keepdim=True) * self.dvv)
        s = torch.exp(-ME * vv / (2 * T_FE * QE)) * (v2 > 0)
        x = (np.arange(nx) + 0.5) * self.dx
        band = np.nonzero((x >= X_LO) & (x <= X_HI))[0]
        self.b0, self.b1 = int(band[0]), int(band[-1]) + 1
        self.src = (self.dt * par("J") / QE / ((self.b1 - self.b0) * self.dx) * s / (s.sum() * self.dvv))[:, None]
        self.c2 = (-QE / ME * par("Ey") * self.dt / self.dv2)[:, None]
        T = T_E * QE
        self.nu = self.dt * QE ** 4 * LN_LAMBDA / (12 * math.pi ** 1.5 * EPS0 ** 2 * math.sqrt(ME) * T ** 1.5) if collisions else 0.0
        m = torch.exp(-ME * v1 ** 2 / (2 * T)) * torch.exp(-ME * v2 ** 2 / (2 * T))
        self.m = (m / (m.sum() * self.dvv))[:, None]

    def density(self, f):
        return f.sum((2, 3)) * self.dvv

    def field(self, n, sigma):
        below = torch.cumsum(n, 1) - 0.5 * n
        return sigma[:, None] / (2 * EPS0) - QE / EPS0 * self.dx * below

    def fluxes(self, f):
        g = (-self.v1 * f[:, 0])[:, :self.i0]
        return g.sum((1, 2)) * self.dvv, (self.delta[:, :self.i0] * g).sum((1, 2)) * self.dvv * (1 - self.refl)

    def add_x(self, f, out, gsee, part):
        i0, ax = self.i0, part * self.cx.abs()
        out -= ax * f
        out[:, :-1, :i0] += ax[:, :, :i0] * f[:, 1:, :i0]
        out[:, 1:, i0:] += ax[:, :, i0:] * f[:, :-1, i0:]
        inflow = gsee.view(-1, 1, 1) * self.gse
        if self.refl:
            inflow = inflow + self.refl * f[:, 0].flip(1)
        out[:, 0, i0:] += ax[:, 0, i0:] * inflow[:, i0:]

    def add_v(self, f, out, n, Ex):
        c1 = (-QE / ME * self.dt / self.dv1 * Ex)[:, :, None, None]
        up, down = c1.clamp(min=0), (-c1).clamp(min=0)
        nu = (self.nu * n)[:, :, None, None]
        out -= (up + down + self.c2 + nu) * f
        out[:, :, 1:] += up * f[:, :, :-1]
        out[:, :, :-1] += down * f[:, :, 1:]
        out[..., 1:] += self.c2 * f[..., :-1]
        out[:, self.b0:self.b1] += self.src
        if self.nu:
            out += (nu * n[:, :, None, None]) * self.m

    def steps(self, f, sigma, count, scheme):
        n = self.density(f)
        for _ in range(count):
            Ex, (gpe, gsee) = self.field(n, sigma), self.fluxes(f)
            charge = gsee - (1 - self.refl) * gpe
            if scheme == "unsplit":
                g = f.clone()
                self.add_x(f, g, gsee, 1.0)
                self.add_v(f, g, n, Ex)
                f = g
            else:
                half = 0.5 if scheme == "strang" else 1.0
                g = f.clone()
                self.add_x(f, g, gsee, half)
                f = g.clone()
                self.add_v(g, f, n, Ex)
                if scheme == "strang":
                    gpe, gsee = self.fluxes(f)
                    charge = 0.5 * charge + 0.5 * (gsee - (1 - self.refl) * gpe)
                    g = f.clone()
                    self.add_x(f, g, gsee, 0.5)
                    f = g
            sigma = sigma + QE * self.dt * charge
            n = self.density(f)
        gpe, gsee = self.fluxes(f)
        return dict(f=f, n_e=n, Ex=self.field(n, sigma), gamma_pe=gpe, gamma_see=gsee, sigma=sigma)


def exact(case, seed):
    c = case
    if c["kind"] in ("run", "restart"):
        f = _f0(_shape(c), c["J"], seed, torch.float64 if c["f64"] else torch.float32).double()[None]
        m = _Model([c], _shape(c), c.get("collisions", False), c.get("reflection", 0.0))
        sigma = torch.tensor([_sigma0(seed)], device="cuda", dtype=torch.float64)
        r = m.steps(f, sigma, c.get("steps", 0), c.get("scheme", "unsplit"))
        r = dict(f=r["f"][0], n_e=r["n_e"][0], Ex=r["Ex"][0], gamma_pe=float(r["gamma_pe"]),
                 gamma_see=float(r["gamma_see"]), sigma=float(r["sigma"]))
        if c["kind"] == "restart":
            del r["sigma"]
        return {k: v if isinstance(v, float) else v.cpu() for k, v in r.items()}
    if c["kind"] == "batch":
        points, dtype = _case_points(c), torch.float64 if c["f64"] else torch.float32
        parts = [None] * len(points)
        for shape in sorted(set(map(_shape, points))):
            at = [i for i, p in enumerate(points) if _shape(p) == shape]
            f = torch.stack([_f0(shape, points[i]["J"], seed * 1009 + i, dtype).double() for i in at])
            sigma = torch.tensor([_sigma0(seed + i) for i in at], device="cuda", dtype=torch.float64)
            r = _Model([points[i] for i in at], shape).steps(f, sigma, c["steps"], "unsplit")
            for q, i in enumerate(at):
                parts[i] = {k: v[q].reshape(-1).cpu() for k, v in r.items()}
        return {k: torch.cat([p[k] for p in parts]).numpy() for k in ("f", "n_e", "Ex", "gamma_pe", "gamma_see", "sigma")}
    if c["kind"] == "moment":
        return _f0(_shape(c), 1.0, seed, torch.float64).sum((1, 2)) * (2 * V1 / c["nv1"]) * (2 * V2 / c["nv2"])
    if c["kind"] == "train":
        return None  # an Adam step turns on the sign of every gradient: no 64-bit run stays beside it
    X, T, w, params = _net_inputs(c, seed)
    y, at = torch.from_numpy(X).cuda().double(), 0
    dims = [c["n_in"]] + [c["width"]] * c["depth"] + [c["n_out"]]
    for q, (a, b) in enumerate(zip(dims, dims[1:])):
        W = torch.from_numpy(params[at:at + a * b]).cuda().double().view(b, a)
        at += a * b + b  # the biases begin as zeros
        y = y @ W.T
        if q < len(dims) - 2:
            y = 0.5 * y * (1 + torch.erf(y / math.sqrt(2.0)))
    return y.cpu().numpy()
