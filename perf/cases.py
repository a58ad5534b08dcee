"""The workloads whose speed this framework is judged by, and how each is prepared, run and checked.

A case is a dict of plain values; its "kind" says which public entry point it goes through:

  step       Integrator: a new state is written into the integrator's Psi (as a chunked driver or the
             RK4 window pool does) and advanced by `steps` RK4 steps
  observe    Integrator.mass() and Integrator.energy() of a state, as at the end of every frame
  batch      BatchIntegrator.step() over many uneven 2D runs
  sur_fwd    Surrogate.forward() with the raw output's masses
  sur_grad   Surrogate.gradients(): forward, loss, backward-data and weight gradients

Sizes come from the workloads of paper_1203_1263_gb300/workloads.py, from the tests and from bench.py.
Initial states are the workloads' (bright and dark solitons, vortices, vortex rings, a trapped vortex
line, Gaussian humps and packets), built with torch on the GPU.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1203_1263_gb300.integrator import BatchIntegrator, Integrator, max_dt
from paper_1203_1263_gb300.surrogate import Surrogate

DILATIONS = (1, 2, 4, 8, 4, 1)   # the 6-layer, 64-channel network of bench.py
CHANNELS = 64


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _step(name, field, shape, dtype, bc, order, steps):
    s = tuple(shape) + (1,) * (3 - len(shape))
    return dict(name=name, kind="step", field=field, dims=len(shape), n0=s[0], n1=s[1], n2=s[2], dtype=dtype, bc=bc,
                order=order, steps=steps)


def listed():
    return [
        # the 1D bright soliton run (2001 sites, Dirichlet, FP64): thousands of tiny, dependent steps
        _step("soliton1d_f64", "bright", (2001,), "c128", "dirichlet", 4, 64),
        # one 32-step window of the focusing 2D problem: training data, window checks and fallback of the surrogate
        _step("window2d_f64", "humps", (256, 256), "c128", "dirichlet", 4, 32),
        # the dark vortex of the 2D timing table at 10^6 sites, FP32 and central differences as that table runs it
        _step("vortex2d_f32", "vortex", (1000, 1000), "c64", "msd", 2, 32),
        # the smallest 3D grid of the timing tables: a step is latency and launches
        _step("ring3d_small_f64", "ring", (21, 21, 21), "c128", "msd", 4, 64),
        # the paper's headline grid, odd sizes, one 56-step frame, FP64
        _step("trap87_f64", "trap", (203, 87, 87), "c128", "msd", 4, 56),
        # the same frame in the precision form: FP32 stages, FP64 master and accumulator
        _step("trap87_mixed", "trap", (203, 87, 87), "c64_acc64", "msd", 4, 56),
        # the large trap-vortex grid, FP64: the plain method at scale
        _step("trap512_f64", "trap", (512, 256, 256), "c128", "msd", 4, 16),
        # the same grid in FP32
        _step("trap512_f32", "trap", (512, 256, 256), "c64", "msd", 4, 16),
        # many uneven 2D runs advanced together (the batch workload's recipe, 96 of its runs)
        dict(name="batch96", kind="batch", runs=96, nmin=64, nmax=1024, steps=16),
        # mass and energy of a large FP64 state: the conserved quantities of every frame
        dict(name="observe256_f64", kind="observe", field="trap", dims=3, n0=256, n1=256, n2=256, dtype="c128", bc="msd",
             order=4),
        # inference of the learned surrogate on a full batch
        dict(name="surrogate_forward", kind="sur_fwd", nb=16, n0=256, n1=256),
        # one gradient of its training
        dict(name="surrogate_gradients", kind="sur_grad", nb=16, n0=256, n1=256),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


_RANGE = {1: (1e3, 3e6), 2: (961, 3e6), 3: (9261, 33e6)}   # sites, per dimension: the timing tables to the large grids
_FIELDS = {1: ("bright", "dark"), 2: ("humps", "vortex", "trap"), 3: ("trap", "ring", "vortex")}


def _draw_grid(rng, dims, lo, hi):
    """Extents of a grid of about log-uniform size, sides uneven by up to a factor of about two."""
    total = _log(rng, lo, hi)
    side = total ** (1.0 / dims)
    w = [_log(rng, 0.75, 1.5) for _ in range(dims)]
    g = math.prod(w) ** (1.0 / dims)
    n = [max(16, int(round(side * x / g))) for x in w]
    return n + [1] * (3 - dims)


def draw(rng):
    kind = rng.choice(["step"] * 12 + ["observe"] * 2 + ["batch"] * 2 + ["sur_fwd", "sur_grad"])
    if kind in ("step", "observe"):
        dims = rng.choice([1, 2, 2, 3, 3, 3])
        lo, hi = _RANGE[dims]
        if kind == "observe":
            hi = min(hi, 17e6)
        n0, n1, n2 = _draw_grid(rng, dims, lo, hi)
        dtype = rng.choice(["c128", "c128", "c64", "c64_acc64"])
        field = rng.choice(_FIELDS[dims])
        bc = rng.choice(["dirichlet", "l0", "periodic"] if field in ("bright", "humps") else ["msd", "msd", "l0"])
        case = dict(kind=kind, field=field, dims=dims, n0=n0, n1=n1, n2=n2, dtype=dtype, bc=bc, order=rng.choice([2, 4, 4]))
        if kind == "step":
            cap = 12 * 33.5e6 * (1.0 if dtype == "c128" else 2.0) / (n0 * n1 * n2)
            case["steps"] = max(1, int(_log(rng, 1, max(1.01, min(100.0, cap)))))
        return case
    if kind == "batch":
        nmin = int(_log(rng, 48, 200))
        nmax = int(_log(rng, 300, 1024))
        runs = max(8, int(_log(rng, 8, 90) * min(1.0, (800.0 / nmax) ** 2)))
        return dict(kind="batch", runs=runs, nmin=nmin, nmax=nmax, steps=int(_log(rng, 1, 16.99)))
    side = lambda: int(_log(rng, 48, 256))  # noqa: E731
    return dict(kind=kind, nb=rng.randint(1, 16), n0=side(), n1=side())


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
F64 = torch.float64


def _uniform(seed, n):
    return np.random.default_rng(int(seed)).random(n)


def _axes(shape, h):
    out = []
    for k, n in enumerate(shape):
        x = (torch.arange(n, dtype=F64, device="cuda") - 0.5 * (n - 1)) * h
        out.append(x.reshape([-1 if j == k else 1 for j in range(len(shape))]))
    return out


def _noise(psi, seed, size=1e-3):
    """A seeded Gaussian phase noise on every site, as on the trapped vortex line's state."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    xi = torch.randn(psi.shape, dtype=F64, device="cuda", generator=g)
    return psi * torch.polar(torch.ones_like(xi), size * xi)


def _shape(c):
    return (c["n0"], c["n1"], c["n2"])[:c["dims"]]


def _problem(c, seed):
    """(psi0 complex128, V float64 or None, h, a, s, largest s|psi|^2) of a grid case."""
    shape, d, u = _shape(c), c["dims"], _uniform(seed, 32)
    f = c["field"]
    if f in ("bright", "dark"):
        h = 0.05 if f == "bright" else 0.1
        (x,) = _axes(shape, h)
        if f == "bright":
            x = x - 0.2 * shape[0] * h * (u[0] - 0.5)
            v = 0.3 + 0.4 * u[1]
            psi = torch.polar(math.sqrt(2.0) / torch.cosh(x), 0.5 * v * x)
            return psi, None, h, 1.0, 1.0, 2.0
        v = 0.3 + 0.4 * u[1]
        amp = torch.tanh(x / math.sqrt(2.0))
        return _noise(amp * torch.polar(torch.ones_like(x), 0.5 * v * x), seed), None, h, 1.0, -1.0, 1.0
    if f == "humps":
        h = 0.2
        y, x = _axes(shape, h)
        psi = torch.zeros(shape, dtype=torch.complex128, device="cuda")
        for j in range(1 + int(u[0] * 4)):
            q = u[1 + 7 * j:8 + 7 * j]
            amp, w, ang = 0.5 + q[0], 0.7 + 0.5 * q[1], 2 * math.pi * q[5]
            x0, y0 = 0.6 * (shape[1] - 1) * h * (q[2] - 0.5), 0.6 * (shape[0] - 1) * h * (q[3] - 0.5)
            env = amp * torch.exp(-((x - x0) ** 2 + (y - y0) ** 2) / (2 * w * w))
            psi += torch.polar(env, q[4] * (math.cos(ang) * x + math.sin(ang) * y))
        return psi, None, h, 1.0, 1.0, 4.0
    if f == "trap":
        # harmonic trap, Thomas-Fermi cloud (zero outside), a vortex line along the first axis, phase noise
        h = 17.2 / (shape[-1] - 1) if d == 3 else 25.0 / (max(shape) - 1)
        ax = _axes(shape, h)
        y, x = ax[-2], ax[-1]
        V = 0.5 * (x * x + y * y)
        if d == 3:
            V = V + 0.125 * ax[0] ** 2
        V = V.expand(shape).contiguous()
        a, mu = 0.5, 4.0
        rho = torch.clamp(mu - V, min=0.0)
        r = torch.sqrt((x - u[0] + 0.5) ** 2 + (y - u[1] + 0.5) ** 2)
        amp = torch.sqrt(rho) * torch.tanh(r * math.sqrt(mu / (2 * a)))
        psi = torch.polar(torch.ones_like(amp), torch.atan2(y - u[1] + 0.5, x - u[0] + 0.5).expand(shape)) * amp
        return _noise(psi, seed), V, h, a, -1.0, mu
    if f == "vortex":
        h = 0.25
        ax = _axes(shape, h)
        y, x = ax[-2] - 2 * h * (u[0] - 0.5), ax[-1] - 2 * h * (u[1] - 0.5)
        amp = torch.tanh(torch.sqrt(x * x + y * y) / math.sqrt(2.0))
        psi = torch.polar(amp, torch.atan2(y, x)).expand(shape)
        return _noise(psi, seed), None, h, 1.0, -1.0, 1.0
    # a vortex ring of radius 5 about the first axis with its back-flow
    h, R = 1.5 if max(shape) < 40 else 0.5, 5.0
    z, y, x = _axes(shape, h)
    z = z - h * (u[0] - 0.5)
    rc = torch.sqrt(x * x + y * y)
    k = 1.0 / math.sqrt(2.0)
    amp = torch.tanh(k * torch.sqrt((rc - R) ** 2 + z * z)) * torch.tanh(k * torch.sqrt((rc + R) ** 2 + z * z))
    Rs = R * k
    v = math.sqrt(2.0) * (math.log(8 * Rs) - 0.615) / (2 * Rs)
    psi = torch.polar(amp, torch.atan2(z, rc - R) - torch.atan2(z, rc + R) + 0.5 * v * z)
    return _noise(psi, seed), None, h, 1.0, -1.0, 1.0


def _dt(c, V, h, a, srho):
    vmax = 0.0 if V is None else float(V.abs().max())
    return 0.8 * max_dt(c["dims"], h, a, c["order"], vmax, srho)


def _batch_runs(c, seed):
    """The batch workload's recipe: uneven sides, a, s, trap or none, order 2 or 4, seeded Gaussian packets
    (the sides are the case's own, the same for every seed)."""
    out = []
    for r in range(c["runs"]):
        u = _uniform(int(seed) * 100003 + r, 16)
        side = _uniform(4 + 16 * r, 1)[0]
        n = c["nmin"] + min(int(side * (c["nmax"] - c["nmin"] + 1)), c["nmax"] - c["nmin"])
        h, a, s = 0.25, 0.5 + 0.5 * u[1], 1.0 if u[2] < 0.5 else -1.0
        order, w = 4 if u[5] < 0.5 else 2, 2.0 + 6.0 * u[6]
        half = 0.25 * (n - 1) * h
        ang = 2 * math.pi * u[10]
        amp = math.sqrt(0.8 * 11.70 * a / (math.pi * w * w)) if s > 0 else 1.0
        y, x = _axes((n, n), h)
        env = amp * torch.exp(-((x - half * (2 * u[7] - 1)) ** 2 + (y - half * (2 * u[8] - 1)) ** 2) / (2 * w * w))
        psi = torch.polar(env, u[9] * (math.cos(ang) * x + math.sin(ang) * y)).to(torch.complex64)
        V = None
        if u[3] < 0.5:
            om = 0.05 + 0.15 * u[4]
            V = (0.5 * om * om * (x * x + y * y)).to(torch.float32)
        vmax = 0.0 if V is None else float(V.abs().max())
        out.append(dict(psi0=psi, V=V, h=h, a=a, s=s, order=order, bc="dirichlet",
                        dt=0.8 * max_dt(2, h, a, order, vmax, amp * amp)))
    return out


def _states(c, seed, salt):
    g = dict(dims=2, n0=c["n0"], n1=c["n1"], n2=1, field="humps")
    return torch.stack([_problem(g, int(seed) * 1009 + salt + i)[0] for i in range(c["nb"])]).to(torch.complex64)


def _pair(c, seed):
    """States and targets that differ from them as one window of the equation makes them differ."""
    x = _states(c, seed, 0)
    return x, x * torch.polar(torch.ones_like(x.real), 0.16 * x.abs() ** 2) + 0.02 * _states(c, seed, 500)


def _params(seed):
    """A network's parameters, layer by layer W [cout][9][cin] then b [cout], uniform in +-1 / sqrt(9 cin)."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 7)
    parts = []
    for l in range(len(DILATIONS)):
        ci = 4 if l == 0 else CHANNELS
        co = 2 if l == len(DILATIONS) - 1 else CHANNELS
        parts.append((2.0 * torch.rand(co * 9 * ci + co, device="cuda", generator=g) - 1.0) / math.sqrt(9.0 * ci))
    return torch.cat(parts)


def prepare(case, seed):
    c = case
    if c["kind"] in ("step", "observe"):
        psi, V, h, a, s, srho = _problem(c, seed)
        g = Integrator(psi, h, a, s, V, c["bc"], c["order"], c["dtype"])
        return dict(case=c, g=g, start=psi.to(g.psi.dtype), dt=_dt(c, V, h, a, srho))
    if c["kind"] == "batch":
        runs = _batch_runs(c, seed)
        for r in runs:
            r["psi0"] = r["psi0"].cpu().numpy()
            r["V"] = None if r["V"] is None else r["V"].cpu().numpy()
        return dict(case=c, b=BatchIntegrator(runs))
    x, y = _pair(c, seed)
    net = Surrogate(c["n0"], c["n1"], channels=CHANNELS, layers=len(DILATIONS), dilations=DILATIONS, max_batch=c["nb"])
    net.load_params(_params(seed))
    return dict(case=c, net=net, x=x, y=y, masses=torch.zeros((c["nb"], 2), dtype=F64, device="cuda"))


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    c = state["case"]
    if c["kind"] == "step":
        g = state["g"]
        g.psi.copy_(state["start"])
        g.step(c["steps"], state["dt"])
        return g.psi
    if c["kind"] == "observe":
        g = state["g"]
        return dict(mass=np.float64(g.mass()), energy=np.float64(g.energy()))
    if c["kind"] == "batch":
        b = state["b"]
        b.step(c["steps"])
        return b.psi if len(b.psi) <= 48 else torch.cat([p.reshape(-1) for p in b.psi])
    net = state["net"]
    if c["kind"] == "sur_fwd":
        out = net.forward(state["x"], masses=state["masses"])
        return dict(psi=out, masses=state["masses"])
    grad, loss = net.gradients(state["x"], state["y"])
    return dict(grad=grad, loss=loss)


def work(case):
    c = case
    if c["kind"] in ("step", "observe"):
        sites = math.prod(_shape(c))
        es = 8 if c["dtype"] == "c64" else 16
        v = 0 if c["field"] != "trap" else (8 if c["dtype"] == "c128" else 4)
        if c["kind"] == "observe":
            return dict(bytes=sites * (2 * es + v), flops=sites * 70)
        # per site and stage: the stencil's sums (4d or 8d adds per component), N, F and the stage update
        per = 2 * (4 if c["order"] == 2 else 8) * c["dims"] + 18
        return dict(bytes=sites * (2 * es + v), flops=4.0 * per * sites * c["steps"])
    if c["kind"] == "batch":
        mean = (c["nmin"] ** 2 + c["nmin"] * c["nmax"] + c["nmax"] ** 2) / 3.0
        return dict(bytes=c["runs"] * mean * 18, flops=4.0 * 42 * c["runs"] * mean * c["steps"])
    sites = c["nb"] * c["n0"] * c["n1"]
    mac = 9.0 * (4 * CHANNELS + (len(DILATIONS) - 2) * CHANNELS * CHANNELS + 2 * CHANNELS)
    if c["kind"] == "sur_fwd":
        return dict(bytes=16.0 * sites, flops=2 * mac * sites)
    return dict(bytes=16.0 * sites, flops=2 * (3 * mac - 9.0 * 4 * CHANNELS) * sites)


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------
def _shift(x, k, s):
    """x at +s along axis k (wrapped; callers drop or replace the sites where a wall is)."""
    return torch.roll(x, -s, k)


def _inner(x, d):
    return x[tuple(slice(1, -1) for _ in range(d))]


def _clamp(x, d):
    """An interior array spread to the whole grid: every boundary site takes its nearest interior site's value."""
    for k in range(d):
        n = x.shape[k]
        idx = torch.cat([torch.zeros(1, dtype=torch.long), torch.arange(n), torch.full((1,), n - 1)]).to(x.device)
        x = x.index_select(k, idx)
    return x


def _rhs(psi, p):
    """F(Psi) at every site, and a Lap Psi (interior sites, or all of a periodic grid)."""
    d, h, a, s, V, bc, order = p["d"], p["h"], p["a"], p["s"], p["V"], p["bc"], p["order"]
    N = s * (psi.real ** 2 + psi.imag ** 2)
    if V is not None:
        N = N - V
    D = -2.0 * d * psi
    for k in range(d):
        D = D + _shift(psi, k, 1) + _shift(psi, k, -1)
    D = D / (h * h)
    if bc == "periodic":
        inner = lambda x: x  # noqa: E731
        Dc = D
    else:
        inner = lambda x: _inner(x, d)  # noqa: E731
        Dc = inner(D)
        pc, Nc = inner(psi), inner(N)
        if order == 4:   # the boundary form of the Laplacian at boundary sites
            if bc == "dirichlet":
                Db = -N * psi / a
            elif bc == "l0":
                Db = torch.zeros_like(psi)
            else:
                m2 = pc.real ** 2 + pc.imag ** 2
                q = torch.where(m2 > 1e-300, (Dc * pc.conj()).real / m2, torch.zeros_like(m2)) + Nc / a
                Db = (_clamp(q, d) - N / a) * psi
            Db[tuple(slice(1, -1) for _ in range(d))] = Dc
            D = Db
    if order == 2:
        L = Dc
    else:   # D - (1/12) [sum_k delta_k^2 D - 2 sum_{j<k} delta_j^2 delta_k^2 Psi / h^2]
        acc = -2.0 * d * D
        for k in range(d):
            acc = acc + _shift(D, k, 1) + _shift(D, k, -1)
        for j in range(d):
            ej = _shift(psi, j, 1) + _shift(psi, j, -1) - 2.0 * psi
            for k in range(j + 1, d):
                acc = acc - (2.0 / (h * h)) * (_shift(ej, k, 1) + _shift(ej, k, -1) - 2.0 * ej)
        L = inner(D) - inner(acc) / 12.0
    F = 1j * (a * L + inner(N) * inner(psi))
    if bc == "periodic":
        return F, a * L
    if bc == "dirichlet":
        out = torch.zeros_like(psi)
    elif bc == "l0":
        out = 1j * N * psi
    else:
        m2 = pc.real ** 2 + pc.imag ** 2
        th = torch.where(m2 > 1e-300, (F * pc.conj()).imag / m2, torch.zeros_like(m2))
        out = 1j * _clamp(th, d) * psi
    out[tuple(slice(1, -1) for _ in range(d))] = F
    return out, a * L


def _rk4(psi, p, dt, steps):
    for _ in range(steps):
        k = _rhs(psi, p)[0]
        acc = k
        k = _rhs(psi + 0.5 * dt * k, p)[0]
        acc = acc + 2.0 * k
        k = _rhs(psi + 0.5 * dt * k, p)[0]
        acc = acc + 2.0 * k
        k = _rhs(psi + dt * k, p)[0]
        psi = psi + (dt / 6.0) * (acc + k)
    return psi


def _conv(h, w, b, dil):
    """3x3 convolution of channels-last states [nb, H, W, ci] with w [co, 9, ci], zero padding."""
    H, W = h.shape[1], h.shape[2]
    hp = torch.nn.functional.pad(h, (0, 0, dil, dil, dil, dil))
    out = b
    for t in range(9):
        y, x = (t // 3) * dil, (t % 3) * dil
        out = out + hp[:, y:y + H, x:x + W, :] @ w[:, t, :].T
    return out


def _network(params, x):
    at, h = 0, None
    m2 = x.real ** 2 + x.imag ** 2
    h = torch.stack([x.real, x.imag, m2 * x.real, m2 * x.imag], -1)
    for l, dil in enumerate(DILATIONS):
        ci = 4 if l == 0 else CHANNELS
        co = 2 if l == len(DILATIONS) - 1 else CHANNELS
        w = params[at:at + co * 9 * ci].reshape(co, 9, ci)
        b = params[at + co * 9 * ci:at + co * 9 * ci + co]
        at += co * 9 * ci + co
        h = _conv(h, w, b, dil)
        if l < len(DILATIONS) - 1:
            h = torch.nn.functional.silu(h)
    return x + torch.complex(h[..., 0], h[..., 1])


def exact(case, seed):
    c = case
    if c["kind"] in ("step", "observe"):
        psi, V, h, a, s, srho = _problem(c, seed)
        dt = _dt(c, V, h, a, srho)
        if c["dtype"] == "c64":
            psi = psi.to(torch.complex64).to(torch.complex128)
        if V is not None and c["dtype"] != "c128":
            V = V.to(torch.float32).to(F64)
        p = dict(d=c["dims"], h=h, a=a, s=s, V=V, bc=c["bc"], order=c["order"])
        if c["kind"] == "step":
            return _rk4(psi, p, dt, c["steps"])
        aL = _rhs(psi, p)[1]
        inner = (lambda x: x) if c["bc"] == "periodic" else (lambda x: _inner(x, c["dims"]))
        q = inner(psi)
        m2 = q.real ** 2 + q.imag ** 2
        e = -(q.conj() * aL).real - 0.5 * s * m2 * m2
        if V is not None:
            e = e + inner(V) * m2
        vol = h ** c["dims"]
        return dict(mass=np.float64(vol * float((psi.real ** 2 + psi.imag ** 2).sum())),
                    energy=np.float64(vol * float(e.sum())))
    if c["kind"] == "batch":
        out = []
        for r in _batch_runs(c, seed):
            p = dict(d=2, h=r["h"], a=r["a"], s=r["s"], V=None if r["V"] is None else r["V"].to(F64), bc=r["bc"],
                     order=r["order"])
            out.append(_rk4(r["psi0"].to(torch.complex128), p, r["dt"], c["steps"]))
        return out if len(out) <= 48 else torch.cat([p.reshape(-1) for p in out])
    x, y = _pair(c, seed)
    x, y = x.to(torch.complex128), y.to(torch.complex128)
    params = _params(seed).to(F64)
    if c["kind"] == "sur_fwd":
        out = torch.cat([_network(params, q[None]) for q in x])
        m = lambda z: (z.real ** 2 + z.imag ** 2).sum((1, 2))  # noqa: E731
        return dict(psi=out, masses=torch.stack([m(x), m(out)], 1))
    params.requires_grad_(True)
    loss = 0.0
    for q, t in zip(x, y):   # one state at a time: the 64-bit activations of a whole batch need not be held
        r = _network(params, q[None]) - t[None]
        part = (r.real ** 2 + r.imag ** 2).sum() / (2.0 * x.numel())
        part.backward()
        loss += float(part)
    return dict(grad=params.grad, loss=loss)
