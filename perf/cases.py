"""The work that programs built on this library have it do, as measurable cases.

Every case goes through the public Python entry points (api.AdiWave,
api.AdiWaveBatch, autograd.simulate).  The kinds:

- run:      one grid, restarted from new initial data and advanced by the time
            loop (reset, run, state), with or without a point source, initial
            velocity, second-order start and receivers;
- step:     the same, one call per time step (a program that looks at the field
            after every step);
- gradient: forward run with receivers and checkpoints, residual, adjoint (the
            inner step of a waveform inversion that keeps its handle);
- autograd: the same through torch.autograd, a handle created and freed by
            every call;
- batch:    many shots on grids of uneven size advanced together;
- model:    the wider problem class (time-dependent coefficient and a source
            field on every level).

cfl is tau max(c) / min(h).  The workloads run at 0.5, the constant-medium
standing wave at 1, the paper's own experiment (dx = 0.01, dt = 0.02, c = 1)
at 2; far above that the elimination switches to FP64 (5 here).
"""
import math

import numpy as np
import torch

F_PEAK = 20.0   # Ricker peak frequency
N_BUMPS = 8


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _run(nx, ny, steps, cfl=0.5, const=False, source=True, n_rec=0, start="paper", psi=False):
    return dict(kind="run", nx=nx, ny=ny, steps=steps, cfl=cfl, const=const, source=source,
                n_rec=n_rec, start=start, psi=psi)


def listed():
    out = []

    def add(name, case):
        out.append(dict(case, name=name))

    # a program that steps one level at a time on a small odd grid: launches only
    add("step_100x75", dict(kind="step", nx=100, ny=75, steps=1, cfl=0.5))
    # the paper's experiment: 99^2 interior nodes, c = 1, dt = 2 dx, 50 steps
    add("paper_99", _run(99, 99, 50, cfl=2.0, const=True, source=False))
    # the constant-medium standing wave of the benchmark
    add("standing_128", _run(128, 128, 200, cfl=1.0, const=True, source=False))
    # a shot of moderate, odd size recorded at a line of receivers
    add("shot_1000", _run(1000, 1000, 40, n_rec=64))
    # a ragged oblong section, initial velocity, second-order start
    add("section_3001x1501", _run(3001, 1501, 20, n_rec=16, start="taylor2", psi=True))
    # the benchmark's 4096^2 run (its 1000 steps, 20 of them)
    add("ricker_4096", _run(4096, 4096, 20))
    # the bandwidth case
    add("ricker_16384", _run(16384, 16384, 6))
    # waveform inversion: the benchmark's adjoint workload, 100 of its 2000 steps
    add("gradient_1024", dict(kind="gradient", nx=1024, ny=1024, steps=100, cfl=0.5, every=50, n_rec=64))
    # the same step written with torch.autograd on a small model
    add("autograd_301", dict(kind="autograd", nx=301, ny=301, steps=60, cfl=0.5, every=20, n_rec=32))
    # half of the benchmark's batch of shots of 256^2 .. 2048^2, 6 of its 500 steps
    add("batch_32", dict(kind="batch", count=32, lo=256, hi=2048, pow2=True, steps=6, cfl=0.5))
    # a time step so long that the elimination runs in FP64
    add("long_step_2048x1500", _run(2048, 1500, 4, cfl=5.0))
    # c(t) and a source field on every level
    add("model_700x900", dict(kind="model", nx=700, ny=900, steps=12, cfl=0.5))
    return out


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(["run", "run", "run", "run", "step", "gradient", "gradient", "autograd",
                       "batch", "batch", "model", "long"])
    if kind in ("run", "step"):
        nx = _logint(rng, 40, 14000)
        ny = min(14000, max(40, int(nx * math.exp(rng.uniform(-1.2, 1.2)))))
        if rng.random() < 0.3:
            nx -= nx % 32
            nx = max(nx, 64)
        if kind == "step":
            nx, ny = min(nx, 3000), min(ny, 3000)
            return dict(kind="step", nx=nx, ny=ny, steps=rng.randint(1, 3), cfl=0.5)
        steps = max(2, min(200, int(8.0e8 / (nx * ny))))
        steps = rng.randint(max(2, steps // 3), steps)
        const = rng.random() < 0.2
        return _run(nx, ny, steps, cfl=rng.choice([0.5, 0.5, 0.5, 0.5, 1.0, 2.0]), const=const,
                    source=not const, n_rec=rng.choice([0, 0, 8, 64]),
                    start=rng.choice(["paper", "paper", "taylor2"]), psi=rng.random() < 0.3)
    if kind in ("gradient", "autograd"):
        hi = 1300 if kind == "gradient" else 500
        nx = _logint(rng, 64, hi)
        ny = min(hi, max(64, int(nx * math.exp(rng.uniform(-0.6, 0.6)))))
        return dict(kind=kind, nx=nx, ny=ny, steps=rng.randint(20, 90), cfl=0.5,
                    every=rng.choice([10, 20, 50]), n_rec=rng.randint(1, 64))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 32), lo=rng.choice([64, 200, 256]),
                    hi=rng.choice([900, 1500, 2048]), pow2=False, steps=rng.randint(2, 8), cfl=0.5)
    if kind == "model":
        return dict(kind="model", nx=_logint(rng, 64, 1400), ny=_logint(rng, 64, 1400),
                    steps=rng.randint(4, 16), cfl=0.5)
    return _run(_logint(rng, 200, 2400), _logint(rng, 200, 2400), rng.randint(2, 5), cfl=5.0)


# ---------------------------------------------------------------------------
# inputs, made from the seed alone
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda:0" if torch.cuda.is_available() else "cpu")


def _nodes(n, dev):
    return (torch.arange(n, dtype=torch.float64, device=dev) + 1.0) / (n + 1)


def _bump_sum(nx, ny, par, dev, block):
    """block(sum of Gaussian bumps) as FP32 [ny, nx], a block of rows at a time."""
    x, y = _nodes(nx, dev), _nodes(ny, dev)
    out = torch.empty((ny, nx), dtype=torch.float32, device=dev)
    gx = torch.stack([torch.exp(-(x - cx) ** 2 / (2 * w * w)) for cx, _, w, _ in par])
    gy = torch.stack([a * torch.exp(-(y - cy) ** 2 / (2 * w * w)) for _, cy, w, a in par])
    rows = max(1, (1 << 25) // nx)
    for j in range(0, ny, rows):
        out[j:j + rows] = block(gy[:, j:j + rows].float().t() @ gx.float())
    return out


def _medium(nx, ny, rng, dev, const):
    """m = c^2, c = 1 or 1 + 2 sigmoid(eight seeded bumps) in (1, 3)."""
    par = [(rng.uniform(0, 1), rng.uniform(0, 1), rng.uniform(0.05, 0.2), rng.uniform(-3, 3))
           for _ in range(N_BUMPS)]
    if const:
        return torch.ones((ny, nx), dtype=torch.float32, device=dev)
    return _bump_sum(nx, ny, par, dev, lambda s: (1.0 + 2.0 * torch.sigmoid(s)) ** 2)


def _pulses(nx, ny, rng, dev, scale=1.0):
    """A smooth wavefield: a dozen seeded Gaussian pulses of both signs."""
    par = [(rng.uniform(0.1, 0.9), rng.uniform(0.1, 0.9), rng.uniform(0.02, 0.08),
            scale * rng.uniform(-1, 1)) for _ in range(12)]
    return _bump_sum(nx, ny, par, dev, lambda s: s)


def _ricker(n, tau, dev):
    t = np.arange(n, dtype=np.float64) * tau
    a = (math.pi * F_PEAK * (t - 1.0 / F_PEAK)) ** 2
    return torch.from_numpy(((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)).to(dev)


def _grid_inputs(case, seed, dev):
    nx, ny, steps = case["nx"], case["ny"], case["steps"]
    rng = np.random.default_rng([seed, nx, ny])
    const = bool(case.get("const"))
    q = dict(m=_medium(nx, ny, rng, dev, const), phi=_pulses(nx, ny, rng, dev))
    cmax = math.sqrt(float(q["m"].max()))
    q["tau"] = case["cfl"] * min(1.0 / (nx + 1), 1.0 / (ny + 1)) / cmax
    q["psi"] = _pulses(nx, ny, rng, dev, 5.0) if case.get("psi") else None
    q["src"] = q["wavelet"] = None
    if case.get("source", True):
        q["src"] = (int(rng.integers(nx // 4, 3 * nx // 4 + 1)), int(rng.integers(ny // 4, 3 * ny // 4 + 1)))
        q["wavelet"] = _ricker(steps + 2, q["tau"], dev)
    q["rec"] = None
    n_rec = case.get("n_rec", 0)
    if n_rec:
        if case["kind"] == "run":  # a line across the section at a tenth of its depth
            iy = min(ny - 1, int(0.1 * (ny + 1)))
            ix = [int((r + 0.5) / n_rec * nx) for r in range(n_rec)]
        else:  # near enough to the source for its waves to arrive within the run
            iy = max(0, q["src"][1] - max(3, int(steps * case["cfl"] / 5)))
            ix = [q["src"][0] + (r - n_rec // 2) * max(1, nx // (4 * n_rec)) for r in range(n_rec)]
        q["rec"] = np.array([[min(nx - 1, max(0, i)), iy] for i in ix], dtype=np.int32)
        g = torch.Generator(device="cpu").manual_seed(seed * 7919 + 13)
        q["data"] = (0.1 * torch.randn((steps, n_rec), generator=g)).to(dev)
    if case["kind"] == "model":
        k = np.arange(steps + 3)
        q["g"] = torch.from_numpy((1.0 + 0.3 * np.sin(0.37 * k + rng.uniform(0, 6))).astype(np.float32)).to(dev)
        q["f"] = torch.stack([_pulses(nx, ny, rng, dev, 50.0) for _ in range(steps + 1)])
    return q


def _batch_shapes(case, seed):
    rng = np.random.default_rng([30_000, case["count"], case["lo"], case["hi"]])
    if case["pow2"]:
        sizes = [2 ** k for k in range(int(math.log2(case["lo"])), int(math.log2(case["hi"])) + 1)]
        return [(int(s), int(s)) for s in rng.choice(sizes, size=case["count"])]
    e = rng.uniform(math.log(case["lo"]), math.log(case["hi"]), size=(case["count"], 2))
    return [(int(math.exp(a)), int(math.exp(b))) for a, b in e]


def _batch_inputs(case, seed, dev):
    return [_grid_inputs(dict(kind="run", nx=nx, ny=ny, steps=case["steps"], cfl=case["cfl"]),
                         seed * 1009 + b, dev) for b, (nx, ny) in enumerate(_batch_shapes(case, seed))]


# ---------------------------------------------------------------------------
# preparation and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2006_10142_gb300 import api
    dev = _device()
    kind = case["kind"]
    if kind == "batch":
        q = _batch_inputs(case, seed, dev)
        sim = api.AdiWaveBatch([p["m"] for p in q], [p["phi"] for p in q], [p["tau"] for p in q])
        return dict(case=case, q=q, sim=sim)
    q = _grid_inputs(case, seed, dev)
    if kind == "autograd":
        q["m"].requires_grad_(True)
        q["wavelet"].requires_grad_(True)
        return dict(case=case, q=q)
    sim = api.AdiWave(q["m"], q["phi"], q["tau"], psi=q["psi"], start=case.get("start", "paper"),
                      src=q["src"], wavelet=q["wavelet"])
    if kind == "gradient":
        sim.set_checkpointing(case["every"])
    if kind == "model":
        sim.set_model("factored", g=q["g"], f=q["f"])
    return dict(case=case, q=q, sim=sim)


def run(state):
    case, q = state["case"], state["q"]
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        sim = state["sim"]
        sim.reset([p["phi"] for p in q])
        sim.run(steps, srcs=[p["src"] for p in q], wavelets=[p["wavelet"] for p in q])
        return [t for b in range(len(q)) for t in sim.state(b)[:2]]
    if kind == "autograd":
        from paper_2006_10142_gb300 import autograd
        q["m"].grad = None
        q["wavelet"].grad = None
        tr = autograd.simulate(q["m"], q["wavelet"], src=q["src"], rec=q["rec"], steps=steps,
                               dt=q["tau"], phi=q["phi"], ckpt_every=case["every"])
        loss = 0.5 * ((tr - q["data"]) ** 2).sum()
        loss.backward()
        return dict(traces=tr.detach(), grad_m=q["m"].grad, grad_wavelet=q["wavelet"].grad)
    sim = state["sim"]
    sim.reset(q["phi"], psi=q["psi"], src=q["src"], wavelet=q["wavelet"])
    if kind == "step":
        for _ in range(steps):
            sim.step(src=q["src"], wavelet=q["wavelet"])
        up, uc, _ = sim.state()
        return dict(u_prev=up, u_cur=uc)
    tr = sim.run(steps, src=q["src"], wavelet=q["wavelet"], rec=q["rec"])
    if kind == "gradient":
        gm, gw = sim.adjoint(tr - q["data"])
        return dict(traces=tr, grad_m=gm, grad_wavelet=gw)
    up, uc, _ = sim.state()
    out = dict(u_prev=up, u_cur=uc)
    if tr is not None:
        out["traces"] = tr
    return out


def work(case):
    """Bytes and operations of one pass.  A step reads u^k, u^{k-1} and m and
    writes u^{k+1} (16 B per point; about 30 operations: right-hand side 9,
    two tridiagonal solves of 9, update 3); the start reads phi and writes two
    levels, the read-out copies two levels.  A reverse step reads two adjoint
    levels and m, the forward state's two increments, and updates the FP64
    gradient and one adjoint level (40 B, 40 operations), after recomputing
    the forward step with its increments kept (24 B)."""
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        pts = sum(nx * ny for nx, ny in _batch_shapes(case, 0))
    else:
        pts = case["nx"] * case["ny"]
    if kind in ("gradient", "autograd"):
        every = case["every"]
        nck = (steps + every - 1) // every
        per = 16 + 24 + 40
        return dict(bytes=pts * (steps * per + 32 * nck + 12 + 8), flops=pts * steps * 100)
    per = 16
    if kind == "model":
        per += 4  # the level's source field
    return dict(bytes=pts * (steps * per + 12 + 16), flops=pts * steps * 30)


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _shift(t, k, axis, fill):
    """t shifted by k along axis (k > 0: element i takes t[i - k]), `fill` outside."""
    n = t.shape[axis]
    out = torch.full_like(t, fill)
    if abs(k) < n:
        src = t.narrow(axis, 0, n - k) if k > 0 else t.narrow(axis, -k, n + k)
        (out.narrow(axis, k, n - k) if k > 0 else out.narrow(axis, 0, n + k)).copy_(src)
    return out


def _solve(s, d, axis):
    """Solution of -s x_{i-1} + (1 + 2 s) x_i - s x_{i+1} = d along axis, by
    parallel cyclic reduction until the couplings vanish."""
    a, b, c, d = -s, 1.0 + 2.0 * s, -s, d.clone()
    # no neighbour outside the line
    a = a.clone()
    c = c.clone()
    a.narrow(axis, 0, 1).zero_()
    c.narrow(axis, s.shape[axis] - 1, 1).zero_()
    h, n = 1, s.shape[axis]
    while h < n:
        blo = _shift(b, h, axis, 1.0)
        k1 = a / blo
        del blo
        bhi = _shift(b, -h, axis, 1.0)
        k2 = c / bhi
        del bhi
        b = b - _shift(c, h, axis, 0.0) * k1 - _shift(a, -h, axis, 0.0) * k2
        d = d - _shift(d, h, axis, 0.0) * k1 - _shift(d, -h, axis, 0.0) * k2
        a, c = -_shift(a, h, axis, 0.0) * k1, -_shift(c, -h, axis, 0.0) * k2
        h *= 2
        if float(torch.maximum(a.abs().max(), c.abs().max())) < 1e-40:
            break
    return d / b


def _lap(u, cx, cy):
    """cx (u_{i-1} - 2u + u_{i+1}) + cy (the same along y), zero ring."""
    r = (-2.0 * (cx + cy)) * u
    r[:, 1:] += cx * u[:, :-1]
    r[:, :-1] += cx * u[:, 1:]
    r[1:] += cy * u[:-1]
    r[:-1] += cy * u[1:]
    return r


class _Exact:
    def __init__(self, q, nx, ny):
        self.m = q["m"].detach().double()
        self.tau = q["tau"]
        self.hx, self.hy = 1.0 / (nx + 1), 1.0 / (ny + 1)
        self.cx, self.cy = (self.tau / self.hx) ** 2, (self.tau / self.hy) ** 2
        self.src = q["src"]
        self.wav = q["wavelet"].detach().double() if q["wavelet"] is not None else None

    def force(self, k):
        """tau^2 f^k at the source node."""
        if self.wav is None or k >= self.wav.numel():
            return 0.0
        return float(self.wav[k]) * self.tau ** 2 / (self.hx * self.hy)

    def start(self, q, kind):
        u0 = q["phi"].double()
        u1 = u0.clone()
        if q["psi"] is not None:
            u1 += self.tau * q["psi"].double()
        if kind == "taylor2":
            u1 += 0.5 * self.m * _lap(u0, self.cx, self.cy)
            if self.src is not None:
                u1[self.src[1], self.src[0]] += 0.5 * self.force(0)
        return u0, u1

    def step(self, up, uc, k, g=None, f=None):
        """(u^{k+1}, w, z)."""
        if g is None:
            r = self.m * _lap(uc, self.cx, self.cy)
            m = self.m
        else:
            at = lambda i: float(g[min(i, g.numel() - 1)])
            r = self.m * (at(k + 1) * _lap(uc, self.cx, self.cy)
                          + 0.5 * (at(k - 1) - at(k + 1)) * _lap(up, self.cx, self.cy))
            if k < f.shape[0]:
                r += self.tau ** 2 * f[k].double()
            m = at(k + 1) * self.m
        if self.src is not None:
            r[self.src[1], self.src[0]] += self.force(k)
        w = _solve(0.5 * self.cx * m, r, 1)
        del r
        z = _solve(0.5 * self.cy * m, w, 0)
        return 2.0 * uc - up + z, w, z


def _exact_gradient(case, q):
    nx, ny, steps = case["nx"], case["ny"], case["steps"]
    e = _Exact(q, nx, ny)
    rec = torch.from_numpy(q["rec"].astype(np.int64)).to(e.m.device)
    rx, ry = rec[:, 0], rec[:, 1]
    up, uc = e.start(q, "paper")
    tr, kept = [], []
    for s in range(steps):
        un, w, z = e.step(up, uc, s + 1)
        tr.append(un[ry, rx].clone())
        kept.append((w, z))
        up, uc = uc, un
    tr = torch.stack(tr)
    resid = tr - q["data"].double()
    gm = torch.zeros_like(e.m)
    gw = torch.zeros(q["wavelet"].numel(), dtype=torch.float64, device=e.m.device)
    sx, sy = 0.5 * e.cx * e.m, 0.5 * e.cy * e.m
    lam = [torch.zeros_like(e.m), torch.zeros_like(e.m)]  # dJ/du^{k+1}, dJ/du^k
    scale = e.tau ** 2 / (e.hx * e.hy)
    ix, iy = e.src
    for s in reversed(range(steps)):
        k = s + 1
        p, o = lam
        p.index_put_((ry, rx), resid[s], accumulate=True)
        w, z = kept[s]
        v = _solve(sy, e.m * p, 0)        # m . Y^{-T} lam
        r = _solve(sx, v, 1)              # m . X^{-T} Y^{-T} lam
        ws = w.clone()
        ws[iy, ix] -= e.force(k)
        gm += (v * (z - w) + r * ws) / e.m ** 2
        if k < gw.numel():
            gw[k] += scale * r[iy, ix] / e.m[iy, ix]
        lam = [o + 2.0 * p + _lap(r, e.cx, e.cy), -p]
    return tr, gm, gw


def exact(case, seed):
    dev = _device()
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        out = []
        for p in _batch_inputs(case, seed, dev):
            ny, nx = p["m"].shape
            e = _Exact(p, nx, ny)
            up, uc = e.start(p, "paper")
            for s in range(steps):
                up, uc = uc, e.step(up, uc, s + 1)[0]
            out += [up, uc]
        return out
    q = _grid_inputs(case, seed, dev)
    if kind in ("gradient", "autograd"):
        tr, gm, gw = _exact_gradient(case, q)
        return dict(traces=tr, grad_m=gm, grad_wavelet=gw)
    e = _Exact(q, case["nx"], case["ny"])
    up, uc = e.start(q, case.get("start", "paper"))
    tr = []
    for s in range(steps):
        un = e.step(up, uc, s + 1, q.get("g"), q.get("f"))[0]
        if q["rec"] is not None:
            rec = torch.from_numpy(q["rec"].astype(np.int64)).to(dev)
            tr.append(un[rec[:, 1], rec[:, 0]].clone())
        up, uc = uc, un
    out = dict(u_prev=up, u_cur=uc)
    if tr:
        out["traces"] = torch.stack(tr)
    return out
