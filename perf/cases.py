"""Performance cases of libwave: what a user of this framework has it compute.

The work is a gradient call (Algorithm 1, or one of the exact modes), a
forward run that makes traces, or one step of a time loop of the caller's own,
in 2D and 3D, in the velocity and the density form, from grids that a launch
latency dominates to grids of a billion cells.  Record lengths are those of
the experiments cut down so that a pass stays below two seconds; the work of a
call is proportional to the record length.

Inputs come from the seed alone (torch on the GPU); `exact` restates the same
calls in plain 64-bit torch.
"""
from __future__ import annotations

import math

import torch

from paper_2509_15744_gb300 import wave as W
from paper_2509_15744_gb300.autograd import WaveProblem, wave_misfit

DEV = "cuda"
H_VEL = 10.0                       # grid spacing of the velocity-form cases [m]
V_MIN, V_MAX = 1500.0, 4500.0      # model range [m/s]
H_DEN, C_MAX_DEN = 2e-3, 509.8366  # spacing [m] and largest wave speed [m/s] of the density form


def _case(name, entry, shape, order, nt, **kw):
    """A case as a flat dict; the shape is slowest axis first (nz = 0 in 2D)."""
    nz, ny, nx = shape if len(shape) == 3 else (0,) + tuple(shape)
    c = dict(entry=entry, nz=nz, ny=ny, nx=nx, order=order, nt=nt, physics="velocity", bc="dirichlet", storage="f32",
             kahan=False, nshots=1, mode="superposition", batched=False, objective="l2", receivers="line", rec_step=2)
    if name is not None:
        c["name"] = name
    c.update(kw)
    return c


def listed():
    return [
        # one evaluation of misfit and gradient of the small 2D inversion (128 x 128, order 2, 400 steps, 64 receivers on
        # the surface), through the differentiable function an optimiser calls: launches and latency count
        _case("misfit_2d_128_o2", "misfit", (128, 128), 2, 400),
        # the paper's inversion problem (251 x 251, Neumann, four sources at the edge midpoints, a receiver on every fifth
        # edge cell), a quarter of its 3200 steps
        _case("gradient_2d_251_o2_4shots", "gradient", (251, 251), 2, 800, bc="neumann", nshots=4, receivers="edges",
              rec_step=5),
        # the paper's topology optimisation problem (363 x 363, density form, patch energy), a third of its 1800 steps,
        # with the exact symmetric mode that its design loop uses
        _case("misfit_2d_363_density_patch", "misfit", (363, 363), 2, 600, physics="density", bc="neumann",
              mode="symmetric", objective="patch", receivers="patch"),
        # a 2D inversion of ordinary size, order 8, a tenth of its 4000 steps: the working set stays in the L2
        _case("gradient_2d_2048_o8", "gradient", (2048, 2048), 8, 400, rec_step=4),
        # the large density-form design problem with its dense patch of 262,144 objective cells
        _case("gradient_2d_4096_density_patch", "gradient", (4096, 4096), 2, 60, physics="density", bc="neumann",
              objective="patch", receivers="patch"),
        # synthetic data on a large ragged 2D grid (the forward-time study), from given initial levels
        _case("forward_2d_6001x8003_o4", "forward", (6001, 8003), 4, 40, rec_step=8),
        # a small 3D problem with the exact reverse-time mode: launches and latency count
        _case("gradient_3d_64x96x130_o4_reverse", "gradient", (64, 96, 130), 4, 100, mode="reverse", bc="neumann"),
        # the density form in 3D, ragged
        _case("gradient_3d_180x210x250_density", "gradient", (180, 210, 250), 2, 30, physics="density",
              mode="symmetric", rec_step=4),
        # synthetic data in 3D with 16-bit storage of the levels, ragged
        _case("forward_3d_300x311x333_o8_bf16", "forward", (300, 311, 333), 8, 40, storage="bf16", rec_step=4),
        # one step of three fields in a time loop of the caller's own, ragged, compensated accumulation
        _case("step_3d_257x300x401_o6_3fields", "step", (257, 300, 401), 6, 1, nshots=3, kahan=True),
        # the main workload: 3D survey, order 8, all shots advanced together, uneven record lengths, 256 x 256 receivers
        _case("gradient_3d_512_o8_8shots", "gradient", (512, 512, 512), 8, 12, nshots=8, batched=True),
        # a billion parameters: 4 shots together, compensated accumulation
        _case("gradient_3d_1024_o8_4shots_kahan", "gradient", (1024, 1024, 1024), 8, 8, nshots=4, batched=True,
              kahan=True, rec_step=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["vel2d", "vel2d", "den2d", "fwd2d", "vel3d", "den3d", "fwd3d", "step", "batched3d"])
    bc = rng.choice(["dirichlet", "neumann"])
    if kind in ("vel2d", "den2d", "fwd2d"):
        n = _log(rng, 64, 4096 if kind != "fwd2d" else 8000)
        shape = (n + rng.randint(-n // 8, n // 8), n + rng.randint(-n // 8, n // 8))
        cells = shape[0] * shape[1]
        nt = max(20, min(600, int(rng.uniform(0.5, 1.5) * 6e8 / cells)))
        if kind == "vel2d":
            return _case(None, rng.choice(["gradient", "misfit"]), shape, rng.choice([2, 2, 4, 6, 8]), nt, bc=bc,
                         nshots=rng.randint(1, 3), kahan=rng.random() < 0.25,
                         mode=rng.choice(["superposition", "superposition", "symmetric", "reverse"]),
                         receivers=rng.choice(["line", "edges"]), rec_step=rng.randint(2, 9))
        if kind == "den2d":
            return _case(None, rng.choice(["gradient", "misfit"]), shape, 2, nt, bc=bc, physics="density",
                         kahan=rng.random() < 0.25, mode=rng.choice(["superposition", "symmetric"]), objective="patch",
                         receivers="patch")
        return _case(None, "forward", shape, rng.choice([2, 4, 8]), nt, bc=bc, rec_step=rng.randint(2, 9))
    n = _log(rng, 40, 512 if kind == "batched3d" else 420)
    shape = tuple(n + rng.randint(-n // 5, n // 5) for _ in range(3))
    cells = shape[0] * shape[1] * shape[2]
    nt = max(8, min(100, int(rng.uniform(0.5, 1.5) * 8e8 / cells)))
    order = rng.choice([2, 4, 6, 8, 8])
    if kind == "vel3d":
        return _case(None, "gradient", shape, order, nt, bc=bc, kahan=rng.random() < 0.25,
                     mode=rng.choice(["superposition", "symmetric", "reverse"]), rec_step=rng.randint(2, 6))
    if kind == "den3d":
        return _case(None, "gradient", shape, 2, nt, bc=bc, physics="density", mode="symmetric",
                     rec_step=rng.randint(2, 6))
    if kind == "fwd3d":
        return _case(None, "forward", shape, order, nt, bc=bc, storage=rng.choice(["f32", "bf16", "f16"]),
                     rec_step=rng.randint(2, 6))
    if kind == "step":
        return _case(None, "step", shape, order, 1, bc=bc, nshots=rng.randint(1, 6), kahan=rng.random() < 0.5)
    return _case(None, "gradient", shape, order, max(8, nt // 3), bc=bc, nshots=rng.randint(2, 9), batched=True,
                 kahan=rng.random() < 0.3, rec_step=rng.randint(2, 6))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_C = {2: (-2.0, 1.0), 4: (-5 / 2, 4 / 3, -1 / 12), 6: (-49 / 18, 3 / 2, -3 / 20, 1 / 90),
      8: (-205 / 72, 8 / 5, -1 / 5, 8 / 315, -1 / 560)}   # central second-derivative weights


def _shape(c):
    return (c["nz"], c["ny"], c["nx"]) if c["nz"] else (c["ny"], c["nx"])


def _spacing(c):
    """(h, dt): half the leapfrog limit of the largest wave speed."""
    w = _C[c["order"]]
    s = abs(w[0] + 2 * sum((-1) ** j * w[j] for j in range(1, len(w))))
    h, vmax = (H_VEL, V_MAX) if c["physics"] == "velocity" else (H_DEN, C_MAX_DEN)
    return h, 0.5 * 2 * h / (vmax * math.sqrt(len(_shape(c)) * s))


def _smooth(shape, gen, modes=6):
    """Smooth random field in [0, 1]: random plane cosines, separable per mode."""
    nz, ny, nx = shape if len(shape) == 3 else (1,) + tuple(shape)
    r = torch.rand(modes, 7, generator=gen, dtype=torch.float64).to(DEV)
    axes = []
    for a, n in enumerate((nz, ny, nx)):
        t = torch.arange(n, dtype=torch.float64, device=DEV) / max(nx, 2)
        axes.append(torch.cos(2 * math.pi * (r[:, 2 * a:2 * a + 1] * 4 * t + r[:, 2 * a + 1:2 * a + 2])))
    amp = (0.2 + r[:, 6:7]) / (1.2 * modes)
    yx = (axes[1][:, :, None] * axes[2][:, None, :]).reshape(modes, -1).float()
    f = ((amp * axes[0]).float().t() @ yx).reshape(nz, ny, nx)
    return (0.5 + 0.5 * f).clamp_(0.0, 1.0).reshape(shape)


def _cells(c):
    """(flat source cells, flat receiver cells) of the survey."""
    shape = _shape(c)
    if len(shape) == 3:
        nz, ny, nx = shape
        side = max(1, math.ceil(math.sqrt(c["nshots"])))
        at = [(2 * ny * nx) + (ny * (2 * i + 1) // (2 * side)) * nx + nx * (2 * j + 1) // (2 * side)
              for i in range(side) for j in range(side)]
        y, x = torch.arange(0, ny, c["rec_step"]), torch.arange(0, nx, c["rec_step"])
        return at[:c["nshots"]], (ny * nx + y[:, None] * nx + x[None, :]).reshape(-1)
    ny, nx = shape
    src = [nx + nx // 2, (ny - 2) * nx + nx // 2, (ny // 2) * nx + 1, (ny // 2) * nx + nx - 2][:c["nshots"]]
    if c["receivers"] == "patch":   # source on the mid row, near enough to reach the patch in half the (shortened) record
        y = torch.arange(3 * ny // 8, 5 * ny // 8)
        x = torch.arange(nx // 8, nx // 8 + max(1, nx // 16))
        reach = max(1, int(0.1 * c["nt"]))
        return [(ny // 2) * nx + max(1, nx // 8 - reach)], (y[:, None] * nx + x[None, :]).reshape(-1)
    line = torch.arange(0, nx, c["rec_step"])
    if c["receivers"] == "line":
        return src, line
    rows = torch.arange(0, ny, c["rec_step"]) * nx
    return src, torch.unique(torch.cat([line, (ny - 1) * nx + line, rows, rows + nx - 1]))


def _inputs(c, seed):
    gen = torch.Generator().manual_seed(1000003 * int(seed) + 17)
    shape = _shape(c)
    h, dt = _spacing(c)
    if c["physics"] == "velocity":
        param = V_MIN + (V_MAX - V_MIN) * _smooth(shape, gen)
    else:   # a design in progress: grey material with small holes
        noise = torch.rand(shape, device=DEV, generator=torch.Generator(DEV).manual_seed(int(seed) + 5))
        param = (0.1 + 0.9 * _smooth(shape, gen) * noise).float()
    src, rec = _cells(c)
    rec = rec.to(DEV)
    shots = []
    for i, s in enumerate(src):
        n = c["nt"] if not c["batched"] else max(4, c["nt"] - (i % 4))   # uneven record lengths
        t = torch.arange(n + 1, dtype=torch.float64, device=DEV) * dt
        f = max(1.0 / (25 * dt), 2.0 / (n * dt)) * (0.9 + 0.2 * float(torch.rand(1, generator=gen)))
        if c["physics"] == "velocity":
            a = (math.pi * f * (t - 1.0 / f)) ** 2
            wav = (1 - 2 * a) * torch.exp(-a)
        else:
            w = 2 * math.pi * f
            wav = torch.where(t <= 2 / f, torch.sin(w * t) * torch.sin(w * t / 4) ** 2, torch.zeros_like(t))
        obs = None
        if c["objective"] == "l2" and c["entry"] != "step":   # arrivals with the moveout of their distance
            idx, at = [], []
            for size in reversed(shape):
                idx.append((rec // math.prod(shape[len(shape) - len(idx):])) % size)
                at.append((s // math.prod(shape[len(shape) - len(at):])) % size)
            dist = torch.sqrt(sum((p.double() - q) ** 2 for p, q in zip(idx, at)))
            speed = (2500.0 if c["physics"] == "velocity" else 343.0) * dt / h   # cells per step
            tau = (t / dt)[None, :] - (dist / speed)[:, None] - 1.0 / (f * dt)
            b = (math.pi * f * dt * tau) ** 2
            amp = (0.05 * h * h) / (1 + dist) ** (0.5 * (len(shape) - 1))
            obs = (amp[:, None] * (1 - 2 * b) * torch.exp(-b)).float().contiguous()
        shots.append((int(s), wav.float(), obs))
    levels = None
    if c["entry"] == "forward":
        a = _smooth(shape, gen) - 0.5
        levels = torch.stack([a, a + 0.02 * (_smooth(shape, gen) - 0.5)])
    elif c["entry"] == "step":
        levels = [_smooth(shape, gen) - 0.5 for _ in range(2 * c["nshots"])]
    return dict(param=param.contiguous(), h=h, dt=dt, rec=rec, shots=shots, levels=levels)


def _sign(f):
    return (1.0, -1.0, 0.5)[f % 3]


# ---------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = dict(case)
    d = _inputs(c, seed)
    shots = [W.Shot(s, wav, d["rec"], obs) for s, wav, obs in d["shots"]]
    if c["entry"] == "misfit":
        problem = WaveProblem(h=d["h"], dt=d["dt"], shots=shots, order=c["order"], physics=c["physics"], bc=c["bc"],
                              storage=c["storage"], kahan=c["kahan"], objective=c["objective"], batched=c["batched"],
                              mode=c["mode"])
        return dict(case=c, param=d["param"].requires_grad_(True), problem=problem)
    model = W.Model(d["param"], d["h"], d["dt"], c["order"], c["physics"], c["bc"], storage=c["storage"],
                    kahan=c["kahan"])
    st = dict(case=c, model=model, shots=shots, init=d["levels"])
    if c["entry"] == "step":
        def pitched(a):
            out = torch.zeros(model.pitched_shape(), dtype=torch.float32, device=DEV)
            out[..., :a.shape[-1]] = a
            return out
        n = c["nshots"]
        st.update(cur=[pitched(a) for a in d["levels"][:n]], prev=[pitched(a) for a in d["levels"][n:]],
                  acc=torch.zeros(model.pitched_shape(), device=DEV), sign=[_sign(f) for f in range(n)], init=None,
                  comp=torch.zeros(model.pitched_shape(), device=DEV) if c["kahan"] else None)
    return st


def run(state):
    c = state["case"]
    if c["entry"] == "misfit":
        cost = wave_misfit(state["param"], state["problem"])
        (grad,) = torch.autograd.grad(cost, state["param"])
        return {"misfit": cost.detach(), "grad": grad}
    m = state["model"]
    if c["entry"] == "gradient":
        grad, misfit, k = m.gradient(state["shots"], objective=c["objective"], mode=c["mode"], batched=c["batched"],
                                     grad_wrt="param")
        return {"misfit": misfit, "grad": grad, "k": k, "norm": m.grad_norm}
    if c["entry"] == "forward":
        traces, final = m.forward(state["shots"], init=state["init"], return_final=True)
        return {"traces": traces, "final": final}
    m.step(state["cur"], state["prev"], acc=state["acc"], comp=state["comp"], acc_sign=state["sign"])
    return {"next": state["prev"], "acc": state["acc"]}


def work(case):
    shape = _shape(case)
    cells, r, nd = math.prod(shape), case["order"] // 2, len(shape)
    if case["physics"] == "velocity":
        step, inc = 3 * r * nd + 4, 4            # stencil and update; sensitivity increment
    else:
        step, inc = 8 * nd + 4, 6 * nd + 5
    steps = sum(case["nt"] if not case["batched"] else max(4, case["nt"] - (i % 4)) for i in range(case["nshots"]))
    _, rec = _cells(case)
    traces = 4 * len(rec) * (steps + case["nshots"])
    if case["entry"] == "step":   # per field: both levels in, one out; coefficients once; accumulator in and out
        acc = 16 if case["kahan"] else 8
        return {"bytes": cells * (12 * case["nshots"] + 4 + acc), "flops": cells * (step + inc) * case["nshots"]}
    if case["entry"] == "forward":   # model and initial levels in, traces and final levels out
        return {"bytes": cells * (4 + 16) + traces, "flops": cells * step * steps}
    fields = 2 if case["mode"] == "superposition" else 3     # time loops of a gradient call
    incs = 2 if case["mode"] != "reverse" else 1
    obs = traces if case["objective"] == "l2" else 0
    return {"bytes": cells * 8 + obs, "flops": cells * steps * (fields * step + incs * inc)}


# ---------------------------------------------------------------------------
# the same calls in plain 64-bit torch
# ---------------------------------------------------------------------------
def _ghosts(u, ax, r, bc):
    """u with r ghost layers at both ends of an axis: the boundary rule."""
    n = u.shape[ax]
    if bc == "neumann":
        return torch.cat([u.narrow(ax, 0, r).flip(ax), u, u.narrow(ax, n - r, r).flip(ax)], ax)
    zero = torch.zeros_like(u.narrow(ax, 0, 1))
    lo, hi = [zero], [zero]
    if r > 1:
        lo, hi = [-u.narrow(ax, 0, r - 1).flip(ax), zero], [zero, -u.narrow(ax, n - r + 1, r - 1).flip(ax)]
    return torch.cat(lo + [u] + hi, ax)


class _Exact:
    def __init__(self, c, d):
        self.c, self.bc, self.r = c, c["bc"], c["order"] // 2
        self.h, self.dt, self.shape = d["h"], d["dt"], _shape(c)
        p = self.p = d["param"].detach().double()
        if c["physics"] == "velocity":
            self.coef, self.da = (p * self.dt / self.h) ** 2, 1.0
            return
        da, db = 1 / 6.87e8 - 1 / 1.419e5, 1 / 2643.0 - 1 / 1.204
        self.coef = self.dt ** 2 / self.h ** 2 / (1 / 1.419e5 + p * da)
        self.b, self.da, self.dbs = 1 / 1.204 + p * db, da, self.dt ** 2 / self.h ** 2 * db

    def _faces(self, u, weight):
        """Sum over the 2 nd faces of weight(b_i, b_j, ghost)(u_j - u_i)."""
        out = torch.zeros_like(u)
        for ax in range(u.dim()):
            n = u.shape[ax]
            ug, bg = _ghosts(u, ax, 1, self.bc), _ghosts(self.b, ax, 1, "neumann")
            for o, edge in ((0, 0), (2, n - 1)):
                out += weight(self.b, bg.narrow(ax, o, n), ug.narrow(ax, o, n) - u, ax, edge)
        return out

    def lap(self, u):
        if self.c["physics"] == "density":
            return self._faces(u, lambda bi, bj, du, ax, e: 2 * bi * bj / (bi + bj) * du)
        w = _C[self.c["order"]]
        out = u.dim() * w[0] * u
        for ax in range(u.dim()):
            g, n = _ghosts(u, ax, self.r, self.bc), u.shape[ax]
            for j in range(1, self.r + 1):
                out += w[j] * (g.narrow(ax, self.r - j, n) + g.narrow(ax, self.r + j, n))
        return out

    def stiff(self, u):
        def weight(bi, bj, du, ax, edge):
            w = 2 * bj ** 2 / (bi + bj) ** 2
            if self.bc == "dirichlet":
                w = w.clone()
                w.select(ax, edge).fill_(1.0)
            return w * du ** 2
        return self._faces(u, weight)

    def step(self, prev, cur, force):
        """force: list of (flat cells, values); returns u^{n+1}."""
        old = prev.clone().reshape(-1)
        for cells, val in force:
            old.index_add_(0, cells, -(self.coef.reshape(-1)[cells] * self.h ** 2) * val)
        return 2 * cur - old.reshape(self.shape) + self.coef * self.lap(cur)

    def inc(self, new, cur, mass, stiff):
        out = self.da * (new - cur) ** 2 if mass else torch.zeros_like(cur)
        if stiff and self.c["physics"] == "density":
            out = out - self.dbs * self.stiff(cur)
        return out


def _exact_gradient(c, d):
    e = _Exact(c, d)
    rec, mode = d["rec"], c["mode"]
    acc, cost, k = torch.zeros_like(e.p), torch.zeros(1, dtype=torch.float64, device=DEV), None
    two = mode in ("symmetric", "reverse")
    for s, wav, obs in d["shots"]:
        n_s, psi = wav.numel() - 1, wav.double()
        at = torch.tensor([s], device=DEV)
        wgt = 1.0 if c["objective"] == "l2" else 2.0 / rec.numel()
        prev, cur = torch.zeros_like(e.p), torch.zeros_like(e.p)
        resid = torch.zeros(n_s + 1, rec.numel(), dtype=torch.float64, device=DEV)
        data = obs.double().t() if obs is not None else torch.zeros_like(resid)
        resid[0], resid[1] = -data[0], -data[1]
        for n in range(1, n_s + 1):
            new = e.step(prev, cur, [(at, psi[n:n + 1])])
            if not two and n <= n_s - 1:
                acc += e.inc(new, cur, True, True)
            prev, cur = cur, new
            if n < n_s:
                resid[n + 1] = cur.reshape(-1)[rec] - data[n + 1]
        cost += 0.5 * wgt * e.dt * resid.square().sum()
        if k is None and mode != "reverse":
            ratio = 1.0 if mode == "symmetric" else (5e-2 if c["physics"] == "density" else 1e-2)
            f2, p2 = wgt * wgt * float(resid[1:].square().sum()), float(psi[1:].square().sum())
            k = ratio * math.sqrt(p2 / f2) if f2 > 0 and p2 > 0 else 1.0
        if mode == "reverse":
            lc, ln, uc, un = torch.zeros_like(cur), torch.zeros_like(cur), prev, cur
            for j in range(n_s, 0, -1):
                u2 = e.step(un, uc, [(at, psi[j:j + 1])])
                l2 = e.step(ln, lc, [(rec, -wgt * resid[j])])
                acc -= (lc - l2) * (uc - u2)
                un, uc, ln, lc = uc, u2, lc, l2
            continue
        for sg in ((1.0, -1.0) if mode == "symmetric" else (1.0,)):
            sc, sn = prev, cur
            for j in range(n_s, 0, -1):
                new = e.step(sn, sc, [(at, psi[j:j + 1]), (rec, -sg * k * wgt * resid[j])])
                acc -= sg * e.inc(new, sc, True, j <= n_s - 1)
                sn, sc = sc, new
    grad = acc / e.dt / (1.0 if mode == "reverse" else (4 * k if mode == "symmetric" else 2 * k))
    if c["physics"] == "velocity":
        grad = grad * (-2 / e.p ** 3)
    out = {"misfit": cost if c["entry"] == "gradient" else cost.reshape(()), "grad": grad}
    if c["entry"] == "gradient":
        out["k"] = torch.tensor([k or 0.0], dtype=torch.float64, device=DEV)
        out["norm"] = grad.norm().reshape(1)
    return out


def exact(case, seed):
    c = dict(case)
    steps = c["nt"] * c["nshots"] * (1 if c["entry"] in ("forward", "step") else 3)
    if math.prod(_shape(c)) * steps * (1 + c["order"]) > 1e12:   # over about 20 seconds
        return None
    d = _inputs(c, seed)
    if c["entry"] in ("misfit", "gradient"):
        return _exact_gradient(c, d)
    e = _Exact(c, d)
    if c["entry"] == "step":
        n, acc, out = c["nshots"], torch.zeros_like(e.p), []
        for f in range(n):
            cur = d["levels"][f].double()
            new = e.step(d["levels"][n + f].double(), cur, [])
            acc += _sign(f) * e.inc(new, cur, True, True)
            out.append(new)

        def pitched(a):
            return torch.nn.functional.pad(a, (0, (-a.shape[-1]) % 128))
        return {"next": [pitched(a) for a in out], "acc": pitched(acc)}
    traces, final = [], None
    for s, wav, _ in d["shots"]:
        at, psi = torch.tensor([s], device=DEV), wav.double()
        prev, cur = d["levels"][0].double(), d["levels"][1].double()
        tr = [prev.reshape(-1)[d["rec"]], cur.reshape(-1)[d["rec"]]]
        for n in range(1, wav.numel()):
            prev, cur = cur, e.step(prev, cur, [(at, psi[n:n + 1])])
            tr.append(cur.reshape(-1)[d["rec"]])
        traces.append(torch.stack(tr[:wav.numel()], 1))
        final = torch.stack([prev, cur])
    return {"traces": traces, "final": final}
