"""The calls that stand for this framework's use, with their inputs and their work.

Every case goes through the public binding (``paper_1702_07760_gb300.sph``) the way a
program on top of it does: ensembles and restarts load a recorded state into a handle, run a
stretch of steps and take the state out again; the logger asks for diagnostics; the surrogate
records rates, jumps and trains.  The stretches start from a drop or a flume in motion (a smooth
cellular or orbital flow over the hydrostatic state, with a little noise), fast enough that the
neighbour lists are rebuilt about as often as in the long runs: every 5 to 20 steps.

``exact`` is the same arithmetic in 64 bits in plain torch (a pair list by cells, the paper's
Sec. II equations term by term, the explicit midpoint step; the message-passing network layer by
layer), without the framework's kernels.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1702_07760_gb300 import sph
from paper_1702_07760_gb300 import surrogate_layout as SL
from paper_1702_07760_gb300 import workloads as WL

K_JUMP = 8       # plain steps one surrogate jump spans


# --------------------------------------------------------------------------
# The cases


def listed():
    return [
        # the 2-D drop of the first example (9 380 particles): the smallest runs, where launches and
        # latency are the time
        dict(name="drop2d", kind="run", dim=2, sx=64, sy=1, sz=128, d=16.0, steps=40),
        # the paper's own drop example (0.2 m tank, open top, 96 148 particles) as its long runs are
        # made: kinematic viscosity, boundary particles keeping their continuity density
        dict(name="paper_cube", kind="paper", shape="cube", visc=1, renorm_walls=0, steps=20),
        # the benchmark's 3-D drop (656 600 particles): an ordinary production run
        dict(name="drop3d", kind="run", dim=3, sx=64, sy=64, sz=128, d=16.0, steps=20),
        # the breaking-wave flume (4 905 180 particles, periodic across, piston, slope, slick): the
        # largest run, lists rebuilt every few steps
        dict(name="flume", kind="flume", width=0.3, group=2000, steps=5),
        # 256 uneven 2-D drops (4.6 M particles) in one persistent launch
        dict(name="batch256", kind="batch", k=256, group=3000, steps=10),
        # a handful of small drops in one persistent launch: grid barriers are the time
        dict(name="batch4", kind="batch", k=4, group=3000, steps=20),
        # a state held in pinned host memory, advanced by one step per call (coupling to a host code)
        dict(name="advance_host", kind="advance", dim=3, sx=64, sy=64, sz=128, d=16.0, steps=1),
        # one evaluation of the rates on a fresh neighbour list, read back: recording training data
        dict(name="record_rates", kind="eval", dim=3, sx=32, sy=32, sz=128, d=20.0),
        # a line of the run log: FP64 diagnostics and the positions for the oil's spread
        dict(name="log_line", kind="log", dim=3, sx=64, sy=64, sz=128, d=16.0),
        # one learned jump over k = 8 steps on the benchmark's drop
        dict(name="jump3d", kind="jump", dim=3, sx=64, sy=64, sz=128, d=16.0),
        # a training step of the surrogate on its 3-D training tank (193 496 particles) ...
        dict(name="train3d", kind="train", dim=3, sx=32, sy=32, sz=128, d=12.0),
        # ... and on a small 2-D tank, where its many launches are the time
        dict(name="train2d", kind="train", dim=2, sx=40, sy=1, sz=64, d=12.0),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above: tanks of 1 k to 800 k particles with odd sides, flumes of
    10 to 60 particles across, batches of 2 to 256, both viscous forms and boundary readings."""
    kind = rng.choice(["run", "run", "paper", "flume", "batch", "advance", "eval", "log", "jump", "train"])
    if kind == "paper":
        return dict(kind=kind, shape=rng.choice(["sphere", "cube"]), visc=rng.randint(0, 1),
                    renorm_walls=rng.randint(0, 1), steps=rng.randint(5, 40))
    if kind == "flume":
        return dict(kind=kind, width=round(5e-3 * rng.randint(10, 60), 6), group=rng.randint(0, 9999),
                    steps=rng.randint(2, 5))
    if kind == "batch":
        return dict(kind=kind, k=_logu(rng, 2, 256), group=rng.randint(0, 9999), steps=rng.randint(5, 10))
    dim = rng.choice([2, 3])
    if dim == 2:
        sx, sy, sz = _logu(rng, 20, 400), 1, _logu(rng, 30, 600)
        d = float(min(sx, sz) // 4)
    else:
        sx, sy, sz = _logu(rng, 10, 72), _logu(rng, 10, 72), _logu(rng, 16, 128)
        d = float(max(4, min(sx, sy, sz) // 4))
    c = dict(kind=kind, dim=dim, sx=sx, sy=sy, sz=sz, d=d)
    if kind == "train":   # training tanks stay below 200 k particles
        c.update(sx=min(sx, 32), sy=min(sy, 32))
    if kind == "run":
        c["steps"] = rng.randint(5, 20) if dim == 3 else rng.randint(10, 60)
    if kind == "advance":
        c["steps"] = rng.randint(1, 8)
    return c


# --------------------------------------------------------------------------
# Inputs


def _tank(case, seed):
    shape = (case["sx"], case["sz"]) if case["dim"] == 2 else (case["sx"], case["sy"], case["sz"])
    return WL.drop_tank(case["dim"], shape, drop_d_dx=case["d"], seed=seed)


def _stir(w, speed, seed, noise=0.02):
    """A smooth cellular flow of the given speed over the fluid (one roll per tank, zero on the
    boundary particles) with `noise` of it as jitter, and the density off its profile by 1e-6."""
    rng = np.random.Generator(np.random.PCG64(seed))
    fl = w.wall == 0
    x, d = w.x[fl], w.dim
    lo, hi = x.min(0), x.max(0)
    s = math.pi * (x - lo) / np.maximum(hi - lo, 1e-30)
    u = np.zeros((len(x), d))
    amp = speed * (1.0 + 0.1 * rng.uniform(-1, 1))
    u[:, 0] = amp * np.sin(s[:, 0]) * np.cos(s[:, d - 1])
    u[:, d - 1] = -amp * np.cos(s[:, 0]) * np.sin(s[:, d - 1])
    u += noise * speed * rng.uniform(-1, 1, u.shape)
    w.u[fl] = u
    w.rho *= 1.0 + 1e-6 * rng.uniform(-1, 1, len(w.rho))
    return w


def _workloads(case, seed):
    """The workloads of a case (one, or the instances of a batch)."""
    kind = case["kind"]
    if kind == "paper":
        w = WL.paper_drop(case["shape"], seed=seed, visc_form=case["visc"], renorm_walls=case["renorm_walls"])
        return [_stir(w, 0.08, seed + 1)]
    if kind == "flume":
        # the tank and its piston signal go by the wave group; the state by the seed
        w = WL.wave_tank(width=case["width"], seed=case["group"], renorm_walls=0)
        # a regular wave of 1 Hz under way: orbital velocities of linear theory
        m = w.meta
        omega = 2.0 * math.pi
        k = WL.dispersion_k(omega, m["depth"])
        fl = w.wall == 0
        rng = np.random.Generator(np.random.PCG64(seed))
        w.rho[fl] *= 1.0 + 1e-6 * rng.uniform(-1, 1, int(fl.sum()))
        ph = k * w.x[fl, 0] + rng.uniform(0, 2 * math.pi)
        z = np.maximum(w.x[fl, 2], 0.0)
        amp = 0.04 * omega / math.sinh(k * m["depth"])
        w.u[fl, 0] = amp * np.cosh(k * z) * np.cos(ph)
        w.u[fl, 2] = amp * np.sinh(k * z) * np.sin(ph)
        return [w]
    if kind == "batch":
        ws = WL.drop_batch_2d(case["k"], seed=case["group"])   # the group draws the tanks and fluids
        return [_stir(w, 0.02, seed + 1 + q) for q, w in enumerate(ws)]
    return [_stir(_tank(case, seed), 0.03, seed + 1)]


def _norm(w):
    """A normalisation block of the size a fit to such trajectories gives: inputs and outputs at
    unit spread for a drop rising at a few centimetres a second."""
    dim = w.dim
    T = K_JUMP * WL.stable_dt(w.params)
    fl = w.wall == 0
    rho0 = np.asarray(w.params["rho0"])[w.phase]
    dev = (w.rho / rho0 - 1.0)[fl]
    a = 5.0
    mu_in = np.concatenate([np.zeros(dim), [dev.mean()], [0.0, 0.0], np.zeros(dim), [0.0]])
    sd_in = np.concatenate([np.full(dim, w.u[fl].std()), [dev.std()], [1.0, 1.0], np.full(dim, T * a), [3e-4]])
    sd_out = np.concatenate([np.full(dim, T * T * a / 12.0), np.full(dim, 0.3 * T * a), [3e-4]])
    return SL.make_norm(dim, mu_in, sd_in, np.zeros(2 * dim + 1), sd_out, 20.0 if dim == 2 else 80.0, T,
                        0.1 * w.u[fl].std(), 0.2 * dev.std())


def _weights(dim, seed):
    return SL.init_weights(dim, seed=seed + 7)


def _target(w, norm, seed):
    """A state one jump later: the uniform motion and a spread of the normalised size around it."""
    dim = w.dim
    rng = np.random.Generator(np.random.PCG64(seed + 11))
    _, _, _, sd, _, T, _, _ = SL.split_norm(norm, dim)
    fl = (w.wall == 0)[:, None]
    rho0 = np.asarray(w.params["rho0"])[w.phase]
    u1 = w.u + fl * rng.standard_normal(w.u.shape) * sd[dim:2 * dim]
    x1 = w.x + fl * (0.5 * T * (w.u + u1) + rng.standard_normal(w.x.shape) * sd[:dim])
    return x1, u1, w.rho + rng.standard_normal(w.n) * sd[2 * dim] * rho0


def _device(*arrays):
    return [torch.tensor(a, dtype=torch.float64, device="cuda") for a in arrays]


def _pinned(*arrays):
    out = []
    for a in arrays:
        t = torch.empty(a.shape, dtype=torch.float64, pin_memory=True).numpy()
        t[...] = a
        out.append(t)
    return out


def _ptrs(tensors):
    return [t.data_ptr() for t in tensors]


def prepare(case, seed):
    """A handle on a stream of the program's own, and the state it will be given."""
    ws = _workloads(case, seed)
    w = ws[0]
    kind = case["kind"]
    stream = torch.cuda.Stream()
    s = dict(case=case, stream=stream)
    if kind == "batch":
        s["sim"] = sph.Simulation.batch(ws, stream=stream.cuda_stream)
        s["dt"], scales = WL.batch_dt(ws)
        s["sim"].set_dt_scales(scales)
    else:
        s["sim"] = sph.Simulation.from_workload(w, stream=stream.cuda_stream)
        s["dt"] = WL.stable_dt(w.params)
    if kind == "flume":
        m = w.meta["piston"]
        s["sim"].set_piston(m["axis"], m["amp"], m["omega"], m["phase"], m["t_end"])
    state = [np.concatenate([getattr(v, f) for v in ws]) for f in ("x", "u", "rho")]
    if kind == "advance":
        s["state"] = _pinned(*state)
        s["out"] = _pinned(*state)
        s["sim"].run(s["dt"], 1)     # the coupling loop has taken a step already
    else:
        s["state"] = _device(*state)
        s["out"] = [torch.empty_like(t) for t in s["state"]]
    if kind == "eval":
        s["out"] = _pinned(np.zeros((w.n, w.dim)), np.zeros(w.n), np.zeros(w.n))
    if kind == "log":
        s["out"] = _pinned(np.zeros((w.n, w.dim)))
        s["sim"].run(s["dt"], 1)
        s["sim"].load_snapshot(*_ptrs(s["state"]))
    if kind in ("jump", "train"):
        norm = _norm(w)
        s["sim"].surrogate_init(_weights(w.dim, seed), norm)
        if kind == "train":
            s["target"] = _device(*_target(w, norm, seed))
    return s


def run(s):
    case, sim = s["case"], s["sim"]
    kind = case["kind"]
    if kind == "advance":
        sim.advance_host(s["dt"], case["steps"], *s["state"], out=s["out"])
        return s["out"]
    if kind == "log":
        d = sim.diagnostics()
        return [d, sim.read("pos", out=s["out"][0])]
    sim.load_snapshot(*_ptrs(s["state"]))
    if kind == "eval":
        sim.eval_rates()
        return [sim.read(f, out=o) for f, o in zip(("acc", "drho", "pressure"), s["out"])]
    if kind == "train":
        loss, grad = sim.surrogate_train_step(*_ptrs(s["target"]), lr=1e-6, update=True, want_grad=True)
        return [loss, grad]
    if kind == "jump":
        sim.surrogate_advance(K_JUMP)
    elif kind == "batch":
        sim.run_persistent(s["dt"], case["steps"])
    else:
        if kind == "flume":
            sim.set_time(0.0)
        sim.run(s["dt"], case["steps"])
    sim.snapshot_to(*_ptrs(s["out"]))
    return s["out"]


# --------------------------------------------------------------------------
# Work: each state read and written once, and the arithmetic of the pairs within 2h (a force term of
# 43 flops twice a step and a renormalisation term of 27 once in 3-D; 33 and 22 in 2-D).


def _particles(case):
    kind = case["kind"]
    if kind == "paper":
        return 96148
    if kind == "flume":
        return int(round(4905180 * case["width"] / 0.3))
    if kind == "batch":
        return 17900 * case["k"]
    if case["dim"] == 2:
        return (case["sx"] + 6) * (case["sz"] + 6)
    return (case["sx"] + 6) * (case["sy"] + 6) * (case["sz"] + 6)


def work(case):
    kind, n = case["kind"], _particles(case)
    dim = 2 if kind == "batch" else case.get("dim", 3)
    pairs = n * (73.6 if dim == 3 else 21.2)
    state = 8.0 * (2 * dim + 1) * n
    step = pairs * (113 if dim == 3 else 88)
    if kind == "log":
        return dict(bytes=state + n + 8.0 * dim * n, flops=20.0 * n)
    if kind == "eval":
        return dict(bytes=state + 8.0 * (dim + 2) * n, flops=pairs * (70 if dim == 3 else 55))
    H, nin, nout, ne = 128, 2 * dim + 4, 2 * dim + 1, 2 * dim + 3
    dense = nin * H + H * H + 2 * (2 * H * H + H * H + 2 * H * H + H * H) + H * H + H * nout
    net = 2.0 * n * dense + 2 * pairs * H * (2 * ne + 6)
    rates = pairs * (70 if dim == 3 else 55)
    if kind == "jump":
        return dict(bytes=2 * state, flops=rates + net)
    if kind == "train":
        return dict(bytes=2 * state + 8.0 * SL.size(dim), flops=rates + 3 * net)
    return dict(bytes=2 * state, flops=step * case["steps"])


# --------------------------------------------------------------------------
# The same in 64 bits


class _Exact:
    """The two-phase method on torch tensors in 64 bits, particle arrays as in the workload."""

    CHUNK = 8_000_000

    def __init__(self, ws, dt, scales=None):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=self.dev)  # noqa: E731
        p = self.p = ws[0].params
        self.dim, self.h = ws[0].dim, p["h"]
        self.x = T(np.concatenate([w.x for w in ws]))
        self.u = T(np.concatenate([w.u for w in ws]))
        self.rho = T(np.concatenate([w.rho for w in ws]))
        self.phase = T(np.concatenate([w.phase for w in ws])).long()
        self.wall = T(np.concatenate([w.wall for w in ws]))
        count = [w.n for w in ws]
        inst = np.repeat(np.arange(len(ws)), count)
        per = lambda f: T(np.array([f(w) for w in ws], float)[inst])  # noqa: E731
        both = lambda f: T(np.array([f(w) for w in ws], float)[inst, np.concatenate([w.phase for w in ws])])  # noqa: E731
        self.rho0, self.mass = both(lambda w: w.params["rho0"]), both(lambda w: w.params["mass"])
        self.mu = both(lambda w: w.params["mu"])
        self.beta = self.rho0 * per(lambda w: w.params["c0"] ** 2) / 7.0
        self.tension = per(lambda w: w.params["alpha_s"])
        self.dt = dt * (per(lambda w: 1.0) if scales is None else T(np.asarray(scales, float)[inst]))
        # instances of a batch side by side, far apart
        self.shift = torch.zeros_like(self.x)
        if len(ws) > 1:
            ext = np.array([w.params["box_hi"][0] - w.params["box_lo"][0] for w in ws])
            self.shift[:, 0] = T((np.cumsum(ext + 10 * self.h) - ext)[inst])
        self.length = [p["box_hi"][a] - p["box_lo"][a] if (p.get("periodic", 0) >> a) & 1 else 0.0
                       for a in range(self.dim)]
        self.g = T(np.array(p["g"][:self.dim], float))
        self.piston = ws[0].meta.get("piston")
        self.t, self.step_no = 0.0, 0
        self.pairs_at = None

    def _pairs(self):
        """Ordered pairs closer than 2.2 h, sorted by the first: a list kept while nothing has moved
        by more than 0.1 h."""
        x = self.x + self.shift
        if self.pairs_at is not None and float((x - self.pairs_at).abs().max()) < 0.05 * self.h:
            return
        self.pairs_at = x
        n, dim, R = len(x), self.dim, 2.2 * self.h
        lo = x.min(0).values
        dims, cell = [], torch.zeros(n, dtype=torch.long, device=self.dev)
        cc = []
        for a in range(dim):
            if self.length[a]:
                m = max(1, int(self.length[a] / R))
                org, e = self.p["box_lo"][a], self.length[a] / m
                c = torch.remainder(torch.floor((x[:, a] - org) / e).long(), m)
            else:
                c = torch.floor((x[:, a] - lo[a]) / R).long()
                m = int(c.max()) + 1
            dims.append(m)
            cc.append(c)
        stride, tot = [], 1
        for a in range(dim):
            stride.append(tot)
            cell += cc[a] * tot
            tot *= dims[a]
        order = torch.argsort(cell)
        sc = cell[order]
        start = torch.searchsorted(sc, torch.arange(tot + 1, device=self.dev))
        got = []
        offs = torch.cartesian_prod(*[torch.arange(-1, 2)] * dim).tolist()
        step = max(1, self.CHUNK // 25)
        for b in range(0, n, step):
            i0 = torch.arange(b, min(n, b + step), device=self.dev)
            for off in offs:
                c = torch.zeros_like(i0)
                ok = torch.ones_like(i0, dtype=torch.bool)
                for a in range(dim):
                    v = cc[a][i0] + off[a]
                    if self.length[a]:
                        v = torch.remainder(v, dims[a])
                    else:
                        ok &= (v >= 0) & (v < dims[a])
                    c += v * stride[a]
                i, c = i0[ok], c[ok]
                s, e = start[c], start[c + 1]
                cnt = e - s
                k = int(cnt.sum())
                if not k:
                    continue
                ii = torch.repeat_interleave(i, cnt)
                first = torch.repeat_interleave(s - (torch.cumsum(cnt, 0) - cnt), cnt)
                jj = order[first + torch.arange(k, device=self.dev)]
                r = self._vec(x, ii, jj)
                keep = ((r * r).sum(1) < R * R) & (ii != jj)
                got.append((ii[keep].int(), jj[keep].int()))
        self.pi = torch.cat([a for a, _ in got])
        self.pj = torch.cat([b for _, b in got])

    def _vec(self, x, i, j):
        r = x[i] - x[j]
        for a in range(self.dim):
            if self.length[a]:
                r[:, a] -= self.length[a] * torch.round(r[:, a] / self.length[a])
        return r

    def _chunks(self):
        x = self.x + self.shift
        for b in range(0, len(self.pi), self.CHUNK):
            i, j = self.pi[b:b + self.CHUNK].long(), self.pj[b:b + self.CHUNK].long()
            r = self._vec(x, i, j)
            r2 = (r * r).sum(1)
            keep = r2 < 4 * self.h * self.h
            i, j, r, r2 = i[keep], j[keep], r[keep], r2[keep]
            yield i, j, r, r2, torch.sqrt(r2)

    def rates(self, renorm):
        """(density after the renormalisation, pressure, acceleration, density rate)."""
        self._pairs()
        h, dim = self.h, self.dim
        ad = 7 / (4 * math.pi * h ** 2) if dim == 2 else 21 / (16 * math.pi * h ** 3)
        rin, vol = self.rho, self.mass / self.rho
        num, den = self.mass * ad, vol * ad
        grad = torch.zeros_like(self.x)
        for i, j, r, r2, d in self._chunks():
            t = 1 - 0.5 * d / h
            same = self.phase[i] == self.phase[j]
            if renorm:
                W = ad * t ** 4 * (2 * d / h + 1) * same
                num.index_add_(0, i, self.mass[j] * W)
                den.index_add_(0, i, vol[j] * W)
            o = ~same
            if bool(o.any()):
                i, j, r, t = i[o], j[o], r[o], t[o]
                f = vol[j] ** 2 * ad * (-5 / h ** 2) * t ** 3 / vol[i]
                grad.index_add_(0, i, f[:, None] * r)
        rho = rin.clone()
        if renorm:
            who = torch.ones_like(rin, dtype=torch.bool) if self.p.get("renorm_walls", 1) else self.wall == 0
            rho = torch.where(who, num / den, rin)
        P = self.beta * ((rho / self.rho0) ** 7 - 1)
        g2 = (grad * grad).sum(1)
        gn = torch.sqrt(g2)
        eye = torch.eye(dim, dtype=torch.float64, device=self.dev)
        face = g2 > 0
        Tn = torch.zeros((len(rho), dim, dim), dtype=torch.float64, device=self.dev)
        gf = grad[face]
        Tn[face] = ((self.tension * (self.mass / rho) ** 2)[face] / gn[face])[:, None, None] * (
            g2[face][:, None, None] / dim * eye - gf[:, :, None] * gf[:, None, :])
        pr, vol = P / rho ** 2, self.mass / rho
        visc = self.mu if self.p["visc_form"] == 0 else self.mu / self.rho0
        acc, div = torch.zeros_like(self.x), torch.zeros_like(rho)
        delta2 = self.p["delta"] ** 2
        for i, j, r, r2, d in self._chunks():
            f = ad * (-5 / h ** 2) * (1 - 0.5 * d / h) ** 3
            uij = self.u[i] - self.u[j]
            c = -self.mass[j] * (pr[i] + pr[j]) * f
            vi, vj = visc[i], visc[j]
            s = vi + vj
            hm = torch.where(s > 0, 2 * vi * vj / torch.where(s > 0, s, torch.ones_like(s)), torch.zeros_like(s))
            k = 2 * hm * vol[j] * f * r2 / (r2 + delta2)
            if self.p["visc_form"] == 0:
                k = k / rho[i]
            acc.index_add_(0, i, c[:, None] * r + k[:, None] * uij)
            div.index_add_(0, i, vol[j] * f * (uij * r).sum(1))
            o = face[i] | face[j]
            if bool(o.any()):
                i, j, r, f = i[o], j[o], r[o], f[o]
                acc.index_add_(0, i, ((Tn[i] + Tn[j]) @ r[:, :, None])[:, :, 0] * (f / self.mass[i])[:, None])
        acc = torch.where((self.wall > 0)[:, None], torch.zeros_like(acc), acc + self.g)
        return rho, P, acc, rho * div

    def _moved(self, t):
        m = self.piston
        X = lambda s: sum(a * (math.sin(w * s + f) - math.sin(f)) for a, w, f in zip(m["amp"], m["omega"], m["phase"]))  # noqa: E731
        U = sum(a * w * math.cos(w * t + f) for a, w, f in zip(m["amp"], m["omega"], m["phase"]))
        return X(t) - X(self.t), U

    def step(self):
        every = self.p["renorm_every"]
        x0, u0 = self.x, self.u
        rho0, _, a, dr = self.rates(every > 0 and self.step_no % every == 0)
        dt, free = self.dt, (self.wall == 0)[:, None]
        pist = (self.wall == 2) if self.piston else None
        at = float(dt[0])

        def place(x, u, t):
            if pist is None:
                return x, u
            dX, U = self._moved(t)
            ax = self.piston["axis"]
            e = torch.zeros(self.dim, dtype=torch.float64, device=self.dev)
            e[ax] = 1.0
            return torch.where(pist[:, None], x0 + dX * e, x), torch.where(pist[:, None], U * e, u)

        half = 0.5 * dt[:, None]
        self.x, self.u = place(torch.where(free, x0 + half * u0, x0), torch.where(free, u0 + half * a, u0),
                               self.t + 0.5 * at)
        self.rho = rho0 + 0.5 * dt * dr
        _, _, a, dr = self.rates(False)
        us = self.u
        self.x, self.u = place(torch.where(free, x0 + dt[:, None] * us, x0), torch.where(free, u0 + dt[:, None] * a, u0),
                               self.t + at)
        self.rho = rho0 + dt * dr
        self.t += at
        self.step_no += 1

    def state(self):
        x = self.x.clone()
        for a in range(self.dim):
            if self.length[a]:
                x[:, a] = self.p["box_lo"][a] + torch.remainder(x[:, a] - self.p["box_lo"][a], self.length[a])
        return [x, self.u, self.rho]


class _Network:
    """The message-passing network in 64 bits on an _Exact state, forward and backward by hand."""

    CHUNK = 400_000

    def __init__(self, E, flat, norm, dim):
        self.E, self.dim = E, dim
        t = lambda a: torch.as_tensor(np.asarray(a, float), device=E.dev)  # noqa: E731
        self.W = {k: t(v) for k, v in SL.unflatten(flat.astype(np.float32).astype(float), dim).items()}
        self.mu_in, self.sd_in, self.mu_out, self.sd_out = (t(v) for v in SL.split_norm(norm, dim)[:4])
        self.k, self.T, self.su, self.sr = SL.split_norm(norm, dim)[4:]
        _, _, self.a, self.dr = E.rates(True)
        self.dev = (E.rho - E.rho0) / E.rho0
        raw = torch.cat([E.u, self.dev[:, None], E.phase[:, None].double(), (E.wall > 0)[:, None].double(),
                         self.T * self.a, (self.T * self.dr / E.rho0)[:, None]], 1)
        self.X = (raw - self.mu_in) / self.sd_in

    def _edges(self):
        E = self.E
        for b in range(0, len(E.pi), self.CHUNK):
            i, j = E.pi[b:b + self.CHUNK].long(), E.pj[b:b + self.CHUNK].long()
            r = E._vec(E.x + E.shift, i, j)
            r2 = (r * r).sum(1)
            keep = r2 < 4 * E.h * E.h
            i, j, r, r2 = i[keep], j[keep], r[keep], r2[keep]
            yield i, j, torch.cat([r / (2 * E.h), torch.sqrt(r2)[:, None] / (2 * E.h),
                                   (E.phase[i] != E.phase[j])[:, None].double(), (E.u[i] - E.u[j]) / self.su,
                                   ((self.dev[i] - self.dev[j]) / self.sr)[:, None]], 1)

    def forward(self):
        W, silu = self.W, torch.nn.functional.silu
        self.z0 = self.X @ W["enc1.w"].T + W["enc1.b"]
        self.h = [silu(self.z0) @ W["enc2.w"].T + W["enc2.b"]]
        self.kept = []
        n = len(self.X)
        self.deg = torch.zeros(n, dtype=torch.float64, device=self.X.device)
        for r in range(2):
            h = self.h[-1]
            P, Q = h @ W[f"r{r}.w1"].T + W[f"r{r}.b1"], h @ W[f"r{r}.w2"].T
            S = torch.zeros_like(h)
            for i, j, e in self._edges():
                S.index_add_(0, i, silu(P[i] + Q[j] + e @ W[f"r{r}.w3"].T))
                if r == 0:
                    self.deg.index_add_(0, i, torch.ones_like(e[:, 0]))
            S /= self.k
            M = S @ W[f"r{r}.we2"].T + (self.deg / self.k)[:, None] * W[f"r{r}.be2"]
            A = torch.cat([h, M], 1)
            Z = A @ W[f"r{r}.n1"].T + W[f"r{r}.n1b"]
            self.kept.append((P, Q, S, A, Z))
            self.h.append(h + silu(Z) @ W[f"r{r}.n2"].T + W[f"r{r}.n2b"])
        self.z2 = self.h[2] @ W["dec1.w"].T + W["dec1.b"]
        return silu(self.z2) @ W["dec2.w"].T + W["dec2.b"]

    def jump(self):
        E, d, T = self.E, self.dim, self.T
        D = self.forward() * self.sd_out + self.mu_out
        free = (E.wall == 0)[:, None]
        du = T * self.a + D[:, d:2 * d]
        return [torch.where(free, E.x + T * (E.u + 0.5 * du) + D[:, :d], E.x), torch.where(free, E.u + du, E.u),
                E.rho + T * self.dr + D[:, 2 * d] * E.rho0]

    def loss_and_gradient(self, x1, u1, r1):
        E, d, T, W = self.E, self.dim, self.T, self.W
        dsilu = lambda z: torch.sigmoid(z) * (1 + z * (1 - torch.sigmoid(z)))  # noqa: E731
        silu = torch.nn.functional.silu
        y = self.forward()
        D = torch.cat([x1 - E.x - 0.5 * T * (E.u + u1), u1 - E.u - T * self.a,
                       ((r1 - E.rho) / E.rho0 - T * self.dr / E.rho0)[:, None]], 1)
        mask = torch.ones_like(y)
        mask[E.wall > 0, :2 * d] = 0
        err = (y - (D - self.mu_out) / self.sd_out) * mask
        loss = float((err * err).sum() / mask.sum())
        dy = 2 * err / mask.sum()
        G = {}
        G["dec2.w"], G["dec2.b"] = dy.T @ silu(self.z2), dy.sum(0)
        dz = dy @ W["dec2.w"] * dsilu(self.z2)
        G["dec1.w"], G["dec1.b"] = dz.T @ self.h[2], dz.sum(0)
        dh = dz @ W["dec1.w"]
        for r in (1, 0):
            P, Q, S, A, Z = self.kept[r]
            h = self.h[r]
            H = h.shape[1]
            G[f"r{r}.n2"], G[f"r{r}.n2b"] = dh.T @ silu(Z), dh.sum(0)
            dz = dh @ W[f"r{r}.n2"] * dsilu(Z)
            G[f"r{r}.n1"], G[f"r{r}.n1b"] = dz.T @ A, dz.sum(0)
            dA = dz @ W[f"r{r}.n1"]
            dM = dA[:, H:]
            G[f"r{r}.we2"], G[f"r{r}.be2"] = dM.T @ S, ((self.deg / self.k)[:, None] * dM).sum(0)
            dS = dM @ W[f"r{r}.we2"] / self.k
            dP, dQ, g3 = torch.zeros_like(h), torch.zeros_like(h), torch.zeros_like(W[f"r{r}.w3"])
            for i, j, e in self._edges():
                q = dS[i] * dsilu(P[i] + Q[j] + e @ W[f"r{r}.w3"].T)
                dP.index_add_(0, i, q)
                dQ.index_add_(0, j, q)
                g3 += q.T @ e
            G[f"r{r}.w3"], G[f"r{r}.b1"] = g3, dP.sum(0)
            G[f"r{r}.w1"], G[f"r{r}.w2"] = dP.T @ h, dQ.T @ h
            dh = dh + dA[:, :H] + dP @ W[f"r{r}.w1"] + dQ @ W[f"r{r}.w2"]
        G["enc2.w"], G["enc2.b"] = dh.T @ silu(self.z0), dh.sum(0)
        dz = dh @ W["enc2.w"] * dsilu(self.z0)
        G["enc1.w"], G["enc1.b"] = dz.T @ self.X, dz.sum(0)
        return [loss, torch.cat([G[name].reshape(-1) for name, _ in SL.layout(d)])]


def _diagnostics(w):
    """The log's quantities by numpy: sums over the fluid, moments of the oil."""
    fl, oil = w.wall == 0, (w.wall == 0) & (w.phase == 1)
    m = np.asarray(w.params["mass"])[w.phase][fl]
    x, u, d = w.x[fl], w.u[fl], w.dim
    xo = w.x[oil]
    c = xo.mean(0)
    ev = np.linalg.eigvalsh((xo - c).T @ (xo - c) / len(xo))
    g = np.asarray(w.params["g"][:d])
    return dict(mass=m.sum(), momentum=(m[:, None] * u).sum(0), e_kin=0.5 * (m * (u * u).sum(1)).sum(),
                e_pot=-(m * (x @ g)).sum(), centroid=c, sphericity=np.sqrt(ev[0] / ev[-1]),
                u_max=np.sqrt((u * u).sum(1)).max(), n_oil=int(oil.sum()))


def exact(case, seed):
    kind = case["kind"]
    ws = _workloads(case, seed)
    w = ws[0]
    if kind == "log":
        return [_diagnostics(w), w.x]
    scales = None
    dt = WL.stable_dt(w.params)
    if kind == "batch":
        dt, scales = WL.batch_dt(ws)
    E = _Exact(ws, dt, scales)
    if kind == "eval":
        _, P, a, dr = E.rates(True)
        return [a, dr, P]
    if kind in ("jump", "train"):
        norm = _norm(w)
        net = _Network(E, _weights(w.dim, seed), norm, w.dim)
        if kind == "jump":
            return net.jump()
        return net.loss_and_gradient(*[torch.as_tensor(a, device=E.dev) for a in _target(w, norm, seed)])
    for _ in range(case["steps"]):
        E.step()
    return E.state()
