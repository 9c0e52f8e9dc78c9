"""The work that a user of this library has it do, as cases to be timed.

Each case is one call, or the few calls of one outer iteration, through the public binding
(``paper_1906_01413_gb300.riot``):

  hvp      riot_hessian_apply on a linearised Lorenz-96 window: the product that every
           method here (RIOT, VarCG, VarBL) spends its time on
  outer    riot_outer_begin on a Lorenz-96 window: trajectory, innovation, gradient
  loop     one inner loop, riot_rsvd and riot_increment, in mixed precision or in FP64
  batch    one outer iteration of several Lorenz-96 windows of uneven size together
  tracer   riot_hessian_apply of the tracer-transport inversion
  emission riot_outer_begin of the tracer-transport inversion (FP64)
  sketch   loss and gradient of the learned sketch network, the step its training repeats

Inputs come from the seed alone and from torch (not from the library), so that they are the
same whatever the library's rounding.  Loops use the paper's Lorenz-96 step dt = 0.01
(Section 3.1) over windows short enough for FP32 products to resolve every pair of the sketch;
results of mixed-precision loops are kept in FP32, which is what such a context resolves.
"""
import random

import numpy as np
import torch

from paper_1906_01413_gb300 import riot as R
from synth.advdiff import AdvDiffConfig

DEV = "cuda:0"
F64, F32 = torch.float64, torch.float32


def listed():
    return [
        # the small parity window at full rank: launch latency and the shortest chunks
        dict(name="hvp_l96_small", kind="hvp", n=40, T=20, dt=0.05, F=8.0, ncols=40, every=1, frac=0.5, ell=2.0),
        # a batch-sized window with odd sizes everywhere
        dict(name="hvp_l96_ragged", kind="hvp", n=1003, T=97, dt=0.01, F=11.3, ncols=77, every=4, frac=0.31, ell=4.0),
        # the headline window's product (512 sketch columns)
        dict(name="hvp_l96_large", kind="hvp", n=4096, T=200, dt=0.05, F=8.0, ncols=512, every=4, frac=0.25, ell=4.0),
        # the widest states the model takes, a short last chunk
        dict(name="hvp_l96_wide", kind="hvp", n=8191, T=150, dt=0.01, F=16.0, ncols=192, every=4, frac=0.1, ell=4.0),
        # what each outer iteration pays before its inner loop, at the headline size
        dict(name="outer_l96", kind="outer", n=4096, T=200, dt=0.01, F=8.0, every=4, frac=0.25, ell=4.0),
        # the headline inner loop: k = 512, one power iteration
        dict(name="loop_l96_mixed", kind="loop", fp64=False, n=4096, T=100, dt=0.01, F=8.0, k=512, q=1, every=4,
             frac=0.25, ell=4.0),
        # the FP64 form of the loop, on a mid-sized window
        dict(name="loop_l96_fp64", kind="loop", fp64=True, n=1000, T=60, dt=0.01, F=8.0, k=128, q=1, every=4,
             frac=0.25, ell=4.0),
        # twelve windows of uneven size, linearised and solved together
        dict(name="batch_l96", kind="batch", nwin=12, n_max=8192, wseed=7),
        # the full tracer box, a slice of 32 sketch columns (a pass of 128 is four of these)
        dict(name="tracer_full", kind="tracer", nx=192, ny=192, nz=30, nb=4, T=240, ncols=32, ntr=20, npt=400),
        # a small ragged box, where a step is shorter than its launch
        dict(name="tracer_box", kind="tracer", nx=37, ny=23, nz=11, nb=3, T=48, ncols=16, ntr=4, npt=60),
        # the FP64 outer iteration of a quarter-size box
        dict(name="emission_outer", kind="emission", nx=96, ny=96, nz=30, nb=4, T=60, ntr=20, npt=100),
        # one training batch of the learned sketch network at its benchmark sizes
        dict(name="sketch_train", kind="sketch", n=4096, batch=8, c_in=8, width=64, m=128, r=128),
    ]


def _log_int(rng, lo, hi):
    return int(min(hi, max(lo, round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    kind = rng.choice(["hvp", "hvp", "hvp", "outer", "loop", "loop", "batch", "tracer", "tracer", "emission", "sketch"])
    win = dict(every=rng.choice([1, 2, 4]), frac=round(rng.uniform(0.1, 0.5), 3), ell=rng.choice([2.0, 4.0]),
               F=round(rng.uniform(8.0, 16.0), 2))
    if kind == "hvp":
        n, T = _log_int(rng, 40, 8192), _log_int(rng, 20, 300)
        cap = max(1, 4096 * 200 * 512 // (n * T))
        return dict(kind=kind, n=n, T=T, dt=0.01, ncols=_log_int(rng, 1, min(512, cap)), **win)
    if kind == "outer":
        return dict(kind=kind, n=_log_int(rng, 40, 8192), T=_log_int(rng, 20, 200), dt=0.01, **win)
    if kind == "loop":
        fp64 = rng.random() < 0.4
        n = _log_int(rng, 200, 2000 if fp64 else 8192)
        win["F"] = round(rng.uniform(8.0, 9.0), 2)
        return dict(kind=kind, fp64=fp64, n=n, T=rng.randint(20, 60), dt=0.01,
                    k=_log_int(rng, 16, min(128 if fp64 else 512, n // 4)), q=rng.randint(0, 1), **win)
    if kind == "batch":
        return dict(kind=kind, nwin=rng.randint(2, 12), n_max=_log_int(rng, 400, 8192), wseed=rng.randrange(1 << 20))
    if kind in ("tracer", "emission"):
        nx, ny, nz = _log_int(rng, 12, 192), _log_int(rng, 10, 192), rng.randint(4, 32)
        T = rng.randint(12, 60)
        cells = nx * ny * nz
        box = dict(kind=kind, nx=nx, ny=ny, nz=nz, nb=rng.randint(1, 4), T=T, ntr=rng.randint(2, 20), npt=rng.randint(40, 400))
        if kind == "tracer":
            box["ncols"] = _log_int(rng, 1, max(1, min(128, 192 * 192 * 30 * 240 * 32 // (cells * T))))
        return box
    return dict(kind=kind, n=_log_int(rng, 256, 4096), batch=rng.randint(1, 8), c_in=rng.choice([4, 8]),
                width=rng.choice([32, 64, 96]), m=rng.choice([64, 100, 128]), r=rng.choice([64, 128]))


# ---------------------------------------------------------------------------------------
# Inputs (torch and numpy only)
# ---------------------------------------------------------------------------------------
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + salt) % (1 << 62))
    return g


def _normal(seed, salt, *shape, dtype=F64):
    return torch.randn(*shape, dtype=dtype, device=DEV, generator=_gen(seed, salt))


def _tend(x, F):
    return (torch.roll(x, -1) - torch.roll(x, 2)) * torch.roll(x, 1) - x + F


def _stages(x, h, F):
    """The four RK4 stage states of one step and the state after it."""
    k1 = _tend(x, F)
    x2 = x + 0.5 * h * k1
    k2 = _tend(x2, F)
    x3 = x + 0.5 * h * k2
    k3 = _tend(x3, F)
    x4 = x + h * k3
    k4 = _tend(x4, F)
    return (x, x2, x3, x4), x + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)


def _taps(n, ell):
    """Offsets and weights of the periodic Gaussian convolution S (unit variance of S S^T)."""
    d = np.arange(n)
    row = sum(np.exp(-((d + j * n) ** 2) / ell ** 2) for j in range(-int(40 * ell / n) - 2, int(40 * ell / n) + 3))
    row /= np.sqrt((row ** 2).sum())
    return [(int(i) if i <= n // 2 else int(i) - n, float(row[i])) for i in range(n) if row[i] > 1e-18 * row[0]]


def _conv(x, taps):
    return sum(w * torch.roll(x, d, -1) for d, w in taps)


def _window(case, seed):
    """Truth on the attractor, observations of it, background; host observation arrays."""
    n, T, dt, F = case["n"], case["T"], case["dt"], case["F"]
    x = F + 0.1 * _normal(seed, 1, n)
    for _ in range(120):   # spin-up at the longer step
        x = _stages(x, 0.05, F)[1]
    pick = np.random.default_rng(int(seed) + 17)
    idx = np.sort(pick.choice(n, max(1, round(case["frac"] * n)), replace=False)).astype(np.int32)
    steps = np.arange(case["every"], T + 1, case["every"], dtype=np.int32)
    at = torch.tensor(idx.astype(np.int64), device=DEV)
    y, t = [], x
    for s in range(1, T + 1):
        t = _stages(t, dt, F)[1]
        if s % case["every"] == 0:
            y.append(t[at])
    y = torch.cat(y) + _normal(seed, 2, len(steps) * idx.size)
    taps = _taps(n, case["ell"])
    return dict(n=n, T=T, dt=dt, F=F, steps=steps, idx=idx, at=at, taps=taps, y=y,
                xb=x + _conv(_normal(seed, 3, n), taps), v0=torch.zeros(n, dtype=F64, device=DEV))


def _context(case, w, kmax, fp64=False):
    st, ix = np.repeat(w["steps"], w["idx"].size), np.tile(w["idx"], w["steps"].size)
    return R.Context(n=w["n"], T=w["T"], dt=w["dt"], F=w["F"], obs_step=st, obs_idx=ix, obs_y=w["y"].cpu().numpy(),
                     obs_sigma=np.ones(st.size), length=case["ell"], sigma_b=1.0, kmax=kmax,
                     precision=R.RIOT_PREC_FP64 if fp64 else R.RIOT_PREC_MIXED)


def _batch_cases(case):
    """The windows of a batch: sizes as the batched workload draws them, at the paper's step."""
    rng = random.Random(case["wseed"])
    out = []
    for _ in range(case["nwin"]):
        n = _log_int(rng, 40, case["n_max"])
        out.append(dict(n=n, T=rng.randint(40, 60), dt=0.01, F=round(rng.uniform(8.0, 9.0), 2), every=4, ell=4.0,
                        frac=round(rng.uniform(0.1, 0.5), 3), k=min(rng.choice([16, 64, 128, 256, 512]), max(8, n // 4))))
    return out


def _box(case, seed):
    c = AdvDiffConfig(name="box", nx=case["nx"], ny=case["ny"], nz=case["nz"], T=case["T"], nblocks=case["nb"],
                      n_tracks=case["ntr"], pts_per_track=case["npt"], seed=int(seed))
    u, v = c.winds()
    step, pos = c.tracks()
    return c, dict(u=u, v=v, amp=c.amplitude(), kz=c.kz(), emis_b=c.background_emissions(), obs_step=step, obs_pos=pos,
                   obs_y=0.2 * np.abs(c.obs_noise(step.size)), obs_sigma=np.full(step.size, 0.1)), \
        0.3 * _normal(seed, 4, c.n)


def _net(case, seed):
    C, W, M, depth, K = case["c_in"], case["width"], case["m"], 4, 5
    chan = [C] + [W] * (depth - 1) + [M]
    p = torch.cat([torch.cat([_normal(seed, 20 + l, chan[l + 1] * chan[l] * K) / (chan[l] * K) ** 0.5,
                              0.1 * _normal(seed, 40 + l, chan[l + 1])]) for l in range(depth)]).to(F32)
    x = _normal(seed, 5, case["batch"], C, case["n"], dtype=F32)
    U = torch.linalg.qr(_normal(seed, 6, case["batch"], case["n"], case["r"], dtype=F32).cpu())[0].mT.to(DEV).contiguous()
    return chan, K, p, x, U


# ---------------------------------------------------------------------------------------
class _Net:
    """Owner of a network handle."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        R.riot_sketchnet_destroy(self.h)


class _Batch:
    """Owner of a batch handle; the contexts outlive it."""

    def __init__(self, ctxs, ks):
        self.ctxs = ctxs
        self.h = R.riot_batch_create([c.h for c in ctxs], ks, 1)

    def __del__(self):
        R.riot_batch_destroy(self.h)


def prepare(case, seed):
    torch.cuda.set_device(0)
    kind, s = case["kind"], {"kind": case["kind"]}
    if kind in ("hvp", "outer"):
        w = _window(case, seed)
        s["xb"], s["v0"] = w["xb"], w["v0"]
        s["ctx"] = _context(case, w, case.get("ncols", 1))
        s["p"] = w["y"].numel()
        if kind == "hvp":
            R.riot_outer_begin(s["ctx"].h, w["xb"], w["v0"])
            s["W"] = _normal(seed, 7, case["ncols"], case["n"], dtype=F32)
            s["Y"] = torch.empty_like(s["W"])
        else:
            s["traj"] = torch.empty(case["T"] + 1, case["n"], dtype=F64, device=DEV)
            s["d"] = torch.empty(s["p"], dtype=F64, device=DEV)
            s["g"] = torch.empty(case["n"], dtype=F64, device=DEV)
    elif kind == "loop":
        w = _window(case, seed)
        s["ctx"] = _context(case, w, case["k"], case["fp64"])
        s.update(k=case["k"], q=case["q"], fp64=case["fp64"], dv=torch.empty(case["n"], dtype=F64, device=DEV),
                 Omega=_normal(seed, 7, case["k"], case["n"], dtype=F32).to(F64 if case["fp64"] else F32))
        R.riot_outer_begin(s["ctx"].h, w["xb"], w["v0"])
    elif kind == "batch":
        cs = _batch_cases(case)
        ws = [_window(c, seed + 31 * i) for i, c in enumerate(cs)]
        ctxs = [_context(c, w, c["k"]) for c, w in zip(cs, ws)]
        s["x0"], s["v0"] = [w["xb"] for w in ws], [w["v0"] for w in ws]
        s["x"], s["v"] = [torch.empty_like(w["xb"]) for w in ws], [torch.empty_like(w["xb"]) for w in ws]
        s["lam"] = [torch.empty(c["k"], dtype=F64, device=DEV) for c in cs]
        s["batch"] = _Batch(ctxs, [c["k"] for c in cs])
    elif kind in ("tracer", "emission"):
        c, box, x = _box(case, seed)
        s["ctx"] = R.Context(nx=c.nx, ny=c.ny, nz=c.nz, nblocks=c.nblocks, T=c.T, dt=c.dt, dx=c.dx, dy=c.dy, dz=c.dz,
                             length=c.ell, sigma_b=c.sigma_b, kmax=case.get("ncols", 1), **box)
        s["xb"], s["v0"] = x, torch.zeros_like(x)
        if kind == "tracer":
            R.riot_outer_begin(s["ctx"].h, x, s["v0"])
            s["W"] = _normal(seed, 7, case["ncols"], c.n, dtype=F32)
            s["Y"] = torch.empty_like(s["W"])
        else:
            s["d"] = torch.empty(box["obs_y"].size, dtype=F64, device=DEV)
            s["g"] = torch.empty(c.n, dtype=F64, device=DEV)
    else:
        chan, K, p, s["x"], s["U"] = _net(case, seed)
        s["net"] = _Net(R.riot_sketchnet_create(case["c_in"], case["width"], case["m"], n_max=case["n"],
                                                batch_max=case["batch"], r_max=case["r"]))
        R.riot_sketchnet_set_params(s["net"].h, p)
        s["grad"] = torch.empty_like(p)
    return s


def run(s):
    kind = s["kind"]
    if kind in ("hvp", "tracer"):
        R.riot_hessian_apply(s["ctx"].h, s["W"], s["Y"])
        return s["Y"]
    if kind == "outer":
        J = R.riot_outer_begin(s["ctx"].h, s["xb"], s["v0"])
        R.riot_get_trajectory(s["ctx"].h, s["traj"])
        R.riot_get_innovation(s["ctx"].h, s["d"])
        R.riot_get_state(s["ctx"].h, g=s["g"])
        return {"J": J, "traj": s["traj"], "d": s["d"], "g": s["g"]}
    if kind == "emission":
        J = R.riot_outer_begin(s["ctx"].h, s["xb"], s["v0"])
        R.riot_get_innovation(s["ctx"].h, s["d"])
        R.riot_get_state(s["ctx"].h, g=s["g"])
        return {"J": J, "d": s["d"], "g": s["g"]}
    if kind == "loop":
        lam = R.riot_rsvd(s["ctx"].h, s["k"], s["q"], Omega=s["Omega"])
        R.riot_increment(s["ctx"].h, s["dv"])
        return {"lam": lam, "dv": s["dv"]} if s["fp64"] else {"lam": lam.astype(np.float32), "dv": s["dv"].to(F32)}
    if kind == "batch":
        ctxs = s["batch"].ctxs
        for c, x, v in zip(ctxs, s["x0"], s["v0"]):
            R.riot_outer_begin(c.h, x, v)
        R.riot_batch_run(s["batch"].h, len(ctxs), sketch_stream=16)
        for c, x, v, lam in zip(ctxs, s["x"], s["v"], s["lam"]):
            R.riot_get_state(c.h, x=x, v=v, lam=lam)
        return {"lam": torch.cat(s["lam"]).to(F32), "v": torch.cat(s["v"]).to(F32), "x": torch.cat(s["x"]).to(F32)}
    loss = R.riot_sketchnet_loss_grad(s["net"].h, s["x"], s["U"], 0.1, s["grad"])
    return {"loss": loss, "grad": s["grad"]}


# ---------------------------------------------------------------------------------------
def work(case):
    """Bytes and operations that one pass cannot do without."""
    kind = case["kind"]

    def l96_product(c, cols):   # tangent linear, adjoint, L and L^T, residuals
        n, T = c["n"], c["T"]
        p = (T // c["every"]) * max(1, round(c["frac"] * n))
        return cols * ((33 + 34) * n * T + 4 * len(_taps(n, c["ell"])) * n + 3 * p)

    if kind == "hvp":
        n, T, k = case["n"], case["T"], case["ncols"]
        return {"bytes": 8 * n * k + 8 * (T + 1) * n, "flops": l96_product(case, k)}
    if kind == "outer":
        n, T = case["n"], case["T"]
        p = (T // case["every"]) * max(1, round(case["frac"] * n))
        return {"bytes": 8 * ((T + 1) * n + 3 * n + 2 * p), "flops": (28 + 34) * n * T + 8 * p}
    if kind in ("loop", "batch"):
        total = {"bytes": 0, "flops": 0}
        for c in ([case] if kind == "loop" else _batch_cases(case)):
            n, T, k, q = c["n"], c["T"], c["k"], c.get("q", 1)
            size = 8 if c.get("fp64") else 4
            total["bytes"] += size * n * k + 8 * ((T + 1) * n + 3 * n)
            # products, q + 1 orthonormalisations, Q^T W, Q^T Y and U = Q Z, the k x k chain
            total["flops"] += (q + 1) * (l96_product(c, k) + 2 * n * k * k) + 6 * n * k * k + 9 * k ** 3
            if kind == "batch":
                total["flops"] += (28 + 34) * n * T
        return total
    if kind in ("tracer", "emission"):
        cells, T, cols = case["nx"] * case["ny"] * case["nz"], case["T"], case.get("ncols", 1)
        n = case["nb"] * case["ny"] * case["nx"]
        size = 4 if kind == "tracer" else 8
        # a step of either direction reads and writes the tracer; four stages of ten operations pairs
        return {"bytes": 2 * T * 2 * size * cells * cols + 2 * size * n * cols,
                "flops": 2 * T * 4 * 20 * cells * cols + 4 * n * (case["nx"] + case["ny"]) * cols}
    n, B, M, r = case["n"], case["batch"], case["m"], case["r"]
    chan = [case["c_in"]] + [case["width"]] * 3 + [M]
    conv = [2 * 5 * a * b * n * B for a, b in zip(chan, chan[1:])]
    return {"bytes": 4 * B * n * (case["c_in"] + r) + 8 * sum(5 * a * b + b for a, b in zip(chan, chan[1:])),
            "flops": 3 * sum(conv) - conv[0] + 2 * B * n * M * (2 * r + 2 * M)}


# ---------------------------------------------------------------------------------------
# The same results in 64 bits, plain torch
# ---------------------------------------------------------------------------------------
class _L96:
    def __init__(self, case, seed):
        self.w = w = _window(case, seed)
        self.every, self.h = case["every"], w["dt"]
        self.stages, self.obs, x = [], [], w["xb"]
        self.traj = [x]
        for s in range(1, w["T"] + 1):
            st, x = _stages(x, w["dt"], w["F"])
            self.stages.append([(torch.roll(X, 1), torch.roll(X, -1) - torch.roll(X, 2)) for X in st])
            self.traj.append(x)
            if s % self.every == 0:
                self.obs.append(x[w["at"]])
        self.d = torch.cat(self.obs) - w["y"]

    @staticmethod
    def _tl(c, s):
        return c[0] * (torch.roll(s, -1, -1) - torch.roll(s, 2, -1)) + c[1] * torch.roll(s, 1, -1) - s

    @staticmethod
    def _ad(c, m):
        p = c[0] * m
        return torch.roll(p, 1, -1) - torch.roll(p, -2, -1) + torch.roll(c[1] * m, -1, -1) - m

    def forward(self, W):
        h, out, x = self.h, [], _conv(W, self.w["taps"])
        for t, c in enumerate(self.stages):
            k1 = self._tl(c[0], x)
            k2 = self._tl(c[1], x + 0.5 * h * k1)
            k3 = self._tl(c[2], x + 0.5 * h * k2)
            k4 = self._tl(c[3], x + h * k3)
            x = x + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
            if (t + 1) % self.every == 0:
                out.append(x[..., self.w["at"]])
        return out

    def backward(self, r):
        h, lam, o = self.h, None, len(r)
        for t in range(len(self.stages) - 1, -1, -1):
            if (t + 1) % self.every == 0:
                o -= 1
                if lam is None:
                    lam = torch.zeros(r[o].shape[:-1] + (self.w["n"],), dtype=F64, device=DEV)
                lam[..., self.w["at"]] += r[o]
            if lam is None:
                continue
            c = self.stages[t]
            l4 = self._ad(c[3], h / 6 * lam)
            l3 = self._ad(c[2], h / 3 * lam + h * l4)
            l2 = self._ad(c[1], h / 3 * lam + 0.5 * h * l3)
            l1 = self._ad(c[0], h / 6 * lam + 0.5 * h * l2)
            lam = lam + l1 + l2 + l3 + l4
        return _conv(lam, self.w["taps"])

    def product(self, W):
        return self.backward(self.forward(W))

    def gradient(self):
        return self.backward(list(self.d.split(self.w["idx"].size)))


def _loop_exact(m, Omega, k, q):
    W = Omega.to(F64)
    Y = m.product(W)
    for _ in range(q):
        W = torch.linalg.qr(Y.mT)[0].mT.contiguous()
        Y = m.product(W)
    Q = torch.linalg.qr(Y.mT)[0]
    K = torch.linalg.solve((Q.mT @ W.mT).mT, (Q.mT @ Y.mT).mT).mT
    lam, Z = torch.linalg.eigh(0.5 * (K + K.mT))
    U, g = Q @ Z, m.gradient()
    c = U.mT @ g
    dv = -U @ (c / (1 + lam)) if float(lam[0]) > 1 else -(g - U @ (c * lam / (1 + lam)))
    return lam.flip(0), dv


class _Tracer:
    def __init__(self, case, seed):
        c, b, x = _box(case, seed)
        t = lambda a: torch.tensor(a, dtype=F64, device=DEV)   # noqa: E731
        self.c, self.p = c, b["obs_y"].size
        u, v = t(b["u"]), t(b["v"])
        uL, uR, vS, vN = u, torch.roll(u, -1, 1), v[:-1], v[1:]
        up, un = (lambda a: a.clamp(min=0)), (lambda a: a.clamp(max=0))
        self.c0 = (un(uL) - up(uR)) / c.dx + (un(vS) - up(vN)) / c.dy
        self.tl = [-un(uR) / c.dx, up(uL) / c.dx, -un(vN) / c.dy, up(vS) / c.dy]   # east, west, north, south
        self.ad = [up(uR) / c.dx, -un(uL) / c.dx, up(vN) / c.dy, -un(vS) / c.dy]
        self.amp = t(b["amp"]).view(-1, 1, 1)
        kz = t(b["kz"]) / c.dz ** 2
        self.kl, self.ku = kz[:-1].clone().view(-1, 1, 1), kz[1:].clone().view(-1, 1, 1)
        self.kl[0], self.ku[-1] = 0, 0
        self.Es = t(b["emis_b"]) * torch.exp(x.view(c.nblocks, c.ny, c.nx)) / c.dz
        self.rinv = 1.0 / t(b["obs_sigma"]) ** 2
        self.y, self.x = t(b["obs_y"]), x
        st, pos = b["obs_step"], b["obs_pos"]
        i0 = np.floor(pos[:, 0]).astype(np.int64)
        j0 = np.minimum(np.floor(pos[:, 1]).astype(np.int64), c.ny - 2)
        l0 = np.minimum(np.floor(pos[:, 2]).astype(np.int64), c.nz - 2)
        f = pos - np.stack([i0, j0, l0], 1)
        cell, wt = [], []
        for q in range(8):
            di, dj, dl = q & 1, (q >> 1) & 1, q >> 2
            cell.append(((l0 + dl) * c.ny + j0 + dj) * c.nx + (i0 + di) % c.nx)
            wt.append(np.prod([f[:, a] if o else 1 - f[:, a] for a, o in enumerate((di, dj, dl))], axis=0))
        self.cell, self.wt = torch.tensor(np.stack(cell), device=DEV), t(np.stack(wt))
        self.at = {int(s): torch.tensor(np.nonzero(st == s)[0], device=DEV) for s in np.unique(st)}

        def root(m, d, wrap):
            a = torch.arange(m, device=DEV)
            a = (a[:, None] - a).abs()
            w, V = torch.linalg.eigh(torch.exp(-(torch.minimum(a, m - a) if wrap else a).to(F64) * d / c.ell))
            return V * w.clamp(min=0).sqrt() @ V.mT

        self.Sx, self.Sy = root(c.nx, c.dx, True), root(c.ny, c.dy, False)

    def prior(self, W):
        f = W.reshape(W.shape[:-1] + (self.c.nblocks, self.c.ny, self.c.nx))
        return (self.c.sigma_b * (self.Sy @ (f @ self.Sx))).reshape(W.shape)

    def tend(self, w, cf):
        a = self.c0 * w
        for coef, shift, dim in zip(cf, (-1, 1, -1, 1), (-1, -1, -2, -2)):
            a += coef * torch.roll(w, shift, dim)
        a *= self.amp
        flux = w[..., 1:, :, :] - w[..., :-1, :, :]
        a[..., :-1, :, :] += self.ku[:-1] * flux
        a[..., 1:, :, :] -= self.kl[1:] * flux
        return a

    def rk4(self, w, cf, src=None):
        def f(z):
            k = self.tend(z, cf)
            if src is not None:
                k[..., 0, :, :] += src
            return k
        h = self.c.dt
        k1 = f(w)
        u1 = w + 0.5 * h * k1
        k2 = f(u1)
        u2 = w + 0.5 * h * k2
        k3 = f(u2)
        u3 = w + h * k3
        k4 = f(u3)
        return w + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4), h / 6 * (w + 2 * u1 + 2 * u2 + u3)[..., 0, :, :]

    def forward(self, src):   # src (cols, nb, ny, nx) -> H c (cols, p)
        c = self.c
        z = torch.zeros(src.shape[0], c.nz, c.ny, c.nx, dtype=F64, device=DEV)
        out = torch.zeros(src.shape[0], self.p, dtype=F64, device=DEV)
        for t in range(c.T):
            z = self.rk4(z, self.tl, src[:, t * c.nblocks // c.T])[0]
            if t + 1 in self.at:
                o = self.at[t + 1]
                out[:, o] = (self.wt[:, o] * z.flatten(1)[:, self.cell[:, o]]).sum(1)
        return out

    def backward(self, r):    # r (cols, p) -> source adjoint (cols, nb, ny, nx)
        c = self.c
        z = torch.zeros(r.shape[0], c.nz, c.ny, c.nx, dtype=F64, device=DEV)
        e = torch.zeros(r.shape[0], c.nblocks, c.ny, c.nx, dtype=F64, device=DEV)
        for t in range(c.T - 1, -1, -1):
            if t + 1 in self.at:
                o = self.at[t + 1]
                for q in range(8):
                    z.flatten(1).index_add_(1, self.cell[q, o], self.wt[q, o] * r[:, o])
            z, s = self.rk4(z, self.ad)
            e[:, t * c.nblocks // c.T] += s
        return e

    def product(self, W):
        src = self.prior(W).view(-1, *self.Es.shape) * self.Es
        e = self.backward(self.rinv * self.forward(src)) * self.Es
        return self.prior(e.reshape(W.shape))


def exact(case, seed):
    torch.cuda.set_device(0)
    kind = case["kind"]
    if kind in ("hvp", "outer", "loop"):
        m = _L96(case, seed)
        if kind == "hvp":
            return m.product(_normal(seed, 7, case["ncols"], case["n"], dtype=F32).to(F64))
        if kind == "outer":
            return {"J": float(0.5 * (m.d @ m.d)), "traj": torch.stack(m.traj), "d": m.d, "g": m.gradient()}
        lam, dv = _loop_exact(m, _normal(seed, 7, case["k"], case["n"], dtype=F32), case["k"], case["q"])
        return {"lam": lam.cpu().numpy(), "dv": dv}
    if kind == "batch":
        return None   # the sketch is the library's own stream
    if kind == "tracer":
        return _Tracer(case, seed).product(_normal(seed, 7, case["ncols"], _box_n(case), dtype=F32).to(F64))
    if kind == "emission":
        m = _Tracer(case, seed)
        d = m.forward(m.Es[None])[0] - m.y
        g = m.prior((m.backward((m.rinv * d)[None])[0] * m.Es).reshape(-1))
        return {"J": float(0.5 * (d * d * m.rinv).sum()), "d": d, "g": g}
    chan, K, p, x, U = _net(case, seed)
    p = p.to(F64).requires_grad_(True)
    a, at = x.to(F64), 0
    for l, (ci, co) in enumerate(zip(chan, chan[1:])):
        w, at = p[at:at + co * ci * K].view(co, ci * K), at + co * ci * K
        bias, at = p[at:at + co].view(1, co, 1), at + co
        cols = torch.stack([torch.roll(a, K // 2 - d, -1) for d in range(K)], 2).flatten(1, 2)
        a = w @ cols + bias
        if l < len(chan) - 2:
            a = torch.tanh(a)
    Ud, m = U.to(F64), case["m"]
    rest = a - (a @ Ud.mT) @ Ud
    sq = a.square().sum((1, 2))
    S = a @ a.mT / (sq / m).view(-1, 1, 1) - torch.eye(m, dtype=F64, device=DEV)
    loss = (rest.square().sum((1, 2)) / sq + 0.1 * S.square().sum((1, 2)) / m ** 2).mean()
    return {"loss": float(loss), "grad": torch.autograd.grad(loss, p)[0].detach()}


def _box_n(case):
    return case["nb"] * case["ny"] * case["nx"]
