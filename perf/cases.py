"""Performance cases of the library: the calls a solver built on it makes, over the sizes it is used at.

    listed()             the named cases
    draw(rng)            one more case of the same ranges
    prepare(case, seed)  the inputs (load profile, point or batch) and the handle a program keeps
    run(state)           one pass through the public entry points (paper_2310_06650_gb300.qg)
    work(case)           bytes and operations one pass cannot do without
    exact(case, seed)    what run returns, in 64 bits, with plain torch

Grids come from synth (the shapes of the tests and of bench.py); a load profile and a point of an
Adam run are drawn from the seed.  A network is made once per process, as a program would.
"""
from __future__ import annotations

import dataclasses
import functools
import math

import numpy as np
import torch

import synth
import synth.grids
from paper_2310_06650_gb300 import qg

DEV = "cuda"
LR, TRAIN_LR, B1, B2, ADAM_EPS = 1e-3, 1e-4, 0.9, 0.999, 1e-8
# the largest draws: elements of the contingency block of the day-ahead grid, buses of a drawn grid
MAX_TMK = 48 * 35000 * 2000
MAX_N = 12000


def listed():
    q = dict(kind="grid")
    m = dict(kind="mlp", n_in=11106, hidden=1024, n_out=27072)  # the warm start of the 617-bus case
    return [
        # the smallest grid with the default options: launches and latency
        dict(q, name="tiny_eval_f64", net="tiny14", prec="f64", do="eval"),
        # every device model (transformers, bid blocks, consumers, on-status), as in batch rounding:
        # a short FP64 Adam run between two rounds
        dict(q, name="mid_devices_solve_f64", net="mid150", prec="f64", do="solve", iters=20, devices="all"),
        # the real-time case: one evaluation (objective and gradient) in mixed precision
        dict(q, name="rt_eval_mixed", net="rt617", prec="mixed", do="eval"),
        # the real-time case: a stretch of the Adam run, the library's main loop
        dict(q, name="rt_solve_mixed", net="rt617", prec="mixed", do="solve", iters=16),
        # the real-time case driven from outside in FP64: evaluation, then the caller's own Adam state
        dict(q, name="rt_step_f64", net="rt617", prec="f64", do="step"),
        # the real-time case from page-locked host buffers, end to end
        dict(q, name="rt_host_mixed", net="rt617", prec="mixed", do="host"),
        # one instance of the largest shape of the batch: 48 periods, dense DC products
        dict(q, name="b1576_eval_mixed", net="b1576", prec="mixed", do="eval"),
        # 32 uneven instances in one handle on the step-size, smoothing and homotopy schedules
        dict(q, name="batch32_sched_mixed", net="batch32", prec="mixed", do="sched", iters=8),
        # the day-ahead grid (sparse DC solver): mixed precision, and FP64 as points are scored
        dict(q, name="da_eval_mixed", net="da23643", prec="mixed", do="eval"),
        dict(q, name="da_eval_f64", net="da23643", prec="f64", do="eval"),
        # the warm-start network: a prediction for a full batch, and a few training steps
        dict(m, name="mlp_forward", batch=64, do="forward"),
        dict(m, name="mlp_train", batch=64, do="train", steps=4),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if rng.random() < 0.25:
        do = rng.choice(["forward", "train"])
        c = dict(kind="mlp", do=do, n_in=logint(40, 11106), hidden=logint(32, 1024), n_out=logint(100, 27072),
                 batch=rng.choice([1, 2, 7, 16, 33, 64]))
        if do == "train":
            c["steps"] = rng.choice([1, 2, 4])
        return c
    c = dict(kind="grid", net="drawn", prec=rng.choice(["mixed", "mixed", "f64"]))
    c["do"] = rng.choice(["eval", "eval", "solve", "sched", "step", "host"])
    n = logint(14, MAX_N)
    T = logint(1, 48)
    M = int(round(rng.uniform(1.45, 1.6) * n)) + 2
    K = max(1, min(2000, int(rng.uniform(0.05, 0.65) * M), MAX_TMK // (T * M)))
    c.update(n=n, T=T, M=M, G=max(2, int(0.146 * n)), K=K, Z=rng.choice([1, 1, 3, 8]) if n > 100 else 1,
             net_seed=rng.randrange(1 << 20))
    if c["do"] in ("solve", "sched"):
        c["iters"] = rng.choice([1, 5, 8, 16]) if n < 2000 else rng.choice([1, 2, 3])
    if n <= 1200 and rng.random() < 0.3:
        c["devices"] = rng.choice(["xf", "bids", "uc", "all"])
    if K >= 20 and rng.random() < 0.2:
        c["frac"] = rng.choice([0.2, 0.5])  # contingency screening: a subset of the outages per evaluation
    if c["prec"] == "mixed" and rng.random() < 0.15:
        c["lodf"] = "bf16x2"  # the compact line-outage block
    return c


# ------------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=4)
def _networks(key):
    """The grids of a case (a list), at their nominal loads."""
    c = dict(key)
    net = c["net"]
    if net == "batch32":
        return synth.batch()
    if net == "b1576":
        g = synth.make_case("b1576_48_1024", 1576, 2301, 230, T=48, K=231, seed=1024, rating_scale=0.8)
    elif net == "drawn":
        g = synth.make_case("drawn", c["n"], c["M"], c["G"], T=c["T"], K=c["K"], n_zone=c["Z"], seed=c["net_seed"])
    else:
        g = {"tiny14": synth.tiny, "mid150": synth.mid, "rt617": synth.rt617, "da23643": synth.dayahead}[net]()
    d = c.get("devices", "")
    if d in ("xf", "all"):
        g = synth.with_transformers(g, 0.15, 1)
    if d in ("bids", "all"):
        g = synth.with_block_bids(g, 3, 0.3, 2)
    if d in ("uc", "all"):
        g = synth.with_commitment(g, 3)
    if net == "drawn":  # rated like the named cases: twice the largest merit-order flow, at least 0.5
        dc = _dc(g)
        f = _flows(g, dc, torch.tensor(_dispatch(g), device=DEV), None)
        rate = torch.clamp(2.0 * f.abs().amax(0), min=0.5).cpu().numpy()
        g = dataclasses.replace(g, s_max=rate, s_max_ctg=rate.copy())
    return [g]


def _grids(case, seed):
    key = tuple(sorted((k, v) for k, v in case.items()
                       if k in ("net", "n", "T", "M", "G", "K", "Z", "net_seed", "devices")))
    return [synth.with_loads(g, synth.load_profiles(g, 1, seed + 7919 * b)[0]) for b, g in enumerate(_networks(key))]


def _cons(g):
    return np.asarray(g.dev_cons, bool) if len(g.dev_cons) else np.zeros(g.n_gen, bool)


def _dispatch(g):
    """Merit-order dispatch of the producers, consumers at their nominal draw."""
    cons = _cons(g)
    p = np.zeros((g.T, g.n_gen))
    p[:, cons] = g.pmax[cons] / 1.2
    need = g.load_p.sum(1) + p.sum(1)
    order = np.flatnonzero(~cons)[np.argsort(g.cost_b[~cons], kind="stable")]
    before = np.concatenate([[0.0], np.cumsum(g.pmax[order])[:-1]])
    p[:, order] = np.clip(need[:, None] - before[None, :], 0.0, g.pmax[order][None, :])
    return p


def _point(g, seed):
    """A point of an Adam run: the merit-order start after its variables have moved a little."""
    rng = np.random.default_rng(seed)
    T, n, G, X = g.T, g.n_bus, g.n_gen, g.n_xf
    v = np.clip(1.0 + 0.01 * rng.standard_normal((T, n)), g.vmin, g.vmax)
    th = 0.01 * rng.standard_normal((T, n))
    th[:, g.ref_bus] = 0.0
    p = np.clip(_dispatch(g) + 0.02 * g.pmax * rng.standard_normal((T, G)), g.pmin, g.pmax)
    q = np.clip(0.1 * g.qmax * rng.standard_normal((T, G)), np.minimum(g.qmin, 0), np.maximum(g.qmax, 0))
    share = g.reserve_req.sum(1, keepdims=True) / np.maximum((g.pmax - p).sum(1, keepdims=True), 1e-9)
    r = np.where(_cons(g), 0.0, np.maximum(g.pmax - p, 0.0) * np.minimum(share, 1.0) * rng.uniform(0.9, 1.1, (T, G)))
    parts = [v, th, p, q, r]
    if X:
        parts += [np.clip(1.0 + 0.02 * rng.standard_normal((T, X)), g.tau_min, g.tau_max),
                  rng.uniform(0.2 * g.phi_min, 0.2 * g.phi_max, (T, X))]
    if g.commit:
        parts.append(rng.uniform(0.7, 1.0, (T, G)))
    return np.concatenate([a.ravel() for a in parts])


def _table(iters):
    """Step size, smoothing and homotopy scale per iteration (Sec. II-F)."""
    t = np.linspace(-1.0, 1.0, iters) if iters > 1 else np.array([-1.0])
    mag = lambda s: np.exp(4 * s) / (0.6 + np.exp(4 * s))  # noqa: E731
    return np.stack([1e-2 * 10.0 ** (mag(t) * -3.0), 5e-2 * 10.0 ** (mag(t - 0.25) * -3.0),
                     0.1 + 0.45 * (t + 1.0)], axis=1)


def _mlp_inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    I, H, O, B = case["n_in"], case["hidden"], case["n_out"], case["batch"]
    N = B * case.get("steps", 1)
    rn = lambda *s: torch.randn(*s, device=DEV, generator=gen)  # noqa: E731
    w = torch.cat([(rn(H, I) * math.sqrt(2 / I)).ravel(), 0.01 * rn(H), (rn(H, H) * math.sqrt(2 / H)).ravel(),
                   0.01 * rn(H), (rn(O, H) * math.sqrt(1 / H)).ravel(), 0.01 * rn(O)])
    x = 0.8 * torch.rand(N, 1, device=DEV, generator=gen) - 0.4 + 0.2 * rn(N, I)  # relative load deviations
    return w, x.contiguous(), 0.5 * rn(N, O)


# ------------------------------------------------------------------------------------------------
# the calls
# ------------------------------------------------------------------------------------------------

class _Mlp:
    def __init__(self, case):
        self.h = qg.qg_mlp_create(case["n_in"], case["hidden"], case["n_out"], case["batch"])
        qg.qg_mlp_set_stream(self.h, torch.cuda.current_stream().cuda_stream)

    def __del__(self):
        torch.cuda.synchronize()
        qg.qg_mlp_destroy(self.h)


def prepare(case, seed):
    s = dict(case)
    if case["kind"] == "mlp":
        w, x, target = _mlp_inputs(case, seed)
        net = _Mlp(case)
        qg.qg_mlp_set_params(net.h, w)
        s.update(net=net, x=x, target=target, y=torch.empty(case["batch"], case["n_out"], device=DEV),
                 loss=torch.zeros(case.get("steps", 1), dtype=torch.float64, device=DEV))
        if case["do"] == "train":
            s.update(w=torch.empty_like(w), g=torch.empty_like(w))
        torch.cuda.synchronize()
        return s
    grids = _grids(case, seed)
    lodf = qg.QG_LODF_BF16X2 if case.get("lodf") == "bf16x2" else qg.QG_LODF_F32
    sol = qg.Solver(grids, precision=qg.QG_FP64 if case["prec"] == "f64" else qg.QG_MIXED, lodf_dtype=lodf,
                    ctg_frac=case.get("frac", 0.0))
    x0 = np.concatenate([_point(g, seed + 104729 * b) for b, g in enumerate(grids)])
    if case["prec"] == "mixed":  # values that the mixed path holds exactly
        x0 = x0.astype(np.float32).astype(np.float64)
    s.update(sol=sol, x=torch.tensor(x0, dtype=sol.dtype, device=DEV))
    if case["do"] == "host":
        pin = lambda a: torch.tensor(a, dtype=torch.float64).pin_memory()  # noqa: E731
        s["pinned"] = [pin(x0), pin(np.zeros(len(grids))), pin(np.zeros(len(x0)))]
        s["host"] = [t.numpy() for t in s["pinned"]]
    elif case["do"] == "step":
        s.update(m=torch.zeros_like(s["x"]), v=torch.zeros_like(s["x"]))
    elif case["do"] == "sched":
        s["table"] = torch.tensor(_table(case["iters"]), device=DEV)
    return s


def run(s):
    if s["kind"] == "mlp":
        h, B = s["net"].h, s["batch"]
        if s["do"] == "forward":
            qg.qg_mlp_forward(h, s["x"], B, s["y"])
            return s["y"]
        for k in range(s["steps"]):
            qg.qg_mlp_train_step(h, s["x"][k * B:], s["target"][k * B:], B, TRAIN_LR, B1, B2, s["loss"][k:])
        qg.qg_mlp_get_params(h, s["w"])
        qg.qg_mlp_get_grads(h, s["g"])
        return {"loss": s["loss"], "w": s["w"], "g": s["g"]}
    sol, x = s["sol"], s["x"]
    if s["do"] == "eval":
        qg.qg_eval_grad(sol.h, x, sol.obj, sol.g)
        return {"obj": sol.obj, "g": sol.g}
    if s["do"] == "step":
        qg.qg_eval_grad(sol.h, x, sol.obj)
        qg.qg_adam_step(sol.h, x, s["m"], s["v"], LR, B1, B2)
        return {"obj": sol.obj, "x": x, "m": s["m"], "v": s["v"]}
    if s["do"] == "host":
        xh, oh, gh = s["host"]
        qg.qg_eval_grad_host(sol.h, xh, oh, gh)
        return {"obj": oh, "g": gh}
    if s["do"] == "solve":
        qg.qg_solve(sol.h, x, s["iters"], LR, B1, B2)
    else:
        qg.qg_solve_schedule(sol.h, x, s["iters"], s["table"], True, B1, B2)
    return {"x": x}


def work(case):
    if case["kind"] == "mlp":
        B, I, H, O = (case[k] for k in ("batch", "n_in", "hidden", "n_out"))
        nw = H * I + H * H + O * H
        act = 4.0 * B * (I + O)
        if case["do"] == "forward":  # the BF16 weights once, the input and the output
            return {"bytes": 2.0 * nw + act, "flops": 2.0 * B * nw}
        # a step: the BF16 weights forward, again backward (not the first layer's), master weights and
        # two moments read and written, the gradient and the BF16 copy written
        step = 2.0 * nw + 2.0 * (H * H + O * H) + 24.0 * nw + 4.0 * nw + 2.0 * nw + act + 4.0 * B * O
        return {"bytes": case["steps"] * step + 16.0 * nw, "flops": case["steps"] * 6.0 * B * nw}
    shapes = {"tiny14": [(14, 20, 5, 4, 20)], "mid150": [(150, 219, 22, 5, 40)], "rt617": [(617, 900, 90, 18, 562)],
              "b1576": [(1576, 2301, 230, 48, 231)], "da23643": [(23643, 35000, 3000, 48, 2000)],
              "batch32": [(n, round(1.46 * n), round(0.146 * n), T, math.ceil(0.146 * n))
                          for n, T in synth.grids.BATCH_SHAPES] * 8}.get(case["net"])
    if shapes is None:
        shapes = [tuple(case[k] for k in ("n", "M", "G", "T", "K"))]
    w = 8 if case["prec"] == "f64" else 4
    nbytes = flops = 0.0
    for n, M, G, T, K in shapes:
        K = math.ceil(case["frac"] * K) if case.get("frac") else K
        n_x = T * (2 * n + 3 * G)
        # x in, the gradient out (Adam: x, m, v in and out), loads, network, the line-outage block (an
        # FP32 block settles nearly every element), the DC solves' operator once
        dc = M * G if n <= 4096 else (0.13 * n) ** 2 + 20 * n
        nbytes += w * n_x * (6 if case["do"] in ("solve", "sched", "step") else 2) + 2 * w * T * n + 7 * w * M
        nbytes += 4.0 * M * K + 8.0 * dc
        # two multiply-adds per (period, branch, outage), two DC products, some 300 operations per
        # branch and period
        flops += 4.0 * T * M * K + 4.0 * T * dc + 300.0 * T * M
    it = case.get("iters", 1)
    return {"bytes": it * nbytes, "flops": it * flops}


# ------------------------------------------------------------------------------------------------
# 64-bit values, with plain torch
# ------------------------------------------------------------------------------------------------

def _t(a):
    return torch.tensor(np.asarray(a), device=DEV)


def _dc(g):
    """Factor of the reduced DC Laplacian and what the flows need."""
    n, M = g.n_bus, g.n_branch
    f, o = _t(g.br_from).long(), _t(g.br_to).long()
    y = _t(g.br_x / (g.br_r ** 2 + g.br_x ** 2))
    Y = torch.zeros(n * n, dtype=torch.float64, device=DEV)
    for a, b, s in ((f, f, 1.0), (o, o, 1.0), (f, o, -1.0), (o, f, -1.0)):
        Y.index_add_(0, a * n + b, s * y)
    Y = Y.view(n, n)
    ref = g.ref_bus
    Y[ref, :] = 0.0
    Y[:, ref] = 0.0
    Y[ref, ref] = 1.0
    C = torch.linalg.cholesky(Y)
    return dict(f=f, o=o, y=y, C=C, n=n, M=M, ref=ref)


def _angles(dc, rhs):
    """Columns of angles for columns of injections, 0 at the reference bus."""
    keep = torch.ones(dc["n"], 1, dtype=torch.float64, device=DEV)
    keep[dc["ref"]] = 0.0
    return torch.cholesky_solve(rhs * keep, dc["C"])


def _flows(g, dc, p, b):
    """Base DC flows (T x M) with the uniform slack; b: the phase shifters' own flows (T x M) or None."""
    sg = _t(np.where(_cons(g), -1.0, 1.0))
    inj = (-_t(g.load_p)).index_add(1, _t(g.gen_bus).long(), sg * p)
    inj = inj - inj.mean(1, keepdim=True)
    if b is not None:
        inj = inj.index_add(1, dc["f"], -b).index_add(1, dc["o"], b)
    th = _angles(dc, inj.T)
    f = (dc["y"][:, None] * (th[dc["f"]] - th[dc["o"]])).T
    return f if b is None else f + b


def _lodf(dc, ctg):
    K = len(ctg)
    rhs = torch.zeros(dc["n"], K, dtype=torch.float64, device=DEV)
    k = torch.arange(K, device=DEV)
    rhs[dc["f"][ctg], k] += 1.0
    rhs[dc["o"][ctg], k] -= 1.0
    u = _angles(dc, rhs)
    L = dc["y"][:, None] * (u[dc["f"]] - u[dc["o"]])
    L = L / (1.0 - L[ctg, k])
    L[ctg, k] = float("nan")  # an outaged branch is not monitored
    return L


class _Exact:
    """Objective and gradient of one instance: the AC, device and reserve terms through autograd, the
    contingency term period by period."""

    def __init__(self, g, frac=0.0):
        self.g, self.dc = g, _dc(g)
        K = math.ceil(frac * g.K) if frac else g.K
        self.ctg = _t(g.ctg[:max(1, K)]).long()
        self.L = _lodf(self.dc, self.ctg)

    def ctg_term(self, f, q2, eps, beta):
        g, s_ctg = self.g, _t(self.g.s_max_ctg)
        z = 0.0
        gf, gq = torch.zeros_like(f), torch.zeros_like(q2)
        step = max(1, (1 << 27) // max(1, g.n_branch))
        for t in range(g.T):
            w = float(g.dt[t]) * g.c_s * beta
            for k0 in range(0, len(self.ctg), step):
                ks = self.ctg[k0:k0 + step]
                L = self.L[:, k0:k0 + step]
                F = f[t][:, None] + L * f[t][ks][None, :]
                s2 = F * F + q2[t][:, None]
                over = s2 > (s_ctg * s_ctg)[:, None]  # false at NaN
                z += w * eps * (F.numel() - len(ks))
                m, k = torch.nonzero(over, as_tuple=True)
                F, s = F[m, k], s2[m, k].sqrt()
                u = s - s_ctg[m]
                val = (u * u + eps * eps).sqrt()
                z += w * (float(val.sum()) - eps * len(m))
                d = w * (u / val) / s
                gf[t].index_add_(0, m, d * F)
                gf[t].index_add_(0, ks[k], d * F * L[m, k])
                gq[t].index_add_(0, m, 0.5 * d)
        return z, gf, gq

    def __call__(self, x, eps=None, beta=None):
        g, dc = self.g, self.dc
        eps = g.eps if eps is None else eps
        beta = g.beta if beta is None else beta
        x = x.detach().clone().requires_grad_(True)
        T, n, G, X = g.T, g.n_bus, g.n_gen, g.n_xf
        sizes = [T * n, T * n] + [T * G] * 3 + ([T * X] * 2 if X else []) + ([T * G] if g.commit else [])
        part = [a.view(T, -1) for a in torch.split(x, sizes)]
        v, th, p, q, r = part[:5]
        u = part[-1] if g.commit else torch.ones_like(p)
        dt = _t(g.dt)[:, None]
        relu = lambda a: (torch.relu(a) ** 2 + eps * eps).sqrt()  # noqa: E731
        soft = lambda a: (a * a + eps * eps).sqrt()  # noqa: E731
        cons = _cons(g)
        sg = _t(np.where(cons, -1.0, 1.0))
        # devices
        en = _t(g.cost_a) * p * p + _t(g.cost_b) * p
        if g.blk_width.size:
            W, C = _t(g.blk_width), _t(g.blk_price)
            lo = torch.cat([torch.zeros_like(W[:, :1]), torch.cumsum(W, 1)[:, :-1]], 1)  # where each block starts
            e = p[:, :, None] - lo
            blk = (C * torch.where(e < 0, torch.zeros_like(e), torch.where(e < W, e, W.expand_as(e)))).sum(2)
            en = torch.where(W.sum(1) > 0, blk, en)
        z = (dt * (sg * en + _t(g.cost_r) * r)).sum()
        wr = g.rho * beta
        z = z + wr * relu(p + r - _t(g.pmax) * u).sum()
        if g.commit:
            du = u - torch.cat([_t(g.u_init)[None], u[:-1]])
            z = z + (dt * _t(g.c_on) * u + _t(g.c_su) * torch.relu(du) + _t(g.c_sd) * torch.relu(-du)).sum()
            z = z + wr * (relu(_t(g.pmin) * u - p) + relu(q - _t(g.qmax) * u) + relu(_t(g.qmin) * u - q)).sum()
        if T > 1:
            lim = _t(g.ramp) * dt[1:]
            z = z + wr * (relu(p[1:] - p[:-1] - lim) + relu(p[:-1] - p[1:] - lim)).sum()
        rz = torch.zeros(T, g.n_zone, dtype=torch.float64, device=DEV).index_add(1, _t(g.gen_zone).long(), r)
        z = z + (dt * g.c_rz * beta * relu(_t(g.reserve_req) - rz)).sum()
        # AC flows (pi model, tap and shift at the from end)
        den = g.br_r ** 2 + g.br_x ** 2
        gs, bs, hc = _t(g.br_r / den), _t(-g.br_x / den), _t(g.br_b / 2)
        tau, phi = torch.ones(T, g.n_branch, dtype=torch.float64, device=DEV), 0.0
        if X:
            xf = _t(g.xf_branch).long()
            tau = tau.index_copy(1, xf, part[5])
            phi = torch.zeros_like(tau).index_copy(1, xf, part[6])
        f, o = dc["f"], dc["o"]
        vf, vo = v[:, f] / tau, v[:, o]
        d = th[:, f] - th[:, o] - phi
        c, s, vv = torch.cos(d), torch.sin(d), vf * vo
        pf = gs * vf * vf + (-gs * c - bs * s) * vv
        qf = -(bs + hc) * vf * vf + (bs * c - gs * s) * vv
        pt = gs * vo * vo + (-gs * c + bs * s) * vv
        qt = -(bs + hc) * vo * vo + (bs * c + gs * s) * vv
        gb = _t(g.gen_bus).long()
        P = _t(g.load_p).index_add(1, f, pf).index_add(1, o, pt).index_add(1, gb, -sg * p)
        Q = _t(g.load_q).index_add(1, f, qf).index_add(1, o, qt).index_add(1, gb, -sg * q)
        z = z + (dt * beta * (g.c_p * soft(P) + g.c_q * soft(Q))).sum()
        sf2, st2 = pf * pf + qf * qf, pt * pt + qt * qt
        z = z + (dt * g.c_s * beta * relu(torch.where(sf2 >= st2, sf2, st2).sqrt() - _t(g.s_max))).sum()
        # contingencies: their value, and a linear form with their gradient
        fl = _flows(g, dc, p, bs * phi if X else None)
        q2 = torch.where(qf * qf >= qt * qt, qf * qf, qt * qt)
        with torch.no_grad():
            zc, gf, gq = self.ctg_term(fl, q2, eps, beta)
        (z + (gf * fl).sum() + (gq * q2).sum()).backward()
        return float(z.detach()) + zc, x.grad

    def box(self):
        g = self.g
        T, n, G = g.T, g.n_bus, g.n_gen
        rows = lambda a: np.tile(a, (T, 1)).ravel()  # noqa: E731
        inf = np.full((T, n), np.inf)
        inf[:, g.ref_bus] = 0.0
        zero = np.zeros(G)
        lo = [rows(g.vmin), -inf.ravel(), rows(zero if g.commit else g.pmin),
              rows(np.minimum(g.qmin, 0) if g.commit else g.qmin), rows(zero)]
        hi = [rows(g.vmax), inf.ravel(), rows(g.pmax), rows(np.maximum(g.qmax, 0) if g.commit else g.qmax),
              rows(np.where(_cons(g), 0.0, g.pmax))]
        if g.n_xf:
            lo += [rows(g.tau_min), rows(g.phi_min)]
            hi += [rows(g.tau_max), rows(g.phi_max)]
        if g.commit:
            lo.append(rows(zero))
            hi.append(rows(np.ones(G)))
        return _t(np.concatenate(lo)), _t(np.concatenate(hi))


def _adam(x, m, v, grad, i, lr, lo=None, hi=None, eps=ADAM_EPS):
    m = B1 * m + (1 - B1) * grad
    v = B2 * v + (1 - B2) * grad * grad
    x = x - lr * (m / (1 - B1 ** i)) / ((v / (1 - B2 ** i)).sqrt() + eps)
    return (x if lo is None else torch.minimum(torch.maximum(x, lo), hi)), m, v


def _exact_mlp(case, seed):
    w, xs, ts = _mlp_inputs(case, seed)
    I, H, O, B = case["n_in"], case["hidden"], case["n_out"], case["batch"]
    sizes = [H * I, H, H * H, H, O * H, O]
    w, xs, ts = w.double(), xs.double(), ts.double()

    def net(w, x):
        W1, b1, W2, b2, W3, b3 = torch.split(w, sizes)
        h = torch.relu(x @ W1.view(H, I).T + b1)
        h = torch.relu(h @ W2.view(H, H).T + b2)
        return h @ W3.view(O, H).T + b3

    if case["do"] == "forward":
        return net(w, xs)
    m = v = torch.zeros_like(w)
    loss = []
    for k in range(case["steps"]):
        w = w.detach().requires_grad_(True)
        e = ((net(w, xs[k * B:(k + 1) * B]) - ts[k * B:(k + 1) * B]) ** 2).mean()
        grad, = torch.autograd.grad(e, w)
        loss.append(float(e))
        w, m, v = _adam(w.detach(), m, v, grad, k + 1, TRAIN_LR)
    return {"loss": np.array(loss), "w": w, "g": grad}


def exact(case, seed):
    if case["kind"] == "mlp":
        return _exact_mlp(case, seed)
    it = case["iters"] if case["do"] in ("solve", "sched") else 1
    grids = _grids(case, seed)
    if it * sum(g.T * g.n_branch * g.K for g in grids) > 4 * MAX_TMK:
        return None
    store = torch.float64 if case["prec"] == "f64" else torch.float32
    out = []
    for b, g in enumerate(grids):
        x = torch.tensor(_point(g, seed + 104729 * b), dtype=store, device=DEV).double()
        ev = _Exact(g, case.get("frac", 0.0))
        if case["do"] in ("eval", "host"):
            obj, grad = ev(x)
            out.append((obj, grad))
            continue
        lo, hi = ev.box()
        m = v = torch.zeros_like(x)
        rows = _table(it) if case["do"] == "sched" else [(LR, None, None)] * it
        for i, (lr, eps, beta) in enumerate(rows):
            obj, grad = ev(x, eps, beta)
            x, m, v = _adam(x, m, v, grad, i + 1, lr, lo, hi)
        out.append((obj, x, m, v))
        del ev
    cat = lambda j: torch.cat([o[j] for o in out])  # noqa: E731
    objs = np.array([o[0] for o in out])
    if case["do"] in ("eval", "host"):
        return {"obj": objs, "g": cat(1)}
    if case["do"] == "step":
        return {"obj": objs, "x": cat(1), "m": cat(2), "v": cat(3)}
    return {"x": cat(1)}
