"""Performance cases of the candidate-scoring library, through its Python entry points.

A case is a plain dict; ``kind`` says which call it stands for:

  step    one optimisation iteration through an engine (GP fit, posterior,
          acquisition, selection), with the per-candidate scores read back and
          the chosen candidates marked in the caller's pool
  gp      the surrogate alone: standardise, fit, posterior at the candidates
  learn   hyperparameters by marginal likelihood (the training direction:
          Adam steps on the analytic gradient, in double precision)
  ascent  the acquisition optimised over the decision space from the best
          candidates (gradients through the posterior)
  topk    the selection alone, on given scores

Inputs follow the synthetic problems of ``workloads.py``: observations on the
unit cube of two or three smooth objectives with noise of variance 1e-4,
lengthscales around 0.2 sqrt(d) (here one per feature, as automatic relevance
determination learns them), a reference point of 1.1 standard deviations,
uniform candidates and standard-normal base samples. ``exact`` restates each
call in 64-bit torch and numpy.
"""
import math

import numpy as np
import torch

from paper_2602_10729_gb300 import boute as bt

F32, F64 = torch.float32, torch.float64
SQRT5, SQRT3 = math.sqrt(5.0), math.sqrt(3.0)
NOISE = 1e-4
REF = 1.1
MODES = {"ehvi": bt.BOUTE_ACQ_EHVI2D, "mc": bt.BOUTE_ACQ_MC_HVI, "nehvi": bt.BOUTE_ACQ_NEHVI}
CODES = (bt.BOUTE_TF_LOG, bt.BOUTE_TF_LOGIT | bt.BOUTE_TF_NEGATE)  # latency, quality
MAX_COUNT = 4  # deployment features of composite problems: GPU counts 0 .. 4
JITTER = 1e-8  # of the in-sample covariance, times the outputscale
INSAMPLE_KEY = 0x6A09E667F3BCC909  # an engine's in-sample normals: seed 0 ^ this key


def _step(name, mode, B, n, d, m, N, k, S=0, comp=False, cons=False, host=False, wait=False):
    c = dict(kind="step", mode=mode, B=B, n=n, d=d, m=m, N=N, k=k, S=S, comp=comp, cons=cons,
             host=host, wait=wait)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the first iterations of a search: few observations, a small pool, and
        # the caller waits for the choice before it evaluates it
        _step("step-tiny", "ehvi", 1, 32, 6, 2, 4096, 8, wait=True),
        # an ordinary iteration: Monte-Carlo improvement over two objectives
        _step("step-mc2", "mc", 1, 128, 12, 2, 65536, 32, S=128),
        # the same with noisy observations: joint in-sample draws
        _step("step-noisy", "nehvi", 1, 128, 12, 2, 65536, 32, S=128),
        # a long search over a large pool, closed-form improvement
        _step("step-large", "ehvi", 1, 512, 16, 2, 1 << 20, 64),
        # the largest: three objectives, a thousand observations, 4 Mi candidates
        _step("step-mc3-largest", "mc", 1, 1024, 24, 3, 1 << 22, 128, S=256),
        # many independent problems at once (one per workload or tenant)
        _step("step-batched", "ehvi", 64, 256, 10, 2, 1 << 18, 16),
        # odd sizes, three objectives under constraints, a sample count of no
        # special form
        _step("step-mc3-odd", "mc", 1, 203, 7, 3, 100003, 17, S=100, cons=True),
        # the composite kernel with outcome transforms and constraints, inputs
        # in (pinned) host memory and the choice back in host memory
        _step("step-composite-host", "ehvi", 1, 333, 16, 2, 262147, 64, comp=True, cons=True,
              host=True, wait=True),
        # the surrogate alone for a few problems of odd size
        dict(kind="gp", name="gp-odd", B=3, n=777, d=20, m=2, N=30011),
        # hyperparameters relearned between iterations from three restarts
        dict(kind="learn", name="learn", B=1, n=128, d=12, m=2, R=3, iters=20),
        # the pool's best candidates refined by gradient ascent
        dict(kind="ascent", name="ascent", B=1, n=200, d=16, S=128, P=32, steps=10),
        # the selection alone, ragged
        dict(kind="topk", name="topk", B=4, N=(1 << 20) + 7, k=100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Multiply-adds of a pass, about, with each acquisition sample as 100."""
    if c["kind"] in ("gp", "step"):
        return c["B"] * c["m"] * (c["N"] * (c["n"] * (c["n"] + 4 * c["d"] + 100) +
                                            100 * c.get("S", 0)) + 30 * c["n"] ** 3)
    return 0


def draw(rng):
    kind = rng.choices(("ehvi", "mc2", "mc3", "nehvi", "gp", "learn", "ascent", "topk"),
                       (4, 3, 2, 2, 2, 2, 1, 1))[0]
    if kind == "topk":
        B = _log(rng, 1, 16)
        N = _log(rng, 2000, (1 << 23) // B)
        return dict(kind="topk", B=B, N=N, k=min(N, _log(rng, 1, 256)))
    d = rng.randint(4, 32)
    if kind == "learn":  # a step costs about n^3
        n = min(_log(rng, 20, 200), 40 * d)
        return dict(kind="learn", B=1, n=n, d=d, m=2, R=rng.randint(1, 6),
                    iters=max(2, min(20, int(20 * (128 / n) ** 3))))
    if kind == "ascent":
        n = min(_log(rng, 20, 500), 40 * d)
        return dict(kind="ascent", B=1, n=n, d=d, S=_log(rng, 32, 256), P=_log(rng, 4, 64),
                    steps=rng.randint(3, 12))
    top = _cost(listed()[4])
    while True:
        n = min(_log(rng, 16, 128 if kind == "nehvi" else 1024), 40 * d)
        B = _log(rng, 1, 4 if kind in ("nehvi", "gp") else 64)
        N = _log(rng, 1000, 1 << (18 if kind == "nehvi" else 21))
        m = 3 if kind == "mc3" else 2
        S = 0 if kind in ("ehvi", "gp") else rng.choice((64, 100, 128, 128, 256, 33))
        k = min(N, _log(rng, 1, 256))
        if kind == "gp":
            c = dict(kind="gp", B=B, n=n, d=d, m=m, N=N)
        else:
            c = _step(None, kind.rstrip("23"), B, n, d, m, N, k, S=S,
                      comp=kind in ("ehvi", "mc2") and rng.random() < 0.3,
                      cons=rng.random() < 0.3, host=kind == "ehvi" and rng.random() < 0.3,
                      wait=rng.random() < 0.3)
            c["wait"] = c["wait"] or c["host"]
        if _cost(c) < 0.5 * top and B * N * max(m * S, 1) < 1 << 30 and B * N < 1 << 24:
            return c


# ---- inputs ---------------------------------------------------------------------------
def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) << 5) + stream)


def _rand(g, *shape, dtype=F64):
    return torch.rand(*shape, generator=g, device="cuda", dtype=dtype)


def _objectives(X, m):
    d = X.shape[-1]
    f = [((X - 0.25) ** 2).sum(-1) / d, ((X - 0.75) ** 2).sum(-1) / d]
    if m == 2:
        f[0] = f[0] + 0.1 * torch.sin(2.0 * math.pi * X[..., 0])
    else:
        f.append(1.0 - torch.exp(-((X - 0.5) ** 2).sum(-1) / (0.1 * d)))
    return torch.stack(f, -1)


def _problem(c, seed):
    """Observations, hyperparameters and (composite problems) kernel parameters."""
    B, n, d, m = c["B"], c["n"], c["d"], c.get("m", 2)
    g = _gen(seed, 0)
    X = _rand(g, B, n, d)
    e = 0.01 * torch.randn(B, n, m, generator=g, device="cuda", dtype=F64)
    ls = 0.2 * math.sqrt(d) * (0.8 + 0.5 * _rand(g, B, m, d))
    s2 = 0.7 + 0.6 * _rand(g, B, m)
    p = dict(X=X, Y=_objectives(X, m) + e, ls=ls, s2=s2, kc=None, dtau=d,
             noise=torch.full((B, m), NOISE, device="cuda", dtype=F64),
             ref=torch.full((B, m), REF, device="cuda", dtype=F64))
    if c.get("comp"):  # routing features, then GPU counts; latency and quality
        dt = p["dtau"] = d // 2
        p["X"] = torch.cat([X[..., :dt], torch.floor(X[..., dt:] * (MAX_COUNT + 1))], -1)
        f = _objectives(torch.cat([X[..., :dt], p["X"][..., dt:] / MAX_COUNT], -1), m) + e
        p["Y"] = torch.stack([torch.exp(f[..., 0]), 1.0 / (1.0 + torch.exp(f[..., 1]))], -1)
        ls[..., dt:] *= MAX_COUNT
        fixed = torch.tensor([0.5, 0.1, 0.05], device="cuda", dtype=F64).expand(B, m, 3)
        p["kc"] = torch.cat([fixed, _rand(g, B, m, d - dt)], -1)
    if c.get("cons"):
        p["cons"] = 0.3 + 0.4 * _rand(g, B, m)
    return p


def _candidates(c, seed, dtau):
    x = _rand(_gen(seed, 1), c["B"], c["N"], c["d"], dtype=F32)
    if dtau < c["d"]:
        x[..., dtau:] = torch.floor(x[..., dtau:] * (MAX_COUNT + 1))
    return x


def _normals(c, seed):
    if not c["S"]:
        return None
    return torch.randn(c["B"], c["N"], c["m"], c["S"], generator=_gen(seed, 2), device="cuda")


def _learn_inputs(c, seed):
    p = _problem(c, seed)
    Y = p["Y"]
    Ys = (Y - Y.mean(1, keepdim=True)) / Y.std(1, keepdim=True)
    th = torch.cat([p["ls"].log(), p["s2"].log()[..., None], p["noise"].log()[..., None] + 3.0], -1)
    th = th[:, :, None, :] + 0.6 * (_rand(_gen(seed, 3), c["B"], c["m"], c["R"], c["d"] + 2) - 0.5)
    return p["X"], Ys.contiguous(), th.contiguous()


def _ascent_inputs(c, seed):
    """Starts: from 64 random points each, the one with the smallest sum of objectives."""
    x = _rand(_gen(seed, 4), c["B"], c["P"], 64, c["d"], dtype=F32)
    best = _objectives(x.double(), 2).sum(-1).argmin(-1)
    X0 = torch.gather(x, 2, best[..., None, None].expand(-1, -1, 1, c["d"]))[:, :, 0]
    eps = torch.randn(2, c["S"], generator=_gen(seed, 5), device="cuda")
    return X0.contiguous(), eps


def _scores(c, seed):
    """Scores as an acquisition gives them: positive and skewed, a fifth exactly zero."""
    g = _gen(seed, 6)
    z = torch.randn(c["B"], c["N"], generator=g, device="cuda")
    return torch.where(z < -0.84, torch.zeros_like(z), torch.exp(2.0 * z))


# ---- what a program holds, and one pass -------------------------------------------------
_streams = []


def _stream():
    """The program's stream (a step is replayed as a graph on any but the default one)."""
    if not _streams:
        _streams.append(torch.cuda.Stream())
    return _streams[0]


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = dict(c=c, stream=_stream())
    dev = lambda *shape, dtype=F32: torch.empty(*shape, dtype=dtype, device="cuda")  # noqa: E731
    if kind == "topk":
        s.update(acq=_scores(c, seed), idx=dev(c["B"], c["k"], dtype=torch.int64),
                 val=dev(c["B"], c["k"]))
        torch.cuda.synchronize()
        return s
    if kind == "learn":
        X, Ys, th = _learn_inputs(c, seed)
        s.update(X=X, Ys=Ys, theta0=th, theta=torch.empty_like(th), grad=torch.empty_like(th),
                 mll=dev(c["B"], c["m"], c["R"], dtype=F64))
        torch.cuda.synchronize()
        return s
    B, n, d, m = c["B"], c["n"], c["d"], c.get("m", 2)
    p = _problem(c, seed)
    if kind == "step":
        N, k = c["N"], c["k"]
        e = bt.boute_engine_create(B, n, d, m, N, MODES[c["mode"]], c["S"], k)
        if c["comp"]:
            bt.boute_engine_set_kernel(e, p["dtau"], p["kc"].cpu().numpy())
            bt.boute_engine_set_outcome_transforms(e, CODES)
        if c["cons"]:
            bt.boute_engine_set_constraints(e, p["cons"].cpu())
        args = [p["X"], p["Y"], p["ls"], p["s2"], p["noise"], p["ref"],
                _candidates(c, seed, p["dtau"]), _normals(c, seed)]
        out = [dev(B, k, dtype=torch.int64), dev(B, k)]
        taken = torch.zeros(B, N, dtype=torch.int8, device="cuda")
        if c["host"]:
            args = [None if a is None else a.cpu().pin_memory() for a in args]
            out, taken = [o.cpu().pin_memory() for o in out], taken.cpu()
        s.update(e=e, args=args, out=out, taken=taken, acq=dev(B, N), mean=dev(B, m, N),
                 var=dev(B, m, N),
                 call=bt.boute_engine_step_host if c["host"] else
                 bt.boute_engine_step if c["wait"] else bt.boute_engine_step_async)
        torch.cuda.synchronize()
        return s
    gp = bt.boute_gp_create(B, n, d, m)
    Ys = torch.empty_like(p["Y"])
    s.update(p, gp=gp, Ys=Ys)
    if kind == "gp":
        s.update(Xc=_candidates(c, seed, d), mean=dev(B, m, c["N"]), var=dev(B, m, c["N"]))
    else:  # the fit and the front of the step whose best candidates are refined
        cap = 2 * n + 2
        mask, P = dev(B, n, dtype=torch.uint8), dev(B, dtype=torch.int32)
        front, K = dev(B, n, m, dtype=F64), dev(B, dtype=torch.int32)
        lower, upper = dev(B, cap, m), dev(B, cap, m)
        bt.boute_standardize(p["Y"], Ys)
        bt.boute_gp_fit(gp, p["X"], Ys, p["ls"], p["s2"], p["noise"])
        bt.boute_pareto_front(Ys, B, n, m, p["ref"], mask, front, P)
        bt.boute_box_decompose(front, P, B, n, m, p["ref"], lower, upper, K)
        if bt.boute_gp_status(gp):
            raise RuntimeError("the fit failed")
        X0, eps = _ascent_inputs(c, seed)
        s.update(lower=lower, upper=upper, K=K, cap=cap, X0=X0, eps=eps, xlo=torch.zeros(d, device="cuda"),
                 xhi=torch.ones(d, device="cuda"), Xo=torch.empty_like(X0), grad=torch.empty_like(X0),
                 acq=dev(B, c["P"]))
    torch.cuda.synchronize()
    return s


LR = 0.01  # of the ascents
LEARN_LR = 0.05


def run(s):
    c, kind = s["c"], s["c"]["kind"]
    with torch.cuda.stream(s["stream"]):
        if kind == "step":
            idx, val = s["out"]
            s["call"](s["e"], *s["args"], idx, val)
            bt.boute_engine_scores(s["e"], acq=s["acq"], mean=s["mean"], var=s["var"])
            # the chosen candidates leave the pool
            s["taken"].zero_().scatter_(1, idx, 1)
            return dict(acq=s["acq"], mean=s["mean"], var=s["var"], val=val, taken=s["taken"])
        if kind == "gp":
            bt.boute_standardize(s["Y"], s["Ys"])
            bt.boute_gp_fit(s["gp"], s["X"], s["Ys"], s["ls"], s["s2"], s["noise"])
            bt.boute_gp_posterior(s["gp"], s["Xc"], c["N"], s["mean"], s["var"])
            return dict(mean=s["mean"], var=s["var"])
        if kind == "learn":
            bt.boute_gp_learn(s["X"], s["Ys"], s["theta0"], c["iters"], LEARN_LR, s["theta"],
                              s["mll"], s["grad"])
            return dict(theta=s["theta"], mll=s["mll"], grad=s["grad"])
        if kind == "ascent":
            bt.boute_acq_optimize(s["gp"], s["lower"], s["upper"], s["K"], s["cap"], s["eps"],
                                  c["S"], s["X0"], c["P"], s["xlo"], s["xhi"], c["steps"], LR,
                                  s["Xo"], s["acq"], s["grad"])
            return dict(X=s["Xo"], acq=s["acq"], grad=s["grad"])
        bt.boute_select_topk(s["acq"], c["B"], c["N"], c["k"], s["idx"], s["val"])
        return dict(idx=s["idx"], val=s["val"])


def work(case):
    c, kind = case, case["kind"]
    B = c["B"]
    if kind == "topk":
        return {"bytes": 4 * B * c["N"] + 12 * B * c["k"], "flops": 0}
    n, d, m = c["n"], c["d"], c.get("m", 2)
    if kind == "learn":  # per step: kernel and gradient entries, factor, its inverse, K^-1
        one = n ** 3 + n * n * (3 * d + 20)
        return {"bytes": 8 * (B * n * (d + m) + 3 * B * m * c["R"] * (d + 2)),
                "flops": B * m * c["R"] * one * (c["iters"] + 1)}
    if kind == "ascent":  # per step: k* and its gradient, W k*, W^T W k*, the draws
        one = 2 * (n * (6 * d + 20) + 2 * n * n) + c["S"] * 100
        return {"bytes": 4 * B * (m * n * n + n * d + 3 * c["P"] * d),
                "flops": B * c["P"] * one * (c["steps"] + 1)}
    N, S = c["N"], c.get("S", 0)
    extra = 2 * n * n + 2 * n * S if c.get("mode") == "nehvi" else 0
    flops = B * m * (N * (n * (n + 1) + n * (3 * d + 15) + extra + 30 * S) + 2 * n ** 3 // 3)
    out = 2 * m + (0 if kind == "gp" else 1)  # mean, var, acq
    return {"bytes": B * (4 * N * (d + out + m * S) + 8 * n * (d + m)), "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "topk":
        return "exact"
    if kind == "learn":  # 64 bits throughout; 1e-13 off where K is ill-conditioned
        return {"rel": 1e-11, "max": 1e-9}
    if kind == "ascent":  # a step's sign hangs on rounding where a gradient entry is near zero
        return {"rel": 5e-3, "max": 0.1}
    if kind == "gp":  # 2e-6 and 8e-6 off the 64-bit values
        return {"rel": 1e-5, "max": 4e-5}
    # 5e-6 and 2e-5 off; a sample within rounding of a threshold counts or does not
    flips = case["cons"] and case["S"] > 0
    return {"rel": 1e-3 if flips else 2e-5, "max": 0.5 if flips else 8e-5,
            "differ": min(0.01, 4.0 / case["N"])}


# ---- the same in 64 bits ----------------------------------------------------------------
def _kernel(xa, xb, ls, s2, dtau, kc):
    """k(xa, xb) without noise: Matern-5/2, or the composite kernel (kc: deployment and
    interaction outputscales, beta, preference entries)."""
    d = xa.shape[1]
    r2 = [xa.new_zeros(xa.shape[0], xb.shape[0]), xa.new_zeros(xa.shape[0], xb.shape[0])]
    for q in range(d):
        z = (xa[:, q, None] - xb[None, :, q]) / ls[q]
        r2[q >= dtau].addcmul_(z, z)
    s = SQRT5 * r2[0].sqrt()
    k52 = (1.0 + s + r2[0].mul_(5.0 / 3.0)) * torch.exp(-s)
    if kc is None:
        return s2 * k52
    s = SQRT3 * r2[1].sqrt()
    k32 = (1.0 + s) * torch.exp(-s)
    wa, wb = (torch.exp(kc[2] * (x[:, dtau:] @ kc[3:])) for x in (xa, xb))
    return s2 * k52 + kc[0] * wa[:, None] * wb[None, :] * k32 + kc[1] * k52 * k32


def _prior(x, s2, dtau, kc):
    if kc is None:
        return s2
    return s2 + kc[1] + kc[0] * torch.exp(kc[2] * (x[:, dtau:] @ kc[3:])) ** 2


def _standardised(c, p):
    Y = p["Y"]
    if c.get("comp"):
        Y = torch.stack([Y[..., 0].log(), -(Y[..., 1] / (1.0 - Y[..., 1])).log()], -1)
    return (Y - Y.mean(1, keepdim=True)) / Y.std(1, keepdim=True)


def _fit(p, Ys, b, t):
    """Kernel matrix without noise, L^-1 and alpha of one problem-objective."""
    X, kc = p["X"][b], None if p["kc"] is None else p["kc"][b, t]
    K0 = _kernel(X, X, p["ls"][b, t], p["s2"][b, t], p["dtau"], kc)
    eye = torch.eye(len(X), device="cuda", dtype=F64)
    L = torch.linalg.cholesky(K0 + p["noise"][b, t] * eye)
    W = torch.linalg.solve_triangular(L, eye, upper=False)
    return K0, W, W.T @ (W @ Ys[b, :, t])


def _chunks(N, per):
    step = max(1, (1 << 25) // per)
    return [(i, min(N, i + step)) for i in range(0, N, step)]


def _posterior(c, p, Ys, Xc):
    B, m, N = c["B"], c["m"], c["N"]
    mean, var = (torch.empty(B, m, N, device="cuda", dtype=F64) for _ in range(2))
    for b in range(B):
        for t in range(m):
            kc = None if p["kc"] is None else p["kc"][b, t]
            _, W, alpha = _fit(p, Ys, b, t)
            for i, j in _chunks(N, c["n"]):
                x = Xc[b, i:j].double()
                ks = _kernel(x, p["X"][b], p["ls"][b, t], p["s2"][b, t], p["dtau"], kc)
                mean[b, t, i:j] = ks @ alpha
                pr = _prior(x, p["s2"][b, t], p["dtau"], kc)
                var[b, t, i:j] = (pr - (ks @ W.T).square_().sum(1)).clamp_(min=0)
    return mean, var


def _front(F, ref):
    """Non-dominated rows of F strictly below ref, by the first objective."""
    F = np.unique(F[(F < ref).all(1)], axis=0)
    le = (F[None, :, :] <= F[:, None, :]).all(2)
    np.fill_diagonal(le, False)
    F = F[~le.any(1)]
    return F[np.lexsort(F.T[::-1])]


def _cells(F, ref):
    """Disjoint boxes (lower, upper per objective) of the region below ref that no row of F
    dominates; two objectives: strips; three: strips per slab of the third."""
    inf = np.inf
    if len(ref) == 2:
        F = _front(F, ref) if len(F) else F.reshape(0, 2)
        a = np.concatenate([[-inf], F[:, 0]])
        b = np.concatenate([F[:, 0], ref[:1]])
        u = np.concatenate([ref[1:], F[:, 1]])
        return [((a[i], -inf), (b[i], u[i])) for i in range(len(a))]
    z = np.concatenate([[-inf], np.unique(F[:, 2]), ref[2:]])
    out = []
    for k in range(len(z) - 1):
        below = F[F[:, 2] <= z[k], :2]
        out += [((*lo, z[k]), (*hi, z[k + 1])) for lo, hi in _cells(below, ref[:2])]
    return out


def _improvement(y, cells):
    h = torch.zeros_like(y[0])
    for lo, hi in cells:
        v = None
        for t, yt in enumerate(y):
            w = (hi[t] - (yt if lo[t] == -math.inf else yt.clamp(min=lo[t]))).clamp_(min=0)
            v = w if v is None else v.mul_(w)
        h += v
    return h


def _psi(v, mu, sd, k):
    """E[(v - Y)+ 1[Y <= k]], Y ~ N(mu, sd^2)."""
    z = ((v if k is None else min(v, k)) - mu) / sd
    return (v - mu) * torch.special.ndtr(z) + sd * torch.exp(-0.5 * z * z) / math.sqrt(2 * math.pi)


def _insample_normals(b, rows, n):
    """Rows of n fp32 normals of problem b: Philox4x64-10 counters (j, row, b, 0), Box-Muller."""
    out = np.empty((rows, n), np.float32)
    for r in range(rows):
        at = ((r << 64) + (b << 128) - 1) % (1 << 256)  # numpy steps the counter first
        w = np.random.Philox(key=INSAMPLE_KEY, counter=at).random_raw(4 * ((n + 3) // 4))
        u = ((w >> np.uint64(11)).astype(np.float64) + 0.5) * 2.0 ** -53
        rad, ang = np.sqrt(-2.0 * np.log(u[0::2])), 2.0 * np.pi * u[1::2]
        out[r] = np.stack([rad * np.cos(ang), rad * np.sin(ang)], 1).reshape(-1)[:n]
    return torch.from_numpy(out).cuda().double()


def _noisy(c, p, Ys, Xc, eps):
    B, n, N, S = c["B"], c["n"], c["N"], c["S"]
    acq = torch.empty(B, N, device="cuda", dtype=F64)
    mean, var = (torch.empty(B, 2, N, device="cuda", dtype=F64) for _ in range(2))
    eye = torch.eye(n, device="cuda", dtype=F64)
    for b in range(B):
        z = _insample_normals(b, 2 * S, n).reshape(2, S, n)
        obj, Yin = [], []
        for t in range(2):
            K0, W, alpha = _fit(p, Ys, b, t)
            V = W @ K0
            Fc = torch.linalg.cholesky(K0 - V.T @ V + JITTER * p["s2"][b, t] * eye)
            Yin.append((K0 @ alpha)[None] + z[t] @ Fc.T)
            obj.append((W, V, Fc, alpha))
        Yin = torch.stack(Yin, 2).cpu().numpy()
        k = p["cons"][b].cpu().numpy() if c["cons"] else np.full(2, np.inf)
        ref = p["ref"][b].cpu().numpy()
        cells = [_cells(Y[(Y <= k).all(1)], ref) for Y in Yin]
        width = max(map(len, cells))
        pad = np.zeros((4, S, width))  # l1, u1, u2 per strip of each draw; zero: no strip
        for s, cs in enumerate(cells):
            for q, (lo, hi) in enumerate(cs):
                pad[:3, s, q] = max(lo[0], -1e300), hi[0], hi[1]
        pad = torch.from_numpy(pad).cuda()
        for i, j in _chunks(N, 4 * max(n, S)):
            x, y = Xc[b, i:j].double(), []
            for t in range(2):
                W, V, Fc, alpha = obj[t]
                ks = _kernel(x, p["X"][b], p["ls"][b, t], p["s2"][b, t], p["dtau"], None)
                a = ks @ W.T
                l = torch.linalg.solve_triangular(Fc, (ks - a @ V).T, upper=False)
                mean[b, t, i:j] = ks @ alpha
                var[b, t, i:j] = (p["s2"][b, t] - (a * a).sum(1) - (l * l).sum(0)).clamp(min=0)
                y.append(mean[b, t, i:j, None] + (z[t] @ l).T +
                         var[b, t, i:j, None].sqrt() * eps[b, i:j, t].double())
            h = torch.zeros_like(y[0])
            for q in range(width):
                l1, u1, u2 = pad[0, :, q], pad[1, :, q], pad[2, :, q]
                h += (u1 - torch.maximum(l1, y[0])).clamp(min=0) * (u2 - y[1]).clamp(min=0)
            if c["cons"]:
                h *= (y[0] <= k[0]) & (y[1] <= k[1])
            acq[b, i:j] = h.mean(1)
    return acq, mean, var


def _exact_step(c, seed):
    p = _problem(c, seed)
    Ys = _standardised(c, p)
    Xc, eps = _candidates(c, seed, p["dtau"]), _normals(c, seed)
    B, m, N = c["B"], c["m"], c["N"]
    if c["mode"] == "nehvi":
        acq, mean, var = _noisy(c, p, Ys, Xc, eps)
    else:
        mean, var = _posterior(c, p, Ys, Xc)
        acq = torch.zeros(B, N, device="cuda", dtype=F64)
        for b in range(B):
            ref = p["ref"][b].cpu().numpy()
            k = p["cons"][b].tolist() if c["cons"] else [None] * m
            cells = _cells(_front(Ys[b].cpu().numpy(), ref), ref)
            for i, j in _chunks(N, 8 * max(1, c["S"])):
                mu, sd = mean[b, :, i:j], var[b, :, i:j].sqrt()
                if c["mode"] == "ehvi":
                    last = 0.0
                    for lo, hi in cells:
                        up = _psi(hi[0], mu[0], sd[0], k[0])
                        acq[b, i:j] += (up - last) * _psi(hi[1], mu[1], sd[1], k[1])
                        last = up
                    continue
                y = [mu[t, :, None] + sd[t, :, None] * eps[b, i:j, t].double() for t in range(m)]
                h = _improvement(y, cells)
                for t in range(m):
                    if c["cons"]:
                        h *= y[t] <= k[t]
                acq[b, i:j] = h.mean(1)
    val, idx = acq.topk(c["k"], 1)
    taken = torch.zeros(B, N, dtype=torch.int8, device="cuda").scatter_(1, idx, 1)
    return dict(acq=acq, mean=mean, var=var, val=val, taken=taken)


def _exact_learn(c, seed):
    X, Ys, th = _learn_inputs(c, seed)
    d, n = c["d"], c["n"]
    lo = torch.tensor([-math.log(1e3)] * (d + 1) + [math.log(1e-4)], device="cuda", dtype=F64)
    hi = torch.tensor([math.log(1e3)] * (d + 1) + [math.log(10.0)], device="cuda", dtype=F64)
    y = Ys.permute(0, 2, 1)[:, :, None, :, None]
    dx = X[:, None, None, :, None, :] - X[:, None, None, None, :, :]
    eye = torch.eye(n, device="cuda", dtype=F64)

    def value_grad(th):
        th = th.detach().requires_grad_()
        r2 = (dx / th[..., None, None, :d].exp()).square().sum(-1)
        s = SQRT5 * (r2 + 1e-300).sqrt()
        K = (1.0 + s + 5.0 / 3.0 * r2) * torch.exp(-s) * th[..., d, None, None].exp()
        L = torch.linalg.cholesky(K + th[..., d + 1, None, None].exp() * eye)
        a = torch.linalg.solve_triangular(L, y.expand(*L.shape[:-1], 1), upper=False)
        mll = (-0.5 * a.square().sum((-1, -2)) - L.diagonal(dim1=-2, dim2=-1).log().sum(-1) -
               0.5 * n * math.log(2 * math.pi))
        return mll.detach(), torch.autograd.grad(mll.sum(), th)[0]

    th = torch.minimum(torch.maximum(th, lo), hi)
    m1, m2 = torch.zeros_like(th), torch.zeros_like(th)
    for it in range(1, c["iters"] + 1):
        g = value_grad(th)[1]
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        th = th + LEARN_LR * (m1 / (1 - 0.9 ** it)) / ((m2 / (1 - 0.999 ** it)).sqrt() + 1e-8)
        th = torch.minimum(torch.maximum(th, lo), hi)
    mll, g = value_grad(th)
    return dict(theta=th, mll=mll, grad=g)


def _exact_ascent(c, seed):
    p = _problem(c, seed)
    Ys = _standardised(c, p)
    X0, eps = _ascent_inputs(c, seed)
    out = dict(X=[], acq=[], grad=[])
    for b in range(c["B"]):
        fits = [_fit(p, Ys, b, t) for t in range(2)]
        ref = p["ref"][b].cpu().numpy()
        cells = _cells(_front(Ys[b].cpu().numpy(), ref), ref)

        def value_grad(x):
            x = x.detach().requires_grad_()
            y = []
            for t, (_, W, alpha) in enumerate(fits):
                z = (x[:, None, :] - p["X"][b][None]) / p["ls"][b, t]
                r2 = z.square().sum(-1)
                s = SQRT5 * (r2 + 1e-300).sqrt()
                ks = p["s2"][b, t] * (1.0 + s + 5.0 / 3.0 * r2) * torch.exp(-s)
                sd = (p["s2"][b, t] - (ks @ W.T).square().sum(1)).clamp(min=1e-300).sqrt()
                y.append((ks @ alpha)[:, None] + sd[:, None] * eps[t].double())
            h = 0.0
            for lo, hi in cells:
                w = hi[0] - (y[0] if lo[0] == -math.inf else y[0].clamp(min=lo[0]))
                h = h + w.clamp(min=0) * (hi[1] - y[1]).clamp(min=0)
            v = h.mean(1)
            return v.detach(), torch.autograd.grad(v.sum(), x)[0]

        x = X0[b].double()
        m1, m2 = torch.zeros_like(x), torch.zeros_like(x)
        for it in range(1, c["steps"] + 1):
            g = value_grad(x)[1]
            m1 = 0.9 * m1 + 0.1 * g
            m2 = 0.999 * m2 + 0.001 * g * g
            x = x + LR * (m1 / (1 - 0.9 ** it)) / ((m2 / (1 - 0.999 ** it)).sqrt() + 1e-8)
            x = x.clamp(0.0, 1.0)
        v, g = value_grad(x)
        for key, a in (("X", x), ("acq", v), ("grad", g)):
            out[key].append(a)
    return {key: torch.stack(a) for key, a in out.items()}


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "topk":
        acq = _scores(c, seed)
        val, idx = torch.sort(acq, dim=1, descending=True, stable=True)
        return dict(idx=idx[:, :c["k"]].contiguous(), val=val[:, :c["k"]].double())
    if kind == "learn":
        return _exact_learn(c, seed)
    if kind == "ascent":
        return _exact_ascent(c, seed)
    if c["B"] * c["m"] * c["N"] * c["n"] ** 2 > 4e12:
        return None  # over about 20 seconds in 64 bits
    if kind == "step":
        return _exact_step(c, seed)
    p = _problem(c, seed)
    mean, var = _posterior(c, p, _standardised(c, p), _candidates(c, seed, c["d"]))
    return dict(mean=mean, var=var)
