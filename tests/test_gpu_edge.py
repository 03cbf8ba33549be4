"""Edge cases of the CUDA path against the oracle: ragged and tiny sizes, one
training point, several output-column passes, extreme dimensions, an empty
front, candidates on training points, zero variance, ties in selection,
shared base normals, per-objective hyperparameters, a singular kernel matrix
and invalid arguments."""
import numpy as np
import pytest

import oracle
from _pipeline import (POST_REL, HostProblem, check_acq, check_acq_end_to_end, check_mean,
                       check_var, gpu_pipeline, host_problem, oracle_fit)
from oracle import pipeline as opl
from paper_2602_10729_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def custom(X, Y, Xc, *, ls=None, s2=None, noise=None, ref=None, mode="ehvi", S=0, k=4,
           eps=None):
    X = np.asarray(X, np.float64)[None] if np.ndim(X) == 2 else np.asarray(X, np.float64)
    Y = np.asarray(Y, np.float64)[None] if np.ndim(Y) == 2 else np.asarray(Y, np.float64)
    Xc = np.asarray(Xc, np.float32)[None] if np.ndim(Xc) == 2 else np.asarray(Xc, np.float32)
    B, n, d = X.shape
    m = Y.shape[2]
    N = Xc.shape[1]
    ls = np.full((B, m, d), 0.3) if ls is None else np.broadcast_to(ls, (B, m, d)).copy()
    s2 = np.ones((B, m)) if s2 is None else np.broadcast_to(s2, (B, m)).copy()
    noise = np.full((B, m), 1e-4) if noise is None else np.broadcast_to(noise, (B, m)).copy()
    ref = np.full((B, m), 1.1) if ref is None else np.broadcast_to(ref, (B, m)).copy()
    w = wl.Workload("custom", B, n, d, m, N, mode, S, min(k, N), tuple(range(B)), 0,
                    ref=tuple(ref[0]))
    return HostProblem(w, X, Y, ls, s2, noise, ref, Xc, eps)


def compare(hp, check_topk=True):
    g = gpu_pipeline(hp)
    assert g["status"] == 0, g["status"]
    w = hp.w
    for b in range(w.B):
        fp = opl.fit_problem(hp.X[b], hp.Y[b], hp.ls[b], hp.s2[b], hp.noise[b], hp.ref[b])
        assert g["mask"][b].tolist() == fp.mask.tolist()
        assert int(g["P"][b]) == fp.front.shape[0]
        mean, var = opl.posterior(fp, hp.Xc[b])
        for t in range(w.m):
            check_mean(g["mean"][b, t], mean[:, t], fp.s2[t])
            check_var(g["var"][b, t], var[:, t], fp.s2[t])
        eps = None if hp.eps is None else hp.eps[b]
        check_acq_end_to_end(g["acq"][b], lambda mm, vv: opl.acquisition(fp, mm, vv, w.mode, eps),
                             g["mean"][b].T, g["var"][b].T, mean, var, fp.s2)
    return g


def rand_problem(seed, n, d, m, N, mode="ehvi", S=0, **kw):
    rng = np.random.default_rng(seed)
    X = rng.random((n, d))
    Y = np.stack([((X - c) ** 2).sum(1) for c in np.linspace(0.2, 0.8, m)], 1)
    Y += rng.normal(0, 0.01, Y.shape)
    Xc = rng.random((N, d)).astype(np.float32)
    eps = rng.standard_normal((1, N, m, S)).astype(np.float32) if mode == "mc" else None
    return custom(X, Y, Xc, mode=mode, S=S, eps=eps, **kw)


@pytest.mark.parametrize("N", [1, 2, 127, 128, 129, 300])
def test_ragged_candidate_counts(N):
    compare(rand_problem(1, 20, 4, 2, N))


@pytest.mark.parametrize("n", [1, 2, 31, 33, 97, 129, 150, 160, 161, 255, 257, 600])
def test_training_set_sizes_and_column_passes(n):
    compare(rand_problem(2, n, 5, 2, 400))


def check_posterior_at(hp, at, mean_g, var_g):
    """Problem 0's means and variances (m x N) at the candidates `at`: POST_REL of the
    prior's scale. The composite kernel's means are never recomputed, so they get in
    addition what rounding K* (a few units in the last place of each value, 16 allowed
    for its exponents) leaves of the terms K*_j alpha_j."""
    fp = oracle_fit(hp, 0)
    mean, var = opl.posterior(fp, hp.Xc[0][at])
    for t in range(hp.w.m):
        g = mean_g[t, at].astype(np.float64)
        if hp.kc is None:
            check_mean(g, mean[:, t], fp.s2[t])
            check_var(var_g[t, at], var[:, t], fp.s2[t])
            continue
        kern, x = (hp.d_tau, hp.kc[0][t]), hp.Xc[0][at].astype(np.float64)
        args = (hp.ls[0][t], hp.s2[0][t], kern)
        prior = max(oracle.kernel(c, c, *args) for c in x)
        terms = [sum(oracle.kernel(c, r, *args) * abs(a) for r, a in zip(hp.X[0], fp.alpha[t]))
                 for c in x]
        bound = 16 * 2.0 ** -23 * np.array(terms) + POST_REL * np.sqrt(prior)
        assert np.all(np.isfinite(g)) and np.all(np.abs(g - mean[:, t]) <= bound)
        check_var(var_g[t, at], var[:, t], prior)


@pytest.mark.parametrize("n,d,comp", [(520, 32, True), (640, 32, True), (640, 16, True),
                                      (640, 24, False), (777, 32, False), (640, 10, False),
                                      (900, 20, True), (1090, 12, False)])
def test_cached_chunks_over_many_tiles(n, d, comp):
    """More than 512 observations (a second group of output blocks takes the
    first one's K* chunks from the cache) and enough candidates that every CTA
    works through several tiles: runs of cached chunks at the end of one tile
    meet the chunks built for the next. Sampled candidates."""
    import dataclasses

    base = wl.scaled(dataclasses.replace(wl.WORKLOADS[2], d=d), N=60011, n=n)
    hp = host_problem(wl.composite(base) if comp else base)
    g = gpu_pipeline(hp)
    assert g["status"] == 0
    check_posterior_at(hp, np.unique(np.r_[np.arange(0, 60011, 233), 60010]), g["mean"][0],
                       g["var"][0])


@pytest.mark.parametrize("d", [1, 3, 8, 9, 13, 17, 25, 32])
def test_dimensions(d):
    # lengthscale 0.2 sqrt(d) as in the workloads; 1-D with few points keeps
    # the kernel matrix well conditioned (see the ill-conditioned test below)
    n, ls = (6, 0.1) if d == 1 else (40, 0.2 * np.sqrt(d))
    compare(rand_problem(3, n, d, 2, 300, ls=ls))


@pytest.mark.parametrize("n,d,m,N,mode,S", [(600, 20, 2, 700, "ehvi", 0),
                                            (777, 24, 3, 385, "mc", 64),
                                            (97, 32, 3, 257, "mc", 64)])
def test_wide_candidates_large_and_ragged(n, d, m, N, mode, S):
    # d > 16: the builders take candidate rows in pairs; n > 512 adds the
    # cached K* chunks of a second group; n, N not multiples of the chunk and
    # the tile; n = 777 with three objectives puts the MC kernel's boxes
    # (2n + 2) just under 48 KB of dynamic shared memory, beside its static
    # staging
    compare(rand_problem(13, n, d, m, N, mode=mode, S=S, ls=0.2 * np.sqrt(d)))


@pytest.mark.parametrize("n", [420, 440])
def test_kstar_side_input_near_48kb(n):
    # K* beside the fit (the engine, few candidates): the side input of
    # n = 420 .. 448 points at d = 12 needs just under 48 KB of dynamic shared
    # memory next to the K* kernel's static array
    import torch

    from paper_2602_10729_gb300 import boute as bt
    w = wl.scaled(wl.WORKLOADS[1], N=2048 + 5, B=1, n=n)
    hp = host_problem(w)
    dev = torch.device("cuda")
    t = lambda a, dt: torch.as_tensor(a, dtype=dt, device=dev)
    e = bt.Engine(1, w.n, w.d, w.m, w.N, bt.BOUTE_ACQ_MC_HVI, w.S, w.k)
    idx = torch.empty((1, w.k), dtype=torch.int64, device=dev)
    val = torch.empty((1, w.k), dtype=torch.float32, device=dev)
    bt.boute_engine_step(e, t(hp.X, torch.float64), t(hp.Y, torch.float64),
                         t(hp.ls, torch.float64), t(hp.s2, torch.float64),
                         t(hp.noise, torch.float64), t(hp.ref, torch.float64),
                         t(hp.Xc, torch.float32), t(hp.eps, torch.float32), idx, val)
    mean = torch.empty((1, w.m, w.N), dtype=torch.float32, device=dev)
    var = torch.empty_like(mean)
    bt.boute_engine_scores(e, None, mean, var)
    torch.cuda.synchronize()
    e.free()
    fp = oracle_fit(hp, 0)
    mo, vo = opl.posterior(fp, hp.Xc[0])
    for tt in range(w.m):
        check_mean(mean[0, tt].cpu().numpy(), mo[:, tt], fp.s2[tt])
        check_var(var[0, tt].cpu().numpy(), vo[:, tt], fp.s2[tt])


# The K* kernel stages the whole side input, which passes a block's shared memory from
# n = 833 at 29 .. 32 dimensions, 961 at 25 .. 28, 1089 at 21 .. 24 and 1601 at 15 or 16
# on: an engine then builds K* inside the posterior, also with so few candidates that
# its buffer is small. Both sides of the lines; then fewer observations in the same engine.
@pytest.mark.parametrize("n,d,comp", [(832, 32, False), (833, 32, False), (1000, 28, False),
                                      (960, 25, True), (961, 25, True), (1024, 32, True),
                                      (1088, 24, False), (1089, 24, False), (1601, 16, False)])
def test_engine_where_the_side_input_passes_shared_memory(n, d, comp):
    import dataclasses

    import torch

    from paper_2602_10729_gb300 import boute as bt
    base = wl.scaled(dataclasses.replace(wl.WORKLOADS[2], d=d), N=300, n=n)
    w = wl.composite(base) if comp else base
    hp = host_problem(w)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    e = bt.Engine(1, n, d, w.m, w.N, bt.BOUTE_ACQ_EHVI2D, 0, w.k)
    if comp:
        bt.boute_engine_set_kernel(e, hp.d_tau, hp.kc)
        bt.boute_engine_set_outcome_transforms(e, list(hp.transforms))
    idx = torch.empty((1, w.k), dtype=torch.int64, device="cuda")
    val = torch.empty((1, w.k), dtype=torch.float32, device="cuda")
    mean = torch.empty((1, w.m, w.N), dtype=torch.float32, device="cuda")
    var = torch.empty_like(mean)
    at = np.arange(0, 300, 7)
    stream = torch.cuda.Stream()  # (steps are captured as graphs)
    for rows in (n, 65):
        if rows < n:
            bt.boute_engine_set_n(e, rows)
            hp.X, hp.Y = hp.X[:, :rows], hp.Y[:, :rows]
        args = [t(hp.X), t(hp.Y), t(hp.ls), t(hp.s2), t(hp.noise), t(hp.ref),
                t(hp.Xc, torch.float32)]
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            bt.boute_engine_step(e, *args, None, idx, val)
            bt.boute_engine_scores(e, None, mean, var)
        torch.cuda.synchronize()
        check_posterior_at(hp, at, mean[0].cpu().numpy(), var[0].cpu().numpy())
    e.free()


@pytest.mark.parametrize("n,d,N,beside", [(128, 24, 143323, True), (32, 20, 389083, True),
                                          (64, 17, 532443, True), (128, 16, 194523, True),
                                          (128, 16, 532443, False), (64, 16, 389083, False),
                                          (160, 7, 129627, False), (128, 24, 600000, False),
                                          (512, 12, 48603, False)])
@pytest.mark.parametrize("comp", [False, True])
def test_kstar_beside_the_fit_where_it_is_faster(n, d, N, beside, comp):
    """A step with K* beside the fit launches one kernel more (its own), as one with few
    candidates does: up to 512 MiB of K* from 17 dimensions on and with the composite kernel,
    256 with 9 to 16 and 65 to 448 observations, else 128."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    hp = rand_problem(31, n, d, 2, 1, ls=0.2 * np.sqrt(d))
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    mib = (N + 127) // 128 * 2 * ((n + 63) // 64) / 32
    beside = mib <= 512 if comp else beside
    count = []
    for cands in (20000, N):
        e = bt.Engine(1, n, d, 2, cands, bt.BOUTE_ACQ_EHVI2D, 0, 4)
        if comp:  # (set while the engine holds fewer observations than it was made for)
            bt.boute_engine_set_n(e, 5)
            bt.boute_engine_set_kernel(e, d // 2, np.full((1, 2, 3 + d - d // 2), 0.1))
            bt.boute_engine_set_n(e, n)
        Xc = torch.rand((1, cands, d), device="cuda")
        idx = torch.empty((1, 4), dtype=torch.int64, device="cuda")
        val = torch.empty((1, 4), dtype=torch.float32, device="cuda")
        l0 = bt.boute_launch_count()
        bt.boute_engine_step(e, t(hp.X), t(hp.Y), t(hp.ls), t(hp.s2), t(hp.noise), t(hp.ref), Xc,
                             None, idx, val)
        count.append(bt.boute_launch_count() - l0)
        e.free()
    assert count[0] - count[1] == (0 if beside else 1)


def test_ill_conditioned_problem_meets_fp32_error_bound():
    """40 points on a line with lengthscale 0.3: cond(K) ~ 2e5, |alpha| ~ 1e3.
    The mean meets 1e-5 (its ill-conditioned rows are recomputed in pairs of floats); the
    variance s2 - ||L^-1 k*||^2 must stay within the error bound of an
    fp32-accurate contraction, eps32 * s2 times cond-scaled terms."""
    hp = rand_problem(12, 40, 1, 2, 300)
    g = gpu_pipeline(hp)
    assert g["status"] == 0
    fp = opl.fit_problem(hp.X[0], hp.Y[0], hp.ls[0], hp.s2[0], hp.noise[0], hp.ref[0])
    mean, var = opl.posterior(fp, hp.Xc[0])
    eps32 = np.finfo(np.float32).eps
    for t in range(2):
        Ks = np.array([[oracle.matern52(c.astype(np.float64), x, hp.ls[0][t], hp.s2[0][t])
                        for x in hp.X[0]] for c in hp.Xc[0]])
        check_mean(g["mean"][0, t], mean[:, t], fp.s2[t])
        W = np.linalg.inv(fp.L[t])
        v = Ks @ W.T
        bound_v = 64 * eps32 * 2 * (np.abs(v) * (np.abs(Ks) @ np.abs(W.T))).sum(1) + 1e-5
        assert np.all(np.abs(g["var"][0, t] - var[:, t]) <= bound_v)


@pytest.mark.parametrize("n,d,N,B", [(60, 5, 20_000, 2), (33, 9, 130, 1), (129, 20, 999, 3)])
def test_ill_conditioned_rows_of_many_tiles(n, d, N, B):
    """Long lengthscales, so that most rows are recomputed, over several tiles per CTA, a
    ragged last tile, problems and objectives; by the handle (K* built inside the posterior)
    and by an engine step (K* staged)."""
    import dataclasses

    import torch

    from paper_2602_10729_gb300 import boute as bt
    w = wl.scaled(dataclasses.replace(wl.WORKLOADS[4], d=d, k=4), N=N, B=B, n=n)
    hp = host_problem(w)
    hp.ls *= 4.0
    g = gpu_pipeline(hp)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    e = bt.Engine(B, n, d, 2, N, bt.BOUTE_ACQ_EHVI2D, 0, 4)
    idx = torch.empty((B, 4), dtype=torch.int64, device="cuda")
    val = torch.empty((B, 4), dtype=torch.float32, device="cuda")
    mean = torch.empty((B, 2, N), dtype=torch.float32, device="cuda")
    bt.boute_engine_step(e, t(hp.X), t(hp.Y), t(hp.ls), t(hp.s2), t(hp.noise), t(hp.ref),
                         t(hp.Xc, torch.float32), None, idx, val)
    bt.boute_engine_scores(e, None, mean, None)
    torch.cuda.synchronize()
    e.free()
    at = np.unique(np.r_[np.arange(0, N, 37), N - 1])
    marked = 0
    for b in range(B):
        fp = oracle_fit(hp, b)
        mo, _ = opl.posterior(fp, hp.Xc[b][at])
        for k in range(2):
            check_mean(g["mean"][b, k, at], mo[:, k], fp.s2[k])
            check_mean(mean[b, k].cpu().numpy()[at], mo[:, k], fp.s2[k])
            ks = np.array([[oracle.matern52(c, x, hp.ls[b][k], hp.s2[b][k]) for x in hp.X[b]]
                           for c in hp.Xc[b][at[:20]].astype(np.float64)])
            terms = ks @ np.abs(fp.alpha[k])
            marked += int((terms > 224 * np.maximum(np.abs(mo[:20, k]), np.sqrt(fp.s2[k]))).sum())
    assert marked > 5 * B


def test_recomputed_means_do_not_hold_up_the_posterior():
    """Every row recomputed: eight times the posterior without any (by one warp of
    four at a time, beside the tensor cores, 24 times)."""
    import dataclasses

    import torch

    from paper_2602_10729_gb300 import boute as bt
    w = wl.scaled(dataclasses.replace(wl.WORKLOADS[4], d=8), N=32768, B=1, n=400)
    hp = host_problem(w)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    X, Y, Xc = t(hp.X), t(hp.Y), t(hp.Xc, torch.float32)
    bt.boute_standardize(Y, Y)
    mean = torch.empty((1, 2, w.N), dtype=torch.float32, device="cuda")
    var = torch.empty_like(mean)
    gp = bt.boute_gp_create(1, w.n, w.d, 2)
    us = []
    for f in (0.4, 2.0):
        bt.boute_gp_fit(gp, X, Y, t(hp.ls * f), t(hp.s2), t(hp.noise))
        assert bt.boute_gp_status(gp) == 0
        us.append(_graph_us(lambda: bt.boute_gp_posterior(gp, Xc, w.N, mean, var), 4))
    gp.free()
    assert us[1] < 14 * us[0], us


def test_three_objectives_monte_carlo_and_box_decomposition():
    hp = rand_problem(4, 90, 6, 3, 500, mode="mc", S=64)
    g = compare(hp)
    # the boxes tile the improvement region: their volume inside [lb, ref]
    # equals vol([lb, ref]) - HV(front)
    fp = opl.fit_problem(hp.X[0], hp.Y[0], hp.ls[0], hp.s2[0], hp.noise[0], hp.ref[0])
    K = int(g["K"][0])
    lo, up = g["lower"][0][:K].astype(np.float64), g["upper"][0][:K].astype(np.float64)
    lb = fp.front.min(0) - 1.0 if len(fp.front) else hp.ref[0] - 1.0
    vol = np.prod(np.clip(up - np.maximum(lo, lb), 0, None), 1).sum()
    want = np.prod(hp.ref[0] - lb) - oracle.hv(fp.front, hp.ref[0])
    assert vol == pytest.approx(want, rel=1e-5)
    assert K <= 2 * len(fp.front) + 1


def test_monte_carlo_scalar_path_and_shared_normals():
    # S = 50 is not a multiple of 128 (scalar path); also shared normals
    hp = rand_problem(5, 50, 4, 2, 260, mode="mc", S=50)
    compare(hp)
    import torch

    from paper_2602_10729_gb300 import boute as bt
    fp = opl.fit_problem(hp.X[0], hp.Y[0], hp.ls[0], hp.s2[0], hp.noise[0], hp.ref[0])
    mean, var = opl.posterior(fp, hp.Xc[0])
    eps1 = hp.eps[0, :1]  # one m x S block for every candidate
    want = oracle.mc_hvi(mean.astype(np.float32).astype(np.float64),
                         var.astype(np.float32).astype(np.float64), eps1, fp.front, fp.ref,
                         eps_stride=0)
    dev = "cuda"
    n, m, N = hp.w.n, 2, 260
    front = torch.zeros((1, n, m), dtype=torch.float64, device=dev)
    front[0, :len(fp.front)] = torch.as_tensor(fp.front)
    P = torch.tensor([len(fp.front)], dtype=torch.int32, device=dev)
    ref = torch.as_tensor(fp.ref[None], device=dev)
    cap = 2 * n + 2
    lower = torch.empty((1, cap, m), dtype=torch.float32, device=dev)
    upper = torch.empty_like(lower)
    K = torch.empty(1, dtype=torch.int32, device=dev)
    bt.boute_box_decompose(front, P, 1, n, m, ref, lower, upper, K)
    acq = torch.empty((1, N), dtype=torch.float32, device=dev)
    bt.boute_acq_mc_hvi(torch.as_tensor(mean.T.astype(np.float32)[None].copy(), device=dev),
                        torch.as_tensor(var.T.astype(np.float32)[None].copy(), device=dev), 1, N,
                        m, lower, upper, K, cap, torch.as_tensor(eps1, device=dev), hp.w.S, 0, acq)
    check_acq(acq.cpu().numpy()[0], want)


def test_empty_front():
    hp = rand_problem(6, 30, 3, 2, 200, ref=-5.0)  # nothing is better than ref
    g = compare(hp)
    assert int(g["P"][0]) == 0


def test_candidates_on_training_points():
    rng = np.random.default_rng(7)
    X = rng.random((25, 3)).astype(np.float32).astype(np.float64)
    Y = np.stack([X.sum(1), (1 - X).sum(1)], 1) + rng.normal(0, 0.01, (25, 2))
    hp = custom(X, Y, X.astype(np.float32), noise=1e-6)
    g = compare(hp)
    assert g["var"].max() < 1e-3


def test_per_objective_hyperparameters():
    """Per-objective lengthscales over an order of magnitude and noise down to
    1e-5: sum_j |K*_j alpha_j| reaches about 220 times the mean's scale, and
    the mean must still meet 1e-5 (the fp32 K* with its exponent-rounding
    correction and compensated sums)."""
    rng = np.random.default_rng(8)
    hp = rand_problem(9, 70, 5, 2, 333)
    hp.ls[0] = rng.uniform(0.1, 1.5, (2, 5))
    hp.s2[0] = [0.5, 2.5]
    hp.noise[0] = [1e-3, 1e-5]
    compare(hp)


@pytest.mark.parametrize("ls_range,noise", [((0.3, 1.5), (1e-3, 1e-4)), ((0.5, 2.0), (1e-3, 1e-5)),
                                            ((0.1, 1.5), (1e-5, 1e-6))])
def test_ill_conditioned_means(ls_range, noise):
    """Longer lengthscales or smaller noise: sum_j |K*_j alpha_j| reaches 270
    to 590 times the mean's scale. Rows beyond 224 times are recomputed in pairs of
    floats; mean and variance meet 1e-5 everywhere."""
    rng = np.random.default_rng(8)
    hp = rand_problem(9, 70, 5, 2, 333)
    hp.ls[0] = rng.uniform(*ls_range, (2, 5))
    hp.s2[0] = [0.5, 2.5]
    hp.noise[0] = list(noise)
    g = gpu_pipeline(hp)
    assert g["status"] == 0
    fp = opl.fit_problem(hp.X[0], hp.Y[0], hp.ls[0], hp.s2[0], hp.noise[0], hp.ref[0])
    mean, var = opl.posterior(fp, hp.Xc[0])
    for t in range(2):
        check_mean(g["mean"][0, t], mean[:, t], fp.s2[t])
        check_var(g["var"][0, t], var[:, t], fp.s2[t])


def test_far_candidates_and_zero_variance_ehvi():
    hp = rand_problem(10, 30, 3, 2, 150)
    hp.Xc[0, :20] += 50.0  # far field: mean 0, var s2
    compare(hp)


# one block, segments of 8192 around their edges, a second and a third level,
# k from 1 to 1024 (above a block's 512 threads the selection searches every key)
@pytest.mark.parametrize("N,k", [(16384, 1024), (16385, 1024), (16385, 512), (24577, 513),
                                 (8193 * 16, 100), (1, 1), (1024, 1024), (2_000_003, 1000),
                                 (140_000, 1024)])
def test_topk_levels_and_k_range(N, k):
    import torch

    from paper_2602_10729_gb300 import boute as bt
    rng = np.random.default_rng(N + k)
    v = rng.standard_normal((4, N)).astype(np.float32)
    v[1] = np.sort(v[1])  # every survivor in one segment, on few threads
    v[2] = np.where(v[2] > 1.0, np.round(v[2], 1), 0.0)  # ties around and at zero
    v[3, rng.random(N) < 0.9] = np.nan
    v[3, : N // 3] = -np.inf
    a = torch.as_tensor(v, device="cuda")
    idx = torch.empty((4, k), dtype=torch.int64, device="cuda")
    val = torch.empty((4, k), dtype=torch.float32, device="cuda")
    bt.boute_select_topk(a, 4, N, k, idx, val)
    key = np.where(np.isnan(v), -np.inf, v)
    for b in range(4):  # the definition: value descending, then index
        want = np.lexsort((np.arange(N), -key[b]))[:k]
        assert np.array_equal(idx[b].cpu().numpy(), want)
        assert np.array_equal(val[b].cpu().numpy(), v[b][want], equal_nan=True)


# blocks of 128 to 1024 threads at their edges, one level and two, scores mostly equal:
# fewer others than k, as many, more, none
@pytest.mark.parametrize("N,k", [(2048, 64), (2048, 65), (2049, 60), (4096, 128), (4096, 129),
                                 (4097, 32), (8192, 256), (8193, 256), (8192, 257), (8192, 1024),
                                 (16384, 7), (20_000, 40), (300_000, 64), (300_000, 700), (60, 60)])
def test_topk_mostly_equal_scores(N, k):
    import torch

    from paper_2602_10729_gb300 import boute as bt
    rng = np.random.default_rng(N + k)
    v = np.zeros((6, N), np.float32)
    for b, others in enumerate((k // 2, k, 2 * k, 0)):
        v[b, rng.permutation(N)[:others]] = rng.random(min(others, N)) + 0.5
    v[4] = np.where(rng.random(N) < 0.5, -1.0, -2.0)  # ties at and below the k-th value
    v[5, rng.permutation(N)[: N - N // 8]] = -np.inf
    a = torch.as_tensor(v, device="cuda")
    idx = torch.empty((6, k), dtype=torch.int64, device="cuda")
    val = torch.empty((6, k), dtype=torch.float32, device="cuda")
    bt.boute_select_topk(a, 6, N, k, idx, val)
    for b in range(6):
        want = np.lexsort((np.arange(N), -v[b]))[:k]
        assert np.array_equal(idx[b].cpu().numpy(), want)
        assert np.array_equal(val[b].cpu().numpy(), v[b][want])


def _graph_us(f, calls=20):
    """Device time of a call, from a graph of several."""
    import torch
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        f()
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            for _ in range(calls):
                f()
        return _median_us(g.replay, 9) / calls


def test_topk_of_mostly_zero_scores_and_of_many_small_problems():
    """Scores that are mostly zero, or a thousand problems of a thousand scores, take a
    few times what one problem with distinct scores takes (they took eight times that)."""
    import torch

    from paper_2602_10729_gb300 import boute as bt

    def us(a, k):
        idx = torch.empty((len(a), k), dtype=torch.int64, device="cuda")
        val = torch.empty((len(a), k), dtype=torch.float32, device="cuda")
        return _graph_us(lambda: bt.boute_select_topk(a, len(a), a.shape[1], k, idx, val))

    a = torch.randn((1, 4096), device="cuda")
    one = us(a, 8)
    assert us(torch.where(a > 3.5, a, torch.zeros_like(a)), 8) < 4 * one
    assert us(torch.randn((1000, 1024), device="cuda"), 32) < 4 * one


# ties, NaN and -0 at one block, several, and hundreds of them
@pytest.mark.parametrize("N,k", [(5000, 40), (5000, 32), (5000, 1), (2048, 7), (40, 32),
                                 (700_001, 32), (700_001, 17), (70_000, 33)])
def test_topk_ties_nan_and_negative_zero(N, k):
    import torch

    from paper_2602_10729_gb300 import boute as bt
    rng = np.random.default_rng(11)
    B = 3
    v = np.round(rng.random((B, N)), 2).astype(np.float32)
    v[0, [i for i in (3, 99) if i < N]] = np.nan
    v[1, :50] = -0.0
    v[1, 50:] = -1.0
    v[2, :] = 0.25  # all equal: the first k indices
    v[0, -1] = 2.0  # the maximum in the ragged tail
    a = torch.as_tensor(v, device="cuda")
    idx = torch.empty((B, k), dtype=torch.int64, device="cuda")
    val = torch.empty((B, k), dtype=torch.float32, device="cuda")
    bt.boute_select_topk(a, B, N, k, idx, val)
    for b in range(B):
        oi, ov = oracle.topk(v[b].astype(np.float64), k)
        assert idx[b].cpu().numpy().tolist() == oi.tolist()
    assert idx[2].cpu().numpy().tolist() == list(range(k))


def test_singular_kernel_matrix_reports_not_pd():
    X = np.array([[0.1, 0.2], [0.1, 0.2], [0.5, 0.5], [0.7, 0.1]])
    Y = np.array([[0.0, 1.0], [0.0, 1.0], [1.0, 0.0], [0.5, 0.5]])
    hp = custom(X, Y, np.zeros((10, 2)), noise=0.0)
    g = gpu_pipeline(hp)
    from paper_2602_10729_gb300 import boute as bt
    assert g["status"] == bt.BOUTE_ERR_NOT_PD
    with pytest.raises(oracle.NotPositiveDefinite):
        oracle.gp_fit(X, Y[:, 0], np.full(2, 0.3), 1.0, 0.0)


def test_invalid_arguments_raise():
    import torch

    from paper_2602_10729_gb300 import boute as bt
    with pytest.raises(bt.BouteError) as e:
        bt.boute_gp_create(1, 10, 40, 2)
    assert e.value.code == bt.BOUTE_ERR_INVALID_ARG
    a = torch.zeros((1, 10), device="cuda")
    idx = torch.empty((1, 11), dtype=torch.int64, device="cuda")
    val = torch.empty((1, 11), device="cuda")
    with pytest.raises(bt.BouteError):
        bt.boute_select_topk(a, 1, 10, 11, idx, val)


# Sizes around a warp of points; every point on the front; ties and signed zeros.
@pytest.mark.parametrize("kind", ["random", "antichain", "ties"])
@pytest.mark.parametrize("n,m", [(1, 2), (31, 3), (32, 2), (33, 3), (130, 4), (513, 2), (257, 3),
                                 (2048, 3)])
def test_front_and_boxes_edges(n, m, kind):
    import torch

    from paper_2602_10729_gb300 import boute as bt
    rng = np.random.default_rng(n + m)
    Y = rng.random((n, m)) - 0.5
    if kind == "antichain":
        Y[:, -1] = -Y[:, :-1].sum(1)
    elif kind == "ties":
        Y = np.round(Y * 4) / 4
        Y[Y == 0] = np.where(rng.random((Y == 0).sum()) < 0.5, 0.0, -0.0)
    ref = np.full(m, 0.3)
    mask_o, order = oracle.pareto_front(Y, ref)
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    mask = torch.empty((1, n), dtype=torch.uint8, device="cuda")
    front = torch.zeros((1, n, m), dtype=torch.float64, device="cuda")
    P = torch.empty(1, dtype=torch.int32, device="cuda")
    bt.boute_pareto_front(t(Y[None]), 1, n, m, t(ref[None]), mask, front, P)
    assert mask.cpu().numpy()[0].astype(bool).tolist() == np.asarray(mask_o).astype(bool).tolist()
    F = front.cpu().numpy()[0, :int(P[0])]
    np.testing.assert_array_equal(F, Y[np.asarray(order)])
    if m == 4:
        return
    cap = 2 * n + 2
    lo = torch.empty((1, cap, m), dtype=torch.float32, device="cuda")
    hi = torch.empty_like(lo)
    K = torch.empty(1, dtype=torch.int32, device="cuda")
    bt.boute_box_decompose(front, P, 1, n, m, t(ref[None]), lo, hi, K)
    k = int(K[0])
    assert 1 <= k <= 2 * F.shape[0] + 1
    lo, hi = (a.cpu().numpy()[0, :k].astype(np.float64) for a in (lo, hi))
    for y in rng.random((20, m)) - 0.6:
        got = np.prod(np.maximum(hi - np.maximum(lo, y), 0.0), 1).sum()
        # the corners are rounded to fp32: 2^-24 of at most 1.1 each, m of them per box
        assert got == pytest.approx(oracle.hvi(F, ref, y), abs=k * m * 1.1 * 2.0 ** -23)


# Rows in pairs (four or eight rows apart) and four or eight columns of a half chunk
# per thread: rows and columns at their edges, every coordinate width.
@pytest.mark.parametrize("d,n,N", [(3, 1, 1), (3, 35, 4), (9, 4, 5), (9, 61, 129), (16, 5, 8),
                                   (16, 33, 133), (20, 7, 9), (24, 41, 137), (32, 9, 127),
                                   (7, 34, 70), (11, 66, 130), (13, 40, 131), (14, 3, 200),
                                   (17, 37, 65), (21, 70, 66), (25, 36, 90), (29, 35, 129)])
def test_row_pairs_and_column_groups(d, n, N):
    hp = rand_problem(100 + d + n, n, d, 2, N)
    hp.ls[0] = 0.2 * np.sqrt(d)
    g = gpu_pipeline(hp)
    assert g["status"] == 0
    fp = oracle_fit(hp, 0)
    mean, var = opl.posterior(fp, hp.Xc[0])
    for t in range(2):
        check_mean(g["mean"][0, t], mean[:, t], fp.s2[t])
        check_var(g["var"][0, t], var[:, t], fp.s2[t])


# Tiles of 32: sizes at their edges, batches that take clusters of 16, 8, 4, 2 and 1
# CTAs, and (n > 1024) the factorisation over the whole GPU.
@pytest.mark.parametrize("n,B", [(1, 1), (32, 3), (33, 1), (65, 40), (97, 2), (160, 1), (161, 1), (192, 2), (193, 1), (224, 40), (256, 40), (288, 20),
                                 (321, 12), (511, 6), (1024, 1), (1025, 1),
                                 (1057, 5), (1300, 1), (2048, 1)])
def test_cluster_fit_edges(n, B):
    w = wl.scaled(wl.WORKLOADS[4], N=130, B=B, n=n)
    hp = host_problem(w)
    g = gpu_pipeline(hp)
    assert g["status"] == 0
    for b in sorted({0, B // 2, B - 1}):
        fp = oracle_fit(hp, b)
        mean, var = opl.posterior(fp, hp.Xc[b])
        for t in range(w.m):
            check_mean(g["mean"][b, t], mean[:, t], fp.s2[t])
            check_var(g["var"][b, t], var[:, t], fp.s2[t])


# Three objectives: passes of 32, 64 and 128 samples with a ragged last one, one sample, and
# a count the register path takes (with and without thresholds).
@pytest.mark.parametrize("S", [1, 31, 32, 33, 64, 65, 100, 127, 129, 200, 256, 300])
def test_three_objective_sample_counts(S):
    hp = rand_problem(S, 25, 4, 3, 77, mode="mc", S=S)
    compare(hp)
    cons = np.full((1, 3), 0.4)
    g = gpu_pipeline(hp, cons=cons)
    fp = oracle_fit(hp, 0)
    want = opl.acquisition(fp, g["mean"][0].T.astype(np.float64), g["var"][0].T.astype(np.float64),
                           "mc", hp.eps[0], cons=cons[0])
    check_acq(g["acq"][0], want)


def test_few_samples_of_three_objectives_cost_less_than_many():
    """Sixteen samples in passes of 32, not padded to the 128 of a full pass (with which
    they took longer than 128 samples do on their own path)."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    rng = np.random.default_rng(5)
    N, K = 20000, 21
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a, np.float32), device="cuda")
    lo = rng.uniform(-2, 0, (1, K, 3))
    hi = lo + rng.uniform(0.1, 1, (1, K, 3))
    mean, var = t(rng.standard_normal((1, 3, N))), t(rng.uniform(0.05, 1, (1, 3, N)))
    lo, hi, Kd = t(lo), t(hi), torch.tensor([K], dtype=torch.int32, device="cuda")
    acq = torch.empty((1, N), device="cuda")

    def us(S):
        eps = torch.randn((1, N, 3, S), device="cuda")
        return _graph_us(lambda: bt.boute_acq_mc_hvi(mean, var, 1, N, 3, lo, hi, Kd, K, eps, S,
                                                     3 * S, acq))
    assert us(16) < 0.95 * us(128)


def test_ehvi_over_the_normal_tail():
    """One front point: EHVI's standardised distances from 0 to 12 on both sides,
    relative. The tail factor is good to 3e-7, phi's exponent t^2 / 2 to an ulp of its
    product (t <= 12: 5e-6), sums and products of a few such terms: 2e-5."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    z = np.linspace(-12, 12, 2001)
    N = z.size
    mean = np.stack([z, 0.3 * z], 0)[None].astype(np.float32)
    var = np.ones((1, 2, N), np.float32)
    F, ref = np.array([[0.0, 0.0]]), np.array([1.1, 1.1])
    t = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")
    acq = torch.empty((1, N), dtype=torch.float32, device="cuda")
    bt.boute_acq_ehvi(t(mean), t(var), 1, N, t(F[None]), torch.ones(1, dtype=torch.int32, device="cuda"),
                      1, t(ref[None]), acq)
    want = oracle.ehvi2d(mean[0].T.astype(np.float64), var[0].T.astype(np.float64), F, ref)
    np.testing.assert_allclose(acq.cpu().numpy()[0], want, rtol=2e-5, atol=1e-36)


def test_status_and_new_handles_beside_a_busy_default_stream():
    """Steps on a stream of their own while something else holds the default stream: a
    status is read and cleared without waiting for it, and a new handle's buffers are
    cleared before they are used, not when the default stream comes to it."""
    import time

    import torch

    from paper_2602_10729_gb300 import boute as bt
    hp = rand_problem(21, 70, 5, 2, 300)
    t = lambda a, dt=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")
    X, ls, s2, nz, Xc = t(hp.X), t(hp.ls), t(hp.s2), t(hp.noise), t(hp.Xc, torch.float32)
    Ys = torch.empty_like(t(hp.Y))
    bt.boute_standardize(t(hp.Y), Ys)
    flat = torch.zeros_like(X)  # equal points, no noise: not positive definite
    mean = torch.empty((1, 2, 300), dtype=torch.float32, device="cuda")
    var = torch.empty_like(mean)
    s = torch.cuda.Stream()
    torch.cuda._sleep(1000)
    torch.cuda.synchronize()
    busy = int(1.2e9)  # clocks: half a second or more
    torch.cuda._sleep(busy)
    gp = bt.boute_gp_create(1, 70, 5, 2)
    with torch.cuda.stream(s):
        bt.boute_gp_fit(gp, X, Ys, ls, s2, nz)
    torch.cuda.synchronize()
    bt.boute_gp_posterior(gp, Xc, 300, mean, var)
    torch.cuda.synchronize()
    fp = oracle_fit(hp, 0)
    mo, vo = opl.posterior(fp, hp.Xc[0])
    for k in range(2):
        check_mean(mean[0, k].cpu().numpy(), mo[:, k], fp.s2[k])
        check_var(var[0, k].cpu().numpy(), vo[:, k], fp.s2[k])
    torch.cuda._sleep(busy)
    t0 = time.monotonic()
    with torch.cuda.stream(s):
        bt.boute_gp_fit(gp, flat, Ys, ls, s2, torch.zeros_like(nz))
        assert bt.boute_gp_status(gp) == bt.BOUTE_ERR_NOT_PD
        assert bt.boute_gp_status(gp) == bt.BOUTE_OK
        bt.boute_gp_fit(gp, flat, Ys, ls, s2, torch.zeros_like(nz))
        s.synchronize()
        assert bt.boute_gp_status(gp) == bt.BOUTE_ERR_NOT_PD
    waited = time.monotonic() - t0
    torch.cuda.synchronize()
    assert waited < 0.25
    gp.free()


def _median_us(f, reps=15):
    import torch
    for _ in range(3):
        f()
    out = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        out.append(a.elapsed_time(b) * 1e3)
    return float(np.median(out))


@pytest.mark.parametrize("n,d,seed,b", [(360, 9, 28, 1), (512, 16, 3, 12), (100, 6, 1, 0)])
def test_fit_does_not_depend_on_the_cluster_size(n, d, seed, b):
    """A problem fitted alone (16 CTAs, or a CTA per block row) and 24 times in a batch (one
    to four CTAs): the same sums in the same order, so the same means to the last bit, also
    where the lanes that send a residual round it differently (the first two)."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    from perf import cases
    B = 4 if b < 4 else 32
    p = cases._problem(dict(B=B, n=n, d=d, m=2), seed)
    Xc = cases._candidates(dict(B=B, N=1000, d=d), seed, d)

    def means(k):
        t = lambda a: a[b:b + 1].expand(k, *a.shape[1:]).contiguous()
        Ys = torch.empty_like(t(p["Y"]))
        bt.boute_standardize(t(p["Y"]), Ys)
        gp = bt.boute_gp_create(k, n, d, 2)
        mean = torch.empty((k, 2, 1000), dtype=torch.float32, device="cuda")
        var = torch.empty_like(mean)
        bt.boute_gp_fit(gp, t(p["X"]), Ys, t(p["ls"]), t(p["s2"]), t(p["noise"]))
        bt.boute_gp_posterior(gp, t(Xc), 1000, mean, var)
        assert bt.boute_gp_status(gp) == 0
        gp.free()
        return mean, var

    (mean, var), (mean1, var1) = means(24), means(1)
    assert torch.equal(mean, mean1.expand_as(mean)) and torch.equal(var, var1.expand_as(var))


@pytest.mark.parametrize("n", [256, 512])
def test_fit_of_problem_objectives_beyond_the_held_clusters(n):
    """15 clusters of 8 fit the device, though 16 of them have no more CTAs than it has
    SMs: 16 problem-objectives take smaller clusters at once, not a second wave (which
    costs half as much again or more; the smaller clusters a quarter)."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    us = []
    for B in (7, 8):
        hp = host_problem(wl.scaled(wl.WORKLOADS[4], N=1, B=B, n=n))
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
        args = [t(a) for a in (hp.X, hp.Y, hp.ls, hp.s2, hp.noise)]
        bt.boute_standardize(args[1], args[1])
        gp = bt.boute_gp_create(B, n, hp.w.d, 2)
        us.append(_median_us(lambda: bt.boute_gp_fit(gp, *args)))
        assert bt.boute_gp_status(gp) == 0
        gp.free()
    assert us[1] < 1.35 * us[0], us


def test_fit_of_many_observations_uses_the_whole_gpu():
    """n = 2048 has eight times the products of n = 1024: over all SMs a fit of one
    objective takes less than twice as long, on the 16 SMs of one cluster four times."""
    import torch

    from paper_2602_10729_gb300 import boute as bt
    us = []
    for n in (1024, 2048):
        hp = host_problem(wl.scaled(wl.WORKLOADS[4], N=1, B=1, n=n))
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
        args = [t(hp.X), t(hp.Y[:, :, :1]), t(hp.ls[:, :1]), t(hp.s2[:, :1]), t(hp.noise[:, :1])]
        bt.boute_standardize(args[1], args[1])
        gp = bt.boute_gp_create(1, n, hp.w.d, 1)
        us.append(_median_us(lambda: bt.boute_gp_fit(gp, *args)))
        assert bt.boute_gp_status(gp) == 0
        gp.free()
    assert us[1] < 2.5 * us[0], us
