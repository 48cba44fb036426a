"""Workloads of the library's public entry points, from the smallest calls to the full-size one.

A case names a recipe (how inputs, partition and outputs are drawn), the sizes and
the call:

  recipe "line"      d-dimensional inputs in [0, 1]^d sorted by the first coordinate
                     (configuration C1, and its ragged variants);
  recipe "clusters"  Gaussian inputs in clusters ordered along their principal axis
                     (C2: equal blocks; C3: uneven ones, d = 21);
  recipe "cube"      inputs in [0, 1]^8 in Morton order (C4, C5).

  call "fit_predict" lma_fit_predict, "fit_then_predict" lma_fit + lma_predict,
  "predict" lma_predict on a model kept in the state, "predict_cov" the same with
  the covariance of every test block, "grad" lma_loglik_grad.

Inputs are drawn on the GPU from the seed; outputs are a random-Fourier-feature
sample of the SE process plus noise.  The launch-shape tuner's timing is off, so
that every process takes the same launch shapes and with them the same order of
the sums (a program that wants the same bits from run to run does the same).
"""
import math

import numpy as np
import torch

import paper_1411_4510_gb300 as L

RFF = 1024  # features of the random-Fourier-feature sample


def listed():
    return [
        # the smallest ordinary problem (configuration C1), handed over as numpy arrays: latency of one whole call
        dict(name="c1_fit_predict_host", call="fit_predict", recipe="line", N=2000, d=2, M=16, s=64, B=1, U=500,
             ell=0.2, noise=0.1, precision="mixed", host=True),
        # the same problem in the FP64 form, the one asked for where FP32 windows are not good enough
        dict(name="c1_fit_predict_fp64", call="fit_predict", recipe="line", N=2000, d=2, M=16, s=64, B=1, U=500,
             ell=0.2, noise=0.1, precision="fp64", host=False),
        # odd sizes everywhere: blocks of uneven size, a longer blanket, |S| not a multiple of anything, fit and
        # prediction as two calls
        dict(name="ragged_fit_then_predict", call="fit_then_predict", recipe="line", N=2977, d=3, M=23, s=77, B=3, U=391,
             ell=0.4, noise=0.1, precision="mixed", host=False, uneven=True),
        # AIMPEAK's shape (configuration C2)
        dict(name="c2_fit_predict", call="fit_predict", recipe="clusters", N=40960, d=5, M=64, s=512, B=1, U=4096,
             ell=1.0, noise=0.05, precision="mixed", host=False),
        # SARCOS's shape (configuration C3): d = 21, uneven clusters, B = 2
        dict(name="c3_fit_predict", call="fit_predict", recipe="clusters", N=49152, d=21, M=96, s=1024, B=2, U=8192,
             ell=3.0, noise=0.1, precision="mixed", host=False, uneven=True),
        # EMSLP's scale (configuration C4), the benchmark's workload
        dict(name="c4_fit_predict", call="fit_predict", recipe="cube", N=2_000_000, d=8, M=2000, s=2048, B=1, U=100_000,
             ell=0.3, noise=0.1, precision="mixed", host=False),
        # serving: a few new points against a fitted C2 model
        dict(name="c2_predict_64", call="predict", recipe="clusters", N=40960, d=5, M=64, s=512, B=1, U=64,
             ell=1.0, noise=0.05, precision="mixed", host=False),
        # a large batch of predictions against a fitted model of C5's size
        dict(name="c5_predict_batch", call="predict", recipe="cube", N=65536, d=8, M=128, s=1024, B=1, U=32768,
             ell=0.3, noise=0.1, precision="mixed", host=False),
        # predictions with the joint covariance of each test block
        dict(name="c2_predict_cov", call="predict_cov", recipe="clusters", N=40960, d=5, M=64, s=512, B=1, U=4096,
             ell=1.0, noise=0.05, precision="mixed", host=False),
        # one step of hyperparameter learning on a small problem (the sizes of the learning tests)
        dict(name="learn_grad", call="grad", recipe="clusters", N=3200, d=5, M=16, s=100, B=1, U=0,
             ell=1.0, noise=0.05, precision="mixed", host=False),
        # one step of hyperparameter learning at configuration C5
        dict(name="c5_grad", call="grad", recipe="cube", N=65536, d=8, M=128, s=1024, B=2, U=0,
             ell=0.3, noise=0.1, precision="mixed", host=False),
        # the same step in the FP64 form on a few thousand points
        dict(name="fp64_grad", call="grad", recipe="clusters", N=5000, d=5, M=20, s=200, B=1, U=0,
             ell=1.0, noise=0.05, precision="fp64", host=False),
    ]


def _loguni(rng, a, b):
    return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))


def draw(rng):
    kind = rng.choice(["line", "line64", "ragged", "clusters", "clusters", "cube", "cube", "predict", "cov", "grad", "grad",
                       "grad64"])
    c = dict(precision="mixed", host=False, uneven=rng.random() < 0.5)
    if kind in ("line", "line64", "ragged"):
        N = _loguni(rng, 500, 8000)
        c.update(call="fit_then_predict" if kind == "ragged" else "fit_predict", recipe="line", N=N, d=rng.randint(2, 4),
                 M=max(4, N // rng.randint(60, 200)), s=rng.randint(16, 128), B=rng.randint(0, 3), U=_loguni(rng, 20, 2000),
                 ell=0.3, noise=0.1, host=kind == "line")
        if kind == "line64":
            c.update(precision="fp64", N=min(N, 4000), M=max(4, min(N, 4000) // rng.randint(100, 200)), B=rng.randint(0, 1))
    elif kind == "clusters":
        N, d = _loguni(rng, 6000, 50000), rng.choice([5, 21])
        c.update(call="fit_predict", recipe="clusters", N=N, d=d, M=max(8, N // rng.randint(400, 700)),
                 s=rng.randint(100, 1024), B=rng.randint(1, 2), U=_loguni(rng, 100, 8192), ell=1.0 if d == 5 else 3.0,
                 noise=0.05 if d == 5 else 0.1)
    elif kind == "cube":
        N = _loguni(rng, 16000, 1_000_000)
        c.update(call="fit_predict", recipe="cube", N=N, d=8, M=N // rng.randint(500, 1000), s=_loguni(rng, 256, 2048),
                 B=rng.randint(1, 2) if N < 100_000 else 1, U=_loguni(rng, 500, 50_000), ell=0.3, noise=0.1)
    elif kind in ("predict", "cov"):
        N = _loguni(rng, 8000, 65000)
        c.update(call="predict" if kind == "predict" else "predict_cov", recipe="cube" if rng.random() < 0.5 else "clusters",
                 N=N, M=N // rng.randint(400, 800), s=rng.randint(128, 1024), B=1,
                 U=_loguni(rng, 16, 32768 if kind == "predict" else 6000))
        c.update(dict(d=8, ell=0.3, noise=0.1) if c["recipe"] == "cube" else dict(d=5, ell=1.0, noise=0.05))
    elif kind == "grad":
        N = _loguni(rng, 2000, 65000)
        c.update(call="grad", recipe="cube" if N > 20000 else "clusters", N=N, M=max(4, N // rng.randint(200, 512)),
                 s=rng.randint(64, 256) if N < 8000 else rng.randint(256, 1024), B=rng.randint(1, 2), U=0)
        c.update(dict(d=8, ell=0.3, noise=0.1) if c["recipe"] == "cube" else dict(d=5, ell=1.0, noise=0.05))
    else:
        N = _loguni(rng, 1000, 6000)
        c.update(call="grad", recipe="clusters", N=N, d=5, M=max(4, N // rng.randint(150, 300)), s=rng.randint(40, 200),
                 B=rng.randint(0, 1), U=0, ell=1.0, noise=0.05, precision="fp64")
    return c


# ---- inputs ------------------------------------------------------------------

def _sizes(case, n):
    """Block sizes: equal (the first ones larger by one), or uneven between about half and one and a half of that."""
    M = case["M"]
    if not case.get("uneven"):
        return [n // M + (1 if m < n % M else 0) for m in range(M)]
    w = [1.0 + 0.5 * math.sin(1.7 * m + 0.4) for m in range(M)]
    cut = [round(n * t) for t in np.cumsum([0.0] + w) / sum(w)]
    return [b - a for a, b in zip(cut, cut[1:])]


def _morton(x, bits=7):
    q = (x * (1 << bits)).long().clamp_(0, (1 << bits) - 1)
    key = torch.zeros(x.shape[0], dtype=torch.int64, device=x.device)
    for b in range(bits - 1, -1, -1):
        for j in range(x.shape[1]):
            key = (key << 1) | ((q[:, j] >> b) & 1)
    return key


def _cluster_keys(x, xu, M, g):
    """Order of the clusters of x along their principal axis, then each point's own projection: (keys of x, keys of xu)."""
    c = x[torch.randperm(x.shape[0], generator=g, device=x.device)[:M]]
    near = lambda p: torch.cat([(a[:, None, :] - c[None]).square().sum(-1).argmin(1) for a in p.split(4096)])  # noqa: E731
    for _ in range(4):
        hot = torch.nn.functional.one_hot(near(x), M).double()
        n = hot.sum(0)[:, None]
        c = torch.where(n > 0, (hot.T @ x) / n.clamp(min=1), c)
    axis = torch.linalg.eigh((c - c.mean(0)).T @ (c - c.mean(0)))[1][:, -1]
    axis = axis * axis[axis.abs().argmax()].sign()
    rank = torch.empty(M, dtype=torch.float64, device=x.device)
    rank[(c @ axis).argsort(stable=True)] = torch.arange(M, dtype=torch.float64, device=x.device)
    key = lambda p: rank[near(p)] + torch.sigmoid(p @ axis) * 0.999  # noqa: E731
    return key(x), (key(xu) if xu.shape[0] else xu[:, 0])


def _inputs(case, seed):
    """X, y, S, XU on the GPU (float64), block_ptr and test_block_ptr (numpy)."""
    g = torch.Generator(device="cuda").manual_seed(1411 + seed)
    N, U, d, M = case["N"], case["U"], case["d"], case["M"]
    new = torch.randn if case["recipe"] == "clusters" else torch.rand
    X = new(N, d, generator=g, device="cuda", dtype=torch.float64)
    XU = new(U, d, generator=g, device="cuda", dtype=torch.float64)
    if case["recipe"] == "line":
        kx, ku = X[:, 0], XU[:, 0]
    elif case["recipe"] == "cube":
        kx, ku = _morton(X), _morton(XU)
    else:
        kx, ku = _cluster_keys(X, XU, M, g)
    kx, order = kx.sort(stable=True)
    X = X[order].contiguous()
    ptr = np.concatenate([[0], np.cumsum(_sizes(case, N))]).astype(np.int64)
    ku, order = ku.sort(stable=True)
    XU = XU[order].contiguous()
    inner = torch.searchsorted(ku.contiguous(), kx[torch.from_numpy(ptr[1:-1]).cuda()].contiguous()).cpu().numpy()
    tptr = np.concatenate([[0], inner, [U]]).astype(np.int64)
    if case["call"] == "predict_cov":  # the covariance blocks' sizes follow the counts: the same for every seed
        tptr = np.arange(M + 1, dtype=np.int64) * U // M
    W = torch.randn(RFF, d, generator=g, device="cuda", dtype=torch.float64) / case["ell"]
    c = torch.rand(RFF, generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
    a = torch.randn(RFF, generator=g, device="cuda", dtype=torch.float64) * math.sqrt(2.0 / RFF)
    y = torch.cat([torch.cos(torch.addmm(c, x, W.T)) @ a for x in X.split(65536)])
    y += case["noise"] * torch.randn(N, generator=g, device="cuda", dtype=torch.float64)
    S = X[torch.randperm(N, generator=g, device="cuda")[:case["s"]].sort()[0]].contiguous()
    return X, y, S, XU, ptr, tptr


def prepare(case, seed):
    L.lma_autotune(False)
    X, y, S, XU, ptr, tptr = _inputs(case, seed)
    if case["host"]:
        X, y, S, XU = (t.cpu().numpy() for t in (X, y, S, XU))
    problem = dict(X=X, y=y, block_ptr=ptr, S=S, B=case["B"], log_ell=np.full(case["d"], math.log(case["ell"])),
                   log_sigma_s=0.0, log_sigma_n=math.log(case["noise"]),
                   precision=L.FP64 if case["precision"] == "fp64" else L.MIXED)
    state = dict(call=case["call"], problem=problem, XU=XU, tptr=tptr)
    if case["call"] in ("predict", "predict_cov"):
        state["model"] = L.lma_fit(**problem)
    return state


def run(state):
    call = state["call"]
    if call == "fit_predict":
        return L.lma_fit_predict(XU=state["XU"], test_block_ptr=state["tptr"], **state["problem"])
    if call == "fit_then_predict":
        model = L.lma_fit(**state["problem"])
        mean, var = L.lma_predict(model, state["XU"], state["tptr"], noisy=False)
        return mean, var, L.lma_model_loglik(model)
    if call == "predict":
        return L.lma_predict(state["model"], state["XU"], state["tptr"])
    if call == "predict_cov":
        mean, var, covs = L.lma_predict_cov(state["model"], state["XU"], state["tptr"])
        return mean, var, torch.cat([c.reshape(-1) for c in covs if c is not None])
    return L.lma_loglik_grad(**state["problem"])


def _test_counts(case):
    """Test points per block as their distribution has them (about even)."""
    return [case["U"] / case["M"]] * case["M"]


def work(case):
    N, d, M, s, B, U = (case[k] for k in ("N", "d", "M", "s", "B", "U"))
    sizes = _sizes(case, N)
    win = [sum(sizes[m:m + B + 1]) for m in range(M)]
    fit = N * s * s + 2 * s ** 3 / 3 + sum(s * n * n + n ** 3 / 3 + n * n * (s + 1) + b * s * s for n, b in zip(win, sizes))
    pred = 2 * U * s * s
    for m, u in enumerate(_test_counts(case)):
        for w in range(max(0, m - B), m + 1):
            n, kept = win[w], win[w] if w == m else sizes[w]
            pred += u * (2 * n * s + n * n + 2 * kept * s)
    inputs = 8 * (N * d + N + s * d)
    call = case["call"]
    if call in ("fit_predict", "fit_then_predict"):
        return dict(bytes=inputs + 8 * U * d + 16 * U, flops=fit + pred)
    if call == "predict":
        # every window factor that a test block needs is read once, and so are its solved rows [r; V]
        factors = sum(4 * (n * n // 2 + (s + 1) * n) for n in win) * min(1.0, U * (B + 1) / M)
        return dict(bytes=8 * U * d + 16 * U + factors, flops=pred)
    if call == "predict_cov":
        cov = sum(u * u for u in _test_counts(case))
        factors = sum(4 * (n * n // 2 + (s + 1) * n) for n in win)
        return dict(bytes=8 * U * d + 16 * U + 8 * cov + factors, flops=pred + cov * (4 * s + 2 * (B + 1) * sizes[0]))
    adj = sum(2 * (2 * (s + 1) + b) * n * n + 2 * s * n * n + s * s * n for n, b in zip(win, sizes)) + 4 * N * s * s + 4 * s ** 3
    return dict(bytes=inputs, flops=fit + adj)


# ---- the same values in 64 bits, by plain torch --------------------------------

def _se(a, b, ss2=1.0):
    d2 = a.square().sum(1)[:, None] + b.square().sum(1)[None] - 2.0 * (a @ b.T)
    return ss2 * torch.exp(-0.5 * d2.clamp(min=0))


def _fit64(X, y, S, ptr, B, log_ell, log_ss, log_sn, jitter=1e-6):
    """Windows (blanket first), their solved rows, beta and L_C: Definitions 1 and 2 in whitened support coordinates."""
    ss2, sn2 = torch.exp(2 * log_ss), torch.exp(2 * log_sn)
    xs, ss = X * torch.exp(-log_ell), S * torch.exp(-log_ell)
    s, M = S.shape[0], len(ptr) - 1
    eye = torch.eye(s, dtype=torch.float64, device=X.device)
    Lss = torch.linalg.cholesky(_se(ss, ss, ss2) + jitter * eye)
    V = torch.linalg.solve_triangular(Lss, _se(ss, xs, ss2), upper=False).T
    wins, G, logdet = [], 0.0, 0.0
    for m in range(M):
        last = min(m + B, M - 1)
        rows = torch.arange(int(ptr[last + 1]) - 1, int(ptr[m]) - 1, -1, device=X.device)
        nB = int(ptr[last + 1] - ptr[m + 1])
        R = _se(xs[rows], xs[rows], ss2) - V[rows] @ V[rows].T + sn2 * torch.eye(len(rows), dtype=torch.float64, device=X.device)
        Lw = torch.linalg.cholesky(R)
        E = torch.linalg.solve_triangular(Lw, torch.cat([y[rows, None], V[rows]], 1), upper=False)
        Z = E[nB:]
        G = G + Z.T @ Z
        logdet = logdet + 2 * torch.log(torch.diagonal(Lw)[nB:]).sum()
        wins.append((rows, nB, Lw, E))
    C = eye + G[1:, 1:]
    Lc = torch.linalg.cholesky(C)
    w = torch.linalg.solve_triangular(Lc, G[1:, :1], upper=False)
    beta = torch.linalg.solve_triangular(Lc.T, w, upper=True)[:, 0]
    ll = (-0.5 * (G[0, 0] - w.square().sum()) - 0.5 * (logdet + 2 * torch.log(torch.diagonal(Lc)).sum())
          - 0.5 * X.shape[0] * math.log(2 * math.pi))
    return dict(xs=xs, ss=ss, V=V, Lss=Lss, Lc=Lc, beta=beta, wins=wins, ll=ll, ss2=ss2, sn2=sn2)


def _predict64(f, XU, tptr, B, log_ell, noisy, cov):
    xu = XU * torch.exp(-log_ell)
    Vu = torch.linalg.solve_triangular(f["Lss"], _se(f["ss"], xu, f["ss2"]), upper=False).T
    prior = f["ss2"] + (f["sn2"] if noisy else 0.0)
    mean, var, covs = [], [], []
    for n in range(len(tptr) - 1):
        u = slice(int(tptr[n]), int(tptr[n + 1]))
        if u.start == u.stop:
            continue
        res, h = Vu[u] @ f["beta"], -Vu[u]
        k = _se(xu[u], xu[u], f["ss2"]) - Vu[u] @ Vu[u].T
        for m in range(max(0, n - B), n + 1):
            rows, nB, Lw, E = f["wins"][m]
            P = torch.linalg.solve_triangular(Lw, _se(f["xs"][rows], xu[u], f["ss2"]) - f["V"][rows] @ Vu[u].T, upper=False)
            kept = slice(0 if m == n else nB, None)
            P, Em = P[kept], E[kept]
            res = res + P.T @ (Em[:, 0] - Em[:, 1:] @ f["beta"])
            h = h + P.T @ Em[:, 1:]
            k = k - P.T @ P
        hc = torch.linalg.solve_triangular(f["Lc"], h.T, upper=False)
        k = k + hc.T @ hc
        k.diagonal().add_(prior - f["ss2"])
        mean.append(res)
        var.append(torch.diagonal(k).clone())
        covs.append(k.reshape(-1))
    out = [torch.cat(mean), torch.cat(var)]
    return out + [torch.cat(covs)] if cov else out


def exact(case, seed):
    if case["N"] * case["s"] ** 2 > 3e11:
        return None  # minutes in 64 bits
    X, y, S, XU, ptr, tptr = _inputs(case, seed)
    hyper = [torch.full((case["d"],), math.log(case["ell"]), dtype=torch.float64, device="cuda"),
             torch.zeros((), dtype=torch.float64, device="cuda"),
             torch.tensor(math.log(case["noise"]), dtype=torch.float64, device="cuda")]
    if case["call"] == "grad":
        hyper = [t.requires_grad_() for t in hyper]
        ll = _fit64(X, y, S, ptr, case["B"], *hyper)["ll"]
        g = torch.autograd.grad(ll, hyper)
        return float(ll), torch.cat([t.reshape(-1) for t in g]).cpu().numpy()
    noisy = case["call"] != "fit_then_predict"
    f = _fit64(X, y, S, ptr, case["B"], *hyper)
    out = _predict64(f, XU, tptr, case["B"], hyper[0], noisy, case["call"] == "predict_cov")
    if case["host"]:
        out = [t.cpu().numpy() for t in out]
    return out + [float(f["ll"])] if case["call"] == "fit_then_predict" else out
