"""The workloads this library is timed on: whole calls of its public entry points, as a
program that uses it makes them.

A case names an entry point (`entry`), a kind of design (`kind`, with the lengthscale, nugget
and start size of that problem, as in paper_1303_0383_gb300/inputs.py), the design's size N,
the number of predictive locations T, the local design size n, the candidate count ncand, the
criterion and the precision.  Entries:
  host       Design.predict on numpy arrays (resident design, results back on the host)
  device     lagp_predict_dev on CUDA tensors with the caller's buffers and workspace
  knn        lagp_knn_dev: the candidate lists alone
  stagewise  predict_stagewise: designs and local maximum-likelihood lengthscales in stages
  batch      lagp_predict_batch_dev: several resident designs, n and ncand per location
"""
import math

import numpy as np
import torch

from paper_1303_0383_gb300 import lagp

# kind: dimension, lengthscale theta, nugget g, start size n0, box of the design
KINDS = {
    "uniform2d": dict(p=2, theta=0.5, g=1e-6, n0=6, lo=-2.0, hi=2.0),
    "grid2d": dict(p=2, theta=0.5, g=1e-6, n0=6, lo=-2.0, hi=2.0),
    "uniform4d": dict(p=4, theta=0.2, g=1e-6, n0=6, lo=0.0, hi=1.0),
    "smooth8d": dict(p=8, theta=1.0, g=1e-4, n0=8, lo=0.0, hi=1.0),
    "borehole": dict(p=8, theta=0.64, g=1e-6, n0=6, lo=0.0, hi=1.0),
}
# the resident designs of a batch: kind and N
BATCH_DESIGNS = (("uniform2d", 40000), ("uniform4d", 200000), ("smooth8d", 100000))


def _case(name, entry, kind, N, T, n, ncand, method="alc", precision="mixed", stages=1):
    c = dict(entry=entry, kind=kind, N=N, T=T, n=n, ncand=ncand, method=method,
             precision=precision, stages=stages)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one location asked for interactively against a resident design: latency
        _case("query-2d", "host", "uniform2d", 40000, 1, 50, 1000),
        # the small 2-d problem, in the default method and precision of Design.predict
        _case("tiny-2d", "host", "uniform2d", 2000, 100, 50, 200, "alc", "fp64"),
        # one replicate of the borehole experiment at fixed lengthscale
        _case("borehole-alc", "device", "borehole", 4000, 500, 50, 1000),
        # the 2-d benchmark workload, results on the host
        _case("uniform2d-alc", "host", "uniform2d", 40000, 10000, 50, 1000),
        # the same surface with every step in FP64, an odd number of locations
        _case("uniform2d-fp64", "device", "uniform2d", 40000, 4001, 50, 1000, "alc", "fp64"),
        # the large 8-d workload: twice the design size and candidates
        _case("smooth8d-alc", "device", "smooth8d", 100000, 10000, 100, 2000),
        # the MSPE criterion on the same workload
        _case("smooth8d-mspe", "device", "smooth8d", 100000, 2000, 100, 2000, "mspe"),
        # the MSPE criterion in FP64 on the larger borehole replicate
        _case("borehole-mspe-fp64", "device", "borehole", 8000, 1000, 50, 1000, "mspe", "fp64"),
        # nearest neighbours, the comparator, on the dense regular grid
        _case("grid2d-nn", "host", "grid2d", 40401, 10000, 50, 1000, "nn", "fp64"),
        # the two-stage scheme with local lengthscales on the borehole
        _case("borehole-stages", "stagewise", "borehole", 4000, 500, 50, 1000, "alc", "mixed", 2),
        # candidate lists alone, for programs that bring their own selection calls
        _case("smooth8d-knn", "knn", "smooth8d", 100000, 10000, 100, 2000),
        # uneven problems over three resident designs in one call
        _case("batch-uneven", "batch", "all", 200000, 3000, 200, 4000),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    entry = rng.choice(["host", "host", "device", "device", "device", "knn", "stagewise", "batch"])
    if entry == "batch":
        c = _case(None, "batch", "all", 200000, _loguniform(rng, 60, 3000), 200, 4000, "alc",
                  rng.choice(["mixed", "mixed", "fp64"]))
    else:
        kind = rng.choice(sorted(KINDS))
        if kind == "grid2d":
            N = rng.randint(60, 201) ** 2
        elif kind == "borehole":
            N = _loguniform(rng, 2000, 8000)
        else:
            N = _loguniform(rng, 2000, 200000 if kind == "uniform4d" else 100000)
        n = rng.randint(30, 100)
        ncand = min(_loguniform(rng, 200, 2000), N)
        method = rng.choice(["alc", "alc", "alc", "mspe", "nn"])
        precision = rng.choice(["mixed", "fp64"])
        T = _loguniform(rng, 1, 10000)
        if entry == "stagewise":
            T, n = min(T, 2000), min(n, 60)
        c = _case(None, entry, kind, N, T, n, ncand, method, precision,
                  rng.choice([1, 2]) if entry == "stagewise" else 1)
    # no dearer than the largest listed case, from the rates of the criteria and precisions
    slow = {"mixed": 1.0, "fp64": 3.0}[c["precision"]] * {"alc": 1.0, "mspe": 4.0, "nn": 1.0}[c["method"]]
    if entry == "stagewise":
        slow *= 2.0
    big = listed()[5]
    while c["T"] > 1 and slow * work(c)["flops"] > 0.8 * work(big)["flops"]:
        c["T"] = max(1, c["T"] * 2 // 3)
    return c


# ------------------------------------------------------------------ inputs

def _response(kind, X):
    """The response surfaces of the synthetic problems at X (numpy, rows are points)."""
    if kind == "uniform2d":
        return X[:, 0] * np.exp(-X[:, 0] ** 2 - X[:, 1] ** 2)
    if kind == "grid2d":
        def w(x):
            return (np.exp(-(x - 1.0) ** 2) + np.exp(-0.8 * (x + 1.0) ** 2)
                    - 0.05 * np.sin(8.0 * (x + 0.1)))
        return -w(X[:, 0]) * w(X[:, 1])
    if kind == "uniform4d":
        return np.prod(np.sin(3.0 * X), axis=1)
    if kind == "smooth8d":
        j = np.arange(1, X.shape[1] + 1)
        return (np.sum(np.sin(2.0 * math.pi * X) / j, axis=1) + X[:, 0] * X[:, 1] * X[:, 2]
                + np.exp(-np.sum((X - 0.5) ** 2, axis=1)))
    lo = np.array([0.05, 100.0, 63070.0, 63.1, 990.0, 700.0, 1120.0, 9855.0])
    hi = np.array([0.15, 5000.0, 115600.0, 116.0, 1110.0, 820.0, 1680.0, 12045.0])
    rw, r, Tu, Tl, Hu, Hl, L, Kw = (lo + (hi - lo) * X).T
    lg = np.log(r / rw)
    return 2.0 * math.pi * Tu * (Hu - Hl) / (lg * (1.0 + 2.0 * L * Tu / (lg * rw ** 2 * Kw) + Tu / Tl))


def _problem(kind, N, T, seed):
    """Design X, Z and predictive locations XX of one problem (numpy)."""
    k = KINDS[kind]
    p, lo, hi = k["p"], k["lo"], k["hi"]
    rng = np.random.default_rng([seed, N, p])
    if kind == "grid2d":  # a regular grid; the locations are anywhere inside it
        m = math.isqrt(N)
        a = np.linspace(lo, hi, m)
        X = np.stack(np.meshgrid(a, a, indexing="ij"), axis=-1).reshape(-1, 2)
        XX = rng.uniform(lo + 0.03, hi - 0.03, size=(T, p))
    elif kind == "borehole":  # one Latin hypercube of N + T points, split
        strata = np.stack([rng.permutation(N + T) for _ in range(p)], axis=1)
        U = (strata + rng.random((N + T, p))) / (N + T)
        X, XX = U[:N], U[N:]
    else:
        X = rng.uniform(lo, hi, size=(N, p))
        XX = rng.uniform(lo, hi, size=(T, p)) * (0.985 if kind == "uniform2d" else 1.0)
    Z = _response(kind, X)
    if kind == "smooth8d":
        Z = Z + rng.normal(0.0, 1e-2, size=Z.shape)
    return np.ascontiguousarray(X), Z, np.ascontiguousarray(XX)


def _batch_problem(case, seed):
    rng = np.random.default_rng([seed, case["T"]])
    T = case["T"]
    designs = [_problem(kind, N, 0, seed + i)[:2] for i, (kind, N) in enumerate(BATCH_DESIGNS)]
    design_of = rng.integers(0, len(designs), size=T).astype(np.int32)
    # the uneven sizes, evenly spread over their ranges, fall on the locations in any order
    n = rng.permutation(np.linspace(30, case["n"], T).round()).astype(np.int32)
    ncand = rng.permutation(np.linspace(500, case["ncand"], T).round()).astype(np.int32)
    lo = np.array([KINDS[k]["lo"] for k, _ in BATCH_DESIGNS])[design_of, None]
    hi = np.array([KINDS[k]["hi"] for k, _ in BATCH_DESIGNS])[design_of, None]
    XX = lo + (hi - lo) * rng.random((T, 8))
    return designs, design_of, n, ncand, XX


def _cuda(a):
    return torch.as_tensor(a, device="cuda")


def _outputs(T, nidx):
    f = dict(dtype=torch.float64, device="cuda")
    return dict(mean=torch.empty(T, **f), s2=torch.empty(T, **f), var=torch.empty(T, **f),
                idx=torch.empty(nidx, dtype=torch.int32, device="cuda"),
                status=torch.empty(T, dtype=torch.int8, device="cuda"))


def prepare(case, seed):
    c = case
    if c["entry"] == "batch":
        designs, design_of, n, ncand, XX = _batch_problem(c, seed)
        D = [dict(X=_cuda(X), Z=_cuda(Z), n0=KINDS[k]["n0"], theta=KINDS[k]["theta"],
                  g=KINDS[k]["g"]) for (X, Z), (k, _) in zip(designs, BATCH_DESIGNS)]
        ws = lagp.workspace(lagp.lagp_predict_batch_workspace_bytes(D, design_of, n, ncand,
                                                                    c["method"], c["precision"]))
        return dict(case=c, D=D, design_of=design_of, n=n, ncand=ncand, XX=_cuda(XX), ws=ws,
                    out=_outputs(c["T"], int(n.sum())))
    X, Z, XX = _problem(c["kind"], c["N"], c["T"], seed)
    if c["entry"] == "host":
        return dict(case=c, design=lagp.Design(X, Z), XX=XX)
    s = dict(case=c, X=_cuda(X), Z=_cuda(Z), XX=_cuda(XX))
    N, T, p = c["N"], c["T"], X.shape[1]
    if c["entry"] == "knn":
        s["cand"] = torch.empty((T, c["ncand"]), dtype=torch.int32, device="cuda")
        s["ws"] = lagp.workspace(lagp.lagp_knn_workspace_bytes(N, T, c["ncand"]))
    elif c["entry"] == "device":
        s["ws"] = lagp.workspace(lagp.lagp_predict_workspace_bytes(N, T, p, c["n"], c["ncand"],
                                                                   c["method"], c["precision"]))
        s["out"] = _outputs(T, (T, c["n"]))
    return s


def run(state):
    s, c = state, state["case"]
    if c["entry"] == "batch":
        o = s["out"]
        lagp.lagp_predict_batch_dev(s["D"], s["XX"], s["design_of"], s["n"], s["ncand"],
                                    c["method"], c["precision"], o["mean"], o["s2"], o["var"],
                                    o["idx"], o["status"], 0, s["ws"])
        return o
    k = KINDS[c["kind"]]
    if c["entry"] == "host":
        return s["design"].predict(s["XX"], k["n0"], c["n"], c["ncand"], k["theta"], k["g"],
                                   c["method"], c["precision"])
    if c["entry"] == "knn":
        lagp.lagp_knn_dev(s["X"], s["XX"], c["ncand"], s["cand"], s["ws"])
        return dict(cand=s["cand"])
    if c["entry"] == "device":
        o = s["out"]
        lagp.lagp_predict_dev(s["X"], s["Z"], s["XX"], k["n0"], c["n"], c["ncand"], k["theta"],
                              k["g"], c["method"], c["precision"], o["mean"], o["s2"], o["var"],
                              o["idx"], o["status"], s["ws"])
        return o
    return lagp.predict_stagewise(s["X"], s["Z"], s["XX"], k["n0"], c["n"], c["ncand"],
                                  k["theta"], k["g"], c["method"], c["precision"], c["stages"])


# ------------------------------------------------------------------ what a pass cannot do without

def _design_flops(n, M, p, method):
    """Flops of one greedy design and its prediction: every pool candidate at step j costs a
    dot with its row of the Cholesky factor (MSPE: three), its squared distance and
    correlation to the new point (an exponential as 20) and the update of its scalars; NN
    needs the n x n factorisation alone."""
    if method == "nn":
        return n ** 3 / 3.0 + n * n / 2.0 * (3 * p + 21) + 2.0 * n * n
    dots, rest = (1, 7) if method == "alc" else (3, 40)
    j = np.arange(n - 1)
    return M * (3 * p + 21) + float(np.sum((M - j - 1) * (dots * 2.0 * j + 3 * p + 21 + rest)))


def _mle_flops(n, p):
    """One Newton iteration of the local likelihood: factor, inverse, the trace of a product
    of two n x n matrices, and the correlations (an exponential as 20)."""
    return 3.0 * n ** 3 + n * n * (1.5 * p + 20.0)


def work(case):
    c = case
    if c["entry"] == "batch":
        # expected values of the uneven sizes, the three designs in equal parts
        T, nb, Mb = c["T"], (30 + c["n"]) / 2.0, (500 + c["ncand"]) / 2.0
        read = sum(N * 8 * (KINDS[k]["p"] + 1) for k, N in BATCH_DESIGNS)
        fl = 0.0
        for k, N in BATCH_DESIGNS:
            per = np.mean([_design_flops(n, Mb, KINDS[k]["p"], c["method"])
                           for n in range(30, c["n"] + 1, 5)])
            fl += T / 3.0 * (per + N * 3.0 * KINDS[k]["p"])
        return dict(bytes=read + T * (64 + 25 + 4 * nb), flops=fl)
    p, N, T, n, M = KINDS[c["kind"]]["p"], c["N"], c["T"], c["n"], c["ncand"]
    if c["entry"] == "knn":
        return dict(bytes=8.0 * p * (N + T) + 4.0 * T * M, flops=3.0 * p * N * T)
    fl = T * (3.0 * p * N + c["stages"] * _design_flops(n, M, p, c["method"]))
    if c["entry"] == "stagewise":
        fl += T * c["stages"] * 8 * _mle_flops(n, p)
    return dict(bytes=8.0 * (N * (p + 1) + T * p) + T * (25.0 + 4 * n), flops=fl)


# ------------------------------------------------------------------ the same in plain torch, 64 bits

def _nearest(X, x, M):
    """The M nearest rows of X for every row of x, by (squared distance, index)."""
    d2 = torch.zeros(x.shape[0], X.shape[0], dtype=torch.float64, device=X.device)
    for k in range(X.shape[1]):
        t = x[:, k, None] - X[None, :, k]
        d2 += t * t
    return torch.topk(d2, M, dim=1, largest=False, sorted=True).indices


def _sq(a, b):
    return ((a - b) ** 2).sum(-1)


def _greedy(X, Z, x, cand, n0, n, theta, g, method, M=None):
    """Local designs (chunk x n, ranks in cand).  theta: one per location; M: candidates per
    location (the others are kept out), or None for all."""
    B, C = cand.shape
    dev, f64 = X.device, torch.float64
    ar = torch.arange(B, device=dev)
    if method == "nn":
        return torch.arange(n, device=dev).expand(B, n).clone()
    Xc = X[cand]                                    # B x C x p
    th = theta[:, None]
    out = torch.zeros(B, n, dtype=torch.long, device=dev)
    free = torch.ones(B, C, dtype=torch.bool, device=dev)
    if M is not None:
        free &= torch.arange(C, device=dev)[None, :] < M[:, None]
    U = torch.zeros(B, n, C, dtype=f64, device=dev)
    v = torch.full((B, C), 1.0 + g, dtype=f64, device=dev)
    rx = _sq(Xc, x[:, None, :])
    kx = torch.exp(-rx / th)
    cov = kx.clone()
    mspe = method == "mspe"
    if mspe:
        Ud = torch.zeros_like(U)
        kdx = kx * rx / th ** 2
    for j in range(n):
        if j < n0:
            s = torch.full((B,), j, device=dev)
        elif not mspe:
            s = torch.where(free & (v > 0), cov * cov / v, torch.full_like(v, -1.0)).argmax(1)
        else:
            s = J.argmin(1)
        out[:, j] = s
        free[ar, s] = False
        if j == n - 1:
            break
        r2 = _sq(Xc, Xc[ar, s][:, None, :])
        k = torch.exp(-r2 / th)
        sq = v[ar, s].sqrt()[:, None]
        us = U[ar, :j, s]
        u = (k - torch.bmm(us[:, None, :], U[:, :j])[:, 0]) / sq
        U[:, j] = u
        ux = (cov[ar, s][:, None]) / sq
        v = v - u * u
        cov = cov - ux * u
        if mspe:
            kd = k * r2 / th ** 2
            Ud[:, j] = (kd - torch.bmm(us[:, None, :], Ud[:, :j])[:, 0]) / sq
            if j + 1 >= max(n0, 3):
                J = _mspe_scores(X, Z, x, cand, out[:, :j + 1], U[:, :j + 1], Ud[:, :j + 1], v,
                                 cov, theta, g, free)
    return out


def _correlations(X, d, theta, g):
    """K + g I, its first and its second derivative in theta, for the designs d (chunk x n)."""
    P = X[d]
    r2 = _sq(P[:, :, None, :], P[:, None, :, :])
    th = theta[:, None, None]
    K = torch.exp(-r2 / th)
    Kd = K * r2 / th ** 2
    Kdd = Kd * (r2 / th ** 2 - 2.0 / th)
    K = K + g * torch.eye(d.shape[1], dtype=K.dtype, device=K.device)
    return K, Kd, Kdd


def _solve(L, B):
    return torch.linalg.solve_triangular(L, B, upper=False)


def _mspe_scores(X, Z, x, cand, sel, U, Ud, v, cov, theta, g, free):
    """The MSPE criterion of every candidate for the designs sel (ranks)."""
    j = sel.shape[1]
    d = torch.gather(cand, 1, sel)
    K, Kd, Kdd = _correlations(X, d, theta, g)
    L = torch.linalg.cholesky(K)
    Y = Z[d][..., None]
    yt = _solve(L, Y)
    Q = _solve(L, _solve(L, Kd).mT)
    R = _solve(L, _solve(L, Kdd).mT)
    r2x = _sq(X[d], x[:, None, :])
    kx = torch.exp(-r2x / theta[:, None])
    ux = _solve(L, kx[..., None])
    udx = _solve(L, (kx * r2x / theta[:, None] ** 2)[..., None])
    r = Q @ yt
    psi = (yt * yt).sum((1, 2))
    wKdw, nr = (yt * r).sum((1, 2)), (r * r).sum((1, 2))
    yRy = (yt * (R @ yt)).sum((1, 2))
    l2 = (-0.5 * (R.diagonal(dim1=1, dim2=2).sum(1) - (Q * Q).sum((1, 2)))
          + j / (2 * psi) * (yRy - 2 * nr) + j / (2 * psi ** 2) * wKdw ** 2)
    dmux = (udx * yt - ux * r).sum((1, 2))
    vx = 1.0 + g - (ux * ux).sum((1, 2))
    kz = (U * Ud).sum(1)
    pc = (Ud * yt).sum(1)
    q = (U * (Q @ U)).sum(1)
    m = (U * r).sum(1)
    one = psi[:, None]
    V = one * v / (j - 2)
    dmu = pc - m
    dV = (-wKdw[:, None] * v - one * (2 * kz - q)) / (j - 2)
    G = -l2[:, None] + dV ** 2 / (2 * V ** 2) + dmu ** 2 / V
    J = one / (j - 2) * (vx[:, None] - cov ** 2 / v) + (dmux ** 2)[:, None] / G
    return torch.where(free & (v > 0) & torch.isfinite(J), J, torch.full_like(J, math.inf))


def _predictive(X, Z, x, d, theta, g, n=None):
    """mean, s2 and var on the designs d; n: sizes (the first n[t] points count), or None."""
    N = d.shape[1]
    K, _, _ = _correlations(X, d, theta, g)
    k = torch.exp(-_sq(X[d], x[:, None, :]) / theta[:, None])
    Y = Z[d]
    nn = torch.full((d.shape[0],), float(N), dtype=torch.float64, device=X.device)
    if n is not None:
        nn = n.to(torch.float64)
        on = torch.arange(N, device=X.device)[None, :] < n[:, None]
        K = torch.where(on[:, :, None] & on[:, None, :], K,
                        torch.eye(N, dtype=K.dtype, device=K.device))
        k, Y = k * on, Y * on
    L = torch.linalg.cholesky(K)
    ux, yt = _solve(L, k[..., None])[..., 0], _solve(L, Y[..., None])[..., 0]
    pv = (yt * yt).sum(1) * (1.0 + g - (ux * ux).sum(1))
    return (ux * yt).sum(1), pv / nn, pv / (nn - 2)


def _mle(X, Z, d, theta0, g, tmin, tmax, maxit=100, tol=1e-8):
    """The lengthscale of largest likelihood of each design: Newton on its derivative, kept
    inside a bracket that the derivative's sign narrows."""
    n = d.shape[1]
    th = theta0.clamp(tmin, tmax)
    lo, hi = torch.full_like(th, tmin), torch.full_like(th, tmax)
    lo_open, hi_open = (torch.ones_like(th, dtype=torch.bool) for _ in range(2))
    live = torch.ones_like(th, dtype=torch.bool)
    Y = Z[d][..., None]
    for _ in range(maxit):
        if not bool(live.any()):
            break
        K, Kd, Kdd = _correlations(X, d, th, g)
        L = torch.linalg.cholesky(K)
        w = torch.cholesky_solve(Y, L)
        A = torch.cholesky_solve(Kd, L)
        psi = (Y * w).sum((1, 2))
        kw = Kd @ w
        q3 = (w * kw).sum((1, 2))
        q1 = (w * (Kdd @ w)).sum((1, 2))
        q2 = (kw * torch.cholesky_solve(kw, L)).sum((1, 2))
        t1 = A.diagonal(dim1=1, dim2=2).sum(1)
        t3 = torch.cholesky_solve(Kdd, L).diagonal(dim1=1, dim2=2).sum(1)
        t2 = (A * A.mT).sum((1, 2))
        d1 = -0.5 * t1 + n / 2.0 * q3 / psi
        d2 = -0.5 * (t3 - t2) + n / (2 * psi) * (q1 - 2 * q2) + n / (2 * psi ** 2) * q3 ** 2
        up, down = live & (d1 > 0), live & (d1 < 0)
        stop = (d1 == 0) | (up & (th >= tmax)) | (down & (th <= tmin))
        lo, hi = torch.where(up, th, lo), torch.where(down, th, hi)
        lo_open &= ~up
        hi_open &= ~down
        tn = th - d1 / d2
        inside = (d2 < 0) & (tn > lo) & (tn < hi)
        other = torch.where((d1 > 0) & hi_open, hi,
                            torch.where((d1 < 0) & lo_open, lo, 0.5 * (lo + hi)))
        tn = torch.where(inside, tn, other)
        small = (tn - th).abs() <= tol * th
        live &= ~stop
        th = torch.where(live, tn, th)
        live &= ~small
    return th


def exact(case, seed):
    c = case
    dev = "cuda"
    if c["entry"] == "batch":
        designs, design_of, n, ncand, XX = _batch_problem(c, seed)
        res = torch.zeros(3, c["T"], dtype=torch.float64, device=dev)
        for i, ((Xh, Zh), (kind, _)) in enumerate(zip(designs, BATCH_DESIGNS)):
            k = KINDS[kind]
            X, Z = _cuda(Xh), _cuda(Zh)
            mine = np.flatnonzero(design_of == i)
            mine = mine[np.argsort(n[mine], kind="stable")]
            for a in range(0, len(mine), 96):
                t = mine[a:a + 96]
                x = _cuda(np.ascontiguousarray(XX[t, :k["p"]]))
                nt, Mt = _cuda(n[t].astype(np.int64)), _cuda(ncand[t].astype(np.int64))
                th = torch.full((len(t),), k["theta"], dtype=torch.float64, device=dev)
                cand = _nearest(X, x, int(ncand[t].max()))
                sel = _greedy(X, Z, x, cand, k["n0"], int(n[t].max()), th, k["g"], c["method"], Mt)
                got = _predictive(X, Z, x, torch.gather(cand, 1, sel), th, k["g"], nt)
                res[:, _cuda(t)] = torch.stack(got)
        return dict(mean=res[0], s2=res[1], var=res[2], idx=None, status=None)
    k = KINDS[c["kind"]]
    Xh, Zh, XXh = _problem(c["kind"], c["N"], c["T"], seed)
    X, Z, XX = _cuda(Xh), _cuda(Zh), _cuda(XXh)
    g, n, M = k["g"], c["n"], c["ncand"]
    if c["entry"] == "knn":
        B = int(max(1, 4e9 / (24.0 * c["N"])))
        return dict(cand=torch.cat([_nearest(X, XX[a:a + B], M).to(torch.int32)
                                    for a in range(0, c["T"], B)]))
    # chunks whose factor rows and distances take at most about 4 GB
    B = int(max(1, min(1000, 4e9 / (8.0 * (n * M * (4 if c["method"] == "mspe" else 1) + 3 * c["N"])))))
    parts = []
    for a in range(0, c["T"], B):
        x = XX[a:a + B]
        th = torch.full((x.shape[0],), k["theta"], dtype=torch.float64, device=dev)
        cand = _nearest(X, x, M)
        d = torch.gather(cand, 1, _greedy(X, Z, x, cand, k["n0"], n, th, g, c["method"]))
        if c["entry"] == "stagewise":
            lim = (k["theta"] / 100.0, k["theta"] * 100.0)
            th = _mle(X, Z, d, th, g, *lim)
            for _ in range(c["stages"] - 1):
                d = torch.gather(cand, 1, _greedy(X, Z, x, cand, k["n0"], n, th, g, c["method"]))
                th = _mle(X, Z, d, th, g, *lim)
        parts.append(_predictive(X, Z, x, d, th, g) + (th,))
    mean, s2, var, theta = (torch.cat(v) for v in zip(*parts))
    out = dict(mean=mean, s2=s2, var=var, idx=None, status=None)
    if c["entry"] == "stagewise":
        out.update(theta=theta, iters=None, mle_status=None)
    if c["entry"] == "host":
        out = {key: v if v is None else v.cpu().numpy() for key, v in out.items()}
    return out
