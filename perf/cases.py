"""What a user of this library has it do, as cases that can be timed.

A case is one call of a public entry point on one set of sizes.  Every fit runs
a fixed budget of iterations per component (`iters`: max_iter with a tolerance
no iteration reaches), so the work of a case follows from its sizes and two
implementations that round differently stop at the same iteration.  Inputs are
the synthetic families of this repository's tests and benchmark, drawn on the
GPU from the seed: planted spectra (s_i = s0 ratio^i plus noise), uniform
matrices (the paper's own), and duplicated columns.
"""
import math

import numpy as np
import torch

import paper_0811_1081_gb300 as gp

TOL = 1e-14  # never reached: the iteration budget ends every component


def listed():
    return [
        # A small table (the repository's 500 x 200 workload): a fit of well under a
        # millisecond per component, where launches and device-side latency count.
        dict(name="small_gs", path="fit", data="planted", M=500, N=200, K=10, iters=15, algo="gs", dtype="f32",
             layout="col", center=0, ratio=0.85),
        # An ordinary table as a C-contiguous tensor of odd sizes, columns centred by the
        # library, residual wanted: the everyday NIPALS call.
        dict(name="ragged_nipals", path="fit", data="planted", M=1003, N=517, K=12, iters=20, algo="nipals",
             dtype="f32", layout="row", center=1, ratio=0.9, want_R=True),
        # A tall, narrow table: many observations of few attributes.
        dict(name="tall_gs", path="fit", data="planted", M=60001, N=130, K=8, iters=15, algo="gs", dtype="f32",
             layout="row", center=1, ratio=0.85),
        # The benchmark workload: 50 components of a 10000 x 2000 matrix by GS-PCA.
        dict(name="headline_gs", path="fit", data="planted", M=10000, N=2000, K=50, iters=25, algo="gs",
             dtype="f32", layout="col", center=0, ratio=0.95),
        # The same matrix by the paper's other algorithm, fewer components.
        dict(name="headline_nipals", path="fit", data="planted", M=10000, N=2000, K=20, iters=25, algo="nipals",
             dtype="f32", layout="col", center=0, ratio=0.95),
        # The residual stored in bfloat16.
        dict(name="bf16_gs", path="fit", data="planted", M=10000, N=2000, K=8, iters=25, algo="gs",
             dtype="bf16", layout="col", center=0, ratio=0.85),
        # The paper's largest matrix (U[0,1), 450 MB): R streams from HBM every pass.
        dict(name="stream_gs", path="fit", data="uniform", M=15000, N=7500, K=6, iters=12, algo="gs", dtype="f32",
             layout="col", center=0, ratio=0.0),
        # Many components (more than 128) of a matrix with nearly duplicated columns.
        dict(name="many_gs", path="fit", data="collinear", M=4096, N=1024, K=160, iters=6, algo="gs", dtype="f32",
             layout="col", center=0, ratio=0.0),
        # The paper's own precision: everything in IEEE double.
        dict(name="f64_gs", path="f64", data="planted", M=4000, N=1500, K=10, iters=20, algo="gs", dtype="f64",
             layout="col", center=0, ratio=0.85),
        # Block power iteration, 16 components at a time.
        dict(name="block", path="block", data="planted", M=10000, N=2000, K=32, iters=6, block=16, dtype="f32",
             layout="col", center=0, ratio=0.9),
        # 128 independent problems of mixed sizes in one launch.
        dict(name="batch_gs", path="batch", data="planted", count=128, m_lo=256, m_hi=8192, n_lo=64, n_hi=1024,
             K=12, iters=12, algo="gs", dtype="f32", ratio=0.85),
        # From and to host memory: the call a program makes whose data is not on the GPU.
        dict(name="host_gs", path="host", data="planted", M=5000, N=1000, K=10, iters=20, algo="gs", dtype="f32",
             layout="row", center=1, ratio=0.85),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["fit"] * 6 + ["f64", "block", "batch", "host"])
    if path == "batch":
        m_lo, n_lo = _log(rng, 64, 512), _log(rng, 32, 96)
        return dict(path=path, data="planted", count=_log(rng, 8, 128), m_lo=m_lo, m_hi=_log(rng, 1000, 8192),
                    n_lo=n_lo, n_hi=_log(rng, 200, 1024), K=rng.randint(4, 12), iters=rng.randint(8, 12),
                    algo=rng.choice(["gs", "gs", "nipals"]), dtype="f32", ratio=0.85)
    c = dict(path=path, data="planted", M=_log(rng, 300, 15000), N=_log(rng, 60, 7500), K=_log(rng, 3, 50),
             iters=rng.randint(10, 25), algo=rng.choice(["gs", "gs", "nipals"]), dtype="f32",
             layout=rng.choice(["col", "row"]), center=rng.choice([0, 0, 1]), ratio=0.9)
    if path == "fit":
        c["dtype"] = rng.choice(["f32", "f32", "f32", "bf16"])
        kind = rng.randint(0, 7)
        if kind == 0:  # tall and narrow
            c["M"], c["N"] = _log(rng, 20000, 100000), _log(rng, 40, 400)
        elif kind == 1 and c["dtype"] == "f32":  # many components
            c.update(data="collinear", M=_log(rng, 1500, 4096), N=2 * _log(rng, 300, 512), K=_log(rng, 70, 160),
                     iters=rng.randint(3, 6), algo="gs")
        elif kind == 2:  # the paper's shape, large
            c["N"] = _log(rng, 2500, 7500)
            c.update(data="uniform", M=2 * c["N"], K=rng.randint(2, 6), iters=rng.randint(6, 12))
    if c["dtype"] == "bf16":  # larger matrices and few, well iterated components: what 8 bits of significand resolve
        c.update(algo="gs", M=max(c["M"], 2000), N=max(c["N"], 500), K=min(c["K"], 6), iters=25)
    if c["algo"] == "nipals":
        c.update(K=min(c["K"], 24), iters=max(c["iters"], 12))
    if path == "f64":
        c["M"], c["N"], c["K"] = _log(rng, 300, 5000), _log(rng, 60, 1600), _log(rng, 3, 10)
        c["dtype"] = "f64"
    if path == "block":
        del c["algo"]
        c.update(N=_log(rng, 200, 3000), K=rng.randint(8, 32), block=rng.choice([4, 8, 11, 16]), iters=rng.randint(3, 6))
    c["K"] = min(c["K"], c["N"] // 4, c["M"] // 4)
    c["ratio"] = 0.85 if c["K"] <= 24 else 0.9
    # no more work than the largest listed cases: 1250 passes over 80 MB
    while c["path"] in ("fit", "host") and c["K"] * (c["iters"] + 1) * (c["M"] * c["N"] + 2e6) > 2.6e10:
        c["K"], c["iters"] = max(2, c["K"] * 3 // 4), max(4, c["iters"] * 9 // 10)
    return c


def _gen(seed, dev):
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    return g


def _planted(g, M, N, K, ratio, dev):
    """A random matrix with the planted singular values 100 ratio^i, and noise."""
    r = min(M, N, 2 * K + 16)
    s = 100.0 * ratio ** torch.arange(r, device=dev, dtype=torch.float64)

    def basis(rows):  # orthonormal columns: a Gaussian matrix times the inverse of its Gram matrix's factor, twice
        A = torch.randn(rows, r, generator=g, device=dev, dtype=torch.float64)
        for _ in range(2):
            A = torch.linalg.solve_triangular(torch.linalg.cholesky(A.t() @ A).t(), A, upper=True, left=False)
        return A

    X = ((basis(M) * s) @ basis(N).t()).float()
    return X.add_(torch.randn(M, N, generator=g, device=dev), alpha=0.01)


def _shapes(case):
    """The sizes of a batch's problems, spread over the logarithms of the ranges (the same for every seed)."""
    g = np.random.RandomState(17 + case["count"])
    u = g.uniform(size=(2, case["count"]))
    f = lambda a, lo, hi: int(round(lo * (hi / lo) ** a))  # noqa: E731
    return [(f(a, case["m_lo"], case["m_hi"]), f(b, case["n_lo"], case["n_hi"])) for a, b in u.T]


def _matrix(case, seed):
    """The input of a single fit, M x N on the GPU (C-contiguous), in the type of the call."""
    dev = "cuda"
    g = _gen(seed, dev)
    M, N = case["M"], case["N"]
    if case["data"] == "uniform":
        X = torch.rand(M, N, generator=g, device=dev)
    elif case["data"] == "collinear":
        B = torch.randn(M, N // 2, generator=g, device=dev)
        E = torch.randn(M, N // 2, generator=g, device=dev)
        X = torch.cat([B, B + 1e-3 * E], dim=1)
    else:
        X = _planted(g, M, N, case["K"], case["ratio"], dev)
    return X.double() if case["dtype"] == "f64" else X


def _batch_matrices(case, seed):
    g = _gen(seed, "cuda")
    return [_planted(g, M, N, case["K"], case["ratio"], "cuda").t().contiguous().t() for M, N in _shapes(case)]


def prepare(case, seed):
    s = {"case": case}
    if case["path"] == "batch":
        Xs = _batch_matrices(case, seed)
        s["batch"] = gp.Batch([dict(X=X, K=min(case["K"], *X.shape)) for X in Xs])
        s["h"] = gp.Handle(max(X.shape[0] for X in Xs), max(X.shape[1] for X in Xs), case["K"], dtype=case["dtype"])
        return s
    X = _matrix(case, seed)
    if case["layout"] == "col":
        X = X.t().contiguous().t()
    s["h"] = gp.Handle(case["M"], case["N"], case["K"], dtype=case["dtype"])
    if case["path"] == "host":
        H = torch.empty(X.shape if case["layout"] == "row" else X.t().shape, pin_memory=True)
        H.copy_(X if case["layout"] == "row" else X.t())
        X = H if case["layout"] == "row" else H.t()
    s["X"] = X
    return s


def run(s):
    c, h = s["case"], s["h"]
    kw = dict(tol=TOL, max_iter=c["iters"])
    if c["path"] == "batch":
        gp.gspca_fit_batched(h.h, s["batch"], algo=c["algo"], **kw)
        rs = s["batch"].results
        return dict(T=torch.cat([r.T.t().reshape(-1) for r in rs]), P=torch.cat([r.P.t().reshape(-1) for r in rs]),
                    lam=torch.cat([r.lam for r in rs]), iters=torch.cat([r.iters for r in rs]))
    X, K = s["X"], c["K"]
    kw.update(center=c["center"])
    if c["path"] == "f64":
        r = h.fit64(X, K, algo=c["algo"], **kw)
    elif c["path"] == "block":
        r = h.fit_block(X, K, block=c["block"], **kw)
    elif c["path"] == "host":
        r = h.fit_host(X, K, algo=c["algo"], **kw)
    else:
        r = h.fit(X, K, algo=c["algo"], want_R=c.get("want_R", False), **kw)
    out = dict(T=r.T, P=r.P, lam=r.lam, iters=r.iters)
    if r.R is not None:
        out["R"] = r.R
    return out


def _work_one(M, N, K, iters, gs, vals=4, blk=1):
    """R's input read once, the factors written once; per pass R u and R^T v, per component the deflation, and for
    GS-PCA the two projections on either side."""
    flops = (iters + 0.5) * 4.0 * M * N * K + 2.0 * M * N * K
    if gs:
        flops += iters * 4.0 * (M + N) * sum(k // blk * blk for k in range(K))
    return vals * (M * N + float(M + N) * K) + 12.0 * K, flops


def work(case):
    if case["path"] == "batch":
        w = [_work_one(M, N, min(case["K"], M, N), case["iters"], case["algo"] == "gs") for M, N in _shapes(case)]
        return {"bytes": sum(x[0] for x in w), "flops": sum(x[1] for x in w)}
    vals = 8 if case["dtype"] == "f64" else 4
    b, f = _work_one(case["M"], case["N"], case["K"], case["iters"], case.get("algo", "gs") == "gs", vals,
                     case.get("block", 1))
    if case.get("want_R"):
        b += vals * case["M"] * case["N"]
    return {"bytes": b, "flops": f}


def _centred(X, center):
    return X - X.mean(0, keepdim=True) if center else X


def _exact_fit(X, K, iters, gs):
    """The method itself in 64 bits: power iterations on the residual, deflation, Gram-Schmidt."""
    R = X
    M, N = R.shape
    V = torch.zeros(M, K, dtype=torch.float64, device=R.device)
    U = torch.zeros(N, K, dtype=torch.float64, device=R.device)
    lam = torch.zeros(K, dtype=torch.float64, device=R.device)
    for k in range(K):
        v = R[:, k].clone()
        for _ in range(iters):
            u = R.t() @ v
            if gs and k:
                u = u - U[:, :k] @ (U[:, :k].t() @ u)
            u = u / u.norm()
            v = R @ u
            if gs and k:
                v = v - V[:, :k] @ (V[:, :k].t() @ v)
            lam[k] = v.norm()
            if gs:
                v = v / lam[k]
        V[:, k], U[:, k] = v, u
        R.addr_(v, u, alpha=-(float(lam[k]) if gs else 1.0))
    return (V * lam if gs else V), U, lam, R


def _exact_block(X, K, b, iters):
    """Block power iteration in 64 bits; the singular values alone, since the vectors' signs are free."""
    R = X
    V = torch.zeros(R.shape[0], 0, dtype=torch.float64, device=R.device)
    U = torch.zeros(R.shape[1], 0, dtype=torch.float64, device=R.device)
    lam = []
    for k0 in range(0, K, b):
        Z = R.t() @ R[:, k0:min(K, k0 + b)]
        Z = Z - U @ (U.t() @ Z)
        for _ in range(iters):
            u = torch.linalg.qr(Z)[0]
            Y = R @ u
            v = torch.linalg.qr(Y - V @ (V.t() @ Y))[0]
            Z = R.t() @ v
            Z = Z - U @ (U.t() @ Z)
        a, s, bt = torch.linalg.svd(Z.t() @ u)
        v, u = v @ a, u @ bt.t()
        R = R - (v * s) @ u.t()
        V, U = torch.cat([V, v], 1), torch.cat([U, u], 1)
        lam.append(s)
    return torch.cat(lam)


def exact(case, seed):
    gs = case.get("algo") == "gs"
    if case["path"] == "batch":
        Ts, Ps, ls, its = [], [], [], []
        for X in _batch_matrices(case, seed):
            K = min(case["K"], *X.shape)
            T, P, lam, _ = _exact_fit(X.double(), K, case["iters"], gs)
            Ts.append(T.t().reshape(-1))
            Ps.append(P.t().reshape(-1))
            ls.append(lam)
        return dict(T=torch.cat(Ts), P=torch.cat(Ps), lam=torch.cat(ls), iters=None)
    X = _centred(_matrix(case, seed).double(), case["center"])
    if case["path"] == "block":
        return dict(T=None, P=None, lam=_exact_block(X, case["K"], case["block"], case["iters"]), iters=None)
    T, P, lam, R = _exact_fit(X, case["K"], case["iters"], gs)
    out = dict(T=T, P=P, lam=lam, iters=None)
    if case.get("want_R"):
        out["R"] = R
    return out
