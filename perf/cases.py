"""The workloads this library is timed on, one case each, through its public entry points.

Products: `matvec_f32` is the reduced-precision product an inner solve iterates with (one
column, or a block of right-hand sides), `matvec_f64` the FP64-class one (impl 1: the outer
directions of the mixed solver and the KPCG_DF64 iterations; impl 0: the certified residual).
Whole calls: a solve at new hyperparameters (preconditioner rebuilt), the stochastic gradient,
predictions, the probit Laplace mode.  Batch: the two operators of one inner iteration of many
uneven systems.  Sizes are those of the library's benchmark, tests and data-set shapes.

The systems of the whole calls have noise variances of 1e-2 to 1e-1 and are solved to 1e-11, so
that their solutions are determined to about 1e-10 whatever the order of the roundings inside.
"""
import math

import numpy as np
import torch

import paper_1602_06693_gb300 as kpcg

DEV = "cuda"


def listed():
    return [
        # the smallest solve: a Concrete-shaped regression (n = 1030, d = 8), sqrt(n) inducing points
        dict(name="solve_concrete", kind="solve", n=1030, d=8, m=33, dist="normal", lo=1.0, hi=1.0,
             noise=1e-2, tol=1e-11),
        # one step of a hyperparameter search: new theta, 1024 inducing points, solve
        dict(name="solve_20k_m1024", kind="solve", n=20000, d=8, m=1024, dist="uniform", lo=0.3,
             hi=3.0, noise=1e-1, tol=1e-11),
        # one gradient of the log likelihood with 16 probes, forward solve and derivative products
        dict(name="grad_5k_t16", kind="grad", n=5000, d=9, m=256, t=16, dist="normal", lo=2.0,
             hi=4.0, noise=1e-1, tol=1e-11),
        # predictive mean and variance at 40 test inputs (blocks of 16, 16 and 8 systems)
        dict(name="predict_4k_40", kind="predict", n=4096, d=8, m=256, ns=40, dist="normal",
             lo=1.0, hi=1.0, noise=1e-2, tol=1e-10),
        # GP classification, the EEG data set's shape: Newton steps around mixed-precision B-solves
        dict(name="laplace_eeg", kind="laplace", n=14979, d=14, m=128, tol=1e-11),
        # a single small product: launches and latency
        dict(name="inner_1k", kind="mv32", impl=6, n=1030, d=8, c=1, dist="uniform", lo=0.3, hi=3.0),
        # the headline system's inner product
        dict(name="inner_65k", kind="mv32", impl=6, n=65536, d=8, c=1, dist="uniform", lo=0.3, hi=3.0),
        # the gradient's inner product: y and 16 probes on the Protein shape (odd n)
        dict(name="inner_45k_c17", kind="mv32", impl=5, n=45730, d=9, c=17, dist="normal", lo=2.0,
             hi=5.0),
        # the headline system's outer direction product
        dict(name="outer_65k", kind="mv64", impl=1, n=65536, d=8, c=1, dist="uniform", lo=0.3, hi=3.0),
        # the outer product of the gradient's block solve
        dict(name="outer_45k_c17", kind="mv64", impl=1, n=45730, d=9, c=17, dist="normal", lo=2.0,
             hi=5.0),
        # the certified residual's product of the headline system
        dict(name="certify_65k", kind="mv64", impl=0, n=65536, d=8, c=1, dist="uniform", lo=0.3, hi=3.0),
        # 32 uneven systems with 9 right-hand sides each: the operators of one inner iteration
        dict(name="batch_32_c9", kind="batch", probs=32, nlo=512, nhi=16384, c=9, noise=1e-1),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["mv32", "mv32", "block32", "outer", "outer", "block64", "certify", "solve",
                       "grad", "predict", "laplace", "batch"])
    dist = rng.choice(["uniform", "normal"])
    lo, hi = (0.3, 3.0) if dist == "uniform" else (1.0, 4.0)
    base = dict(dist=dist, lo=lo, hi=hi)
    if kind == "mv32":
        return dict(kind="mv32", impl=6, n=_logu(rng, 300, 65536), d=rng.randint(2, 16),
                    c=rng.randint(1, 3), **base)
    if kind == "block32":
        return dict(kind="mv32", impl=5, n=_logu(rng, 300, 45730), d=rng.randint(2, 16),
                    c=rng.randint(4, 17), **base)
    if kind == "outer":
        return dict(kind="mv64", impl=1, n=_logu(rng, 300, 65536), d=rng.randint(2, 16), c=1, **base)
    if kind == "block64":
        return dict(kind="mv64", impl=1, n=_logu(rng, 300, 30000), d=rng.randint(2, 10),
                    c=rng.randint(2, 17), **base)
    if kind == "certify":
        return dict(kind="mv64", impl=0, n=_logu(rng, 300, 50000), d=rng.randint(2, 12),
                    c=rng.randint(1, 2), **base)
    d = rng.randint(6, 12)
    if kind == "solve":
        n = _logu(rng, 600, 20000)
        return dict(kind="solve", n=n, d=d, m=rng.randint(16, min(1024, n // 4)), dist="normal", lo=1.0,
                    hi=2.0, noise=10.0 ** rng.uniform(-2, -1), tol=1e-11)
    if kind == "grad":
        n = _logu(rng, 600, 5000)
        return dict(kind="grad", n=n, d=d, m=rng.randint(16, n // 8), t=rng.randint(4, 16),
                    dist="normal", lo=2.0, hi=4.0, noise=1e-1, tol=1e-11)
    if kind == "predict":
        n = _logu(rng, 600, 4096)
        return dict(kind="predict", n=n, d=d, m=rng.randint(16, n // 8), ns=rng.randint(1, 40),
                    dist="normal", lo=1.0, hi=2.0, noise=10.0 ** rng.uniform(-2, -1), tol=1e-10)
    if kind == "laplace":
        n = _logu(rng, 600, 14979)
        return dict(kind="laplace", n=n, d=rng.randint(8, 16), m=rng.randint(16, 128), tol=1e-11)
    return dict(kind="batch", probs=rng.randint(4, 32), nlo=512, nhi=_logu(rng, 1024, 16384),
                c=rng.randint(1, 9), noise=1e-1)


# ------------------------------------------------------------------ inputs
def _batch_shapes(case):
    """(n, d) of each problem: sizes log-uniform, the same for every seed of a case."""
    r = np.random.default_rng(case["probs"] * 100003 + case["nhi"])
    return [(int(round(math.exp(r.uniform(math.log(case["nlo"]), math.log(case["nhi"]))))),
             int(r.integers(6, 17))) for _ in range(case["probs"])]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _inputs(n, d, dist, g):
    if dist == "uniform":
        return torch.rand((n, d), device=DEV, dtype=torch.float32, generator=g)
    return torch.randn((n, d), device=DEV, dtype=torch.float32, generator=g)


def _theta(rng, d, lo, hi, s2=1.0):
    """ARD log parameters, lengthscales log-uniform in [lo, hi]."""
    return np.concatenate([rng.uniform(math.log(lo), math.log(hi), d), [math.log(s2)]])


def _targets(X, g):
    """A smooth signal plus white noise."""
    Xd = X.double()
    return torch.sin(Xd).sum(1) + 0.1 * torch.randn(X.shape[0], device=DEV, dtype=torch.float64,
                                                    generator=g)


def _subset(rng, n, m):
    return np.sort(rng.choice(n, size=m, replace=False)).astype(np.int64)


def _block(n, c, dtype, g):
    """n x c standard-normal block, column-major."""
    return torch.randn((c, n), device=DEV, dtype=dtype, generator=g).t()


def _data(case, seed):
    """Everything a case's inputs consist of, without the library."""
    rng, g, kind = np.random.default_rng(seed), _gen(seed), case["kind"]
    D = {}
    if kind == "batch":
        D["problems"] = []
        c = case["c"]
        for n, d in _batch_shapes(case):
            lt = _theta(rng, d, 0.3 * math.sqrt(d), math.sqrt(d), math.exp(rng.uniform(-0.7, 0.7)))
            m = min(512, max(64, n // 8))
            D["problems"].append(dict(X=_inputs(n, d, "normal", g), theta=lt, noise=case["noise"],
                                      idx=_subset(rng, n, m), V=_block(n, c, torch.float32, g),
                                      R=_block(n, c, torch.float32, g)))
        return D
    n, d = case["n"], case["d"]
    if kind == "laplace":
        X = torch.randn((n, d), device=DEV, dtype=torch.float64, generator=g)
        X = ((X - X.mean(0)) / X.std(0)).float().contiguous()
        y = torch.where(torch.sin(X.double()).sum(1) >= 0, 1.0, -1.0).double()
        flip = torch.rand(n, device=DEV, generator=g) < 0.05
        D.update(X=X, y=torch.where(flip, -y, y).contiguous(), noise=1.0,
                 theta=np.concatenate([np.full(d, 0.5 * math.log(d)), [math.log(4.0)]]),
                 idx=_subset(rng, n, case["m"]))
        return D
    D.update(X=_inputs(n, d, case["dist"], g), theta=_theta(rng, d, case["lo"], case["hi"]),
             noise=case.get("noise", 1e-4))
    if kind in ("mv32", "mv64"):
        D["V"] = _block(n, case["c"], torch.float32 if kind == "mv32" else torch.float64, g)
        return D
    D["y"] = _targets(D["X"], g)
    D["idx"] = _subset(rng, n, case["m"])
    if kind == "grad":
        D["probes"] = torch.sign(_block(n, case["t"], torch.float64, g).t() + 1e-300).t()
    if kind == "predict":
        D["Xs"] = _inputs(case["ns"], d, case["dist"], g)
    return D


def prepare(case, seed):
    D, kind = _data(case, seed), case["kind"]
    S = dict(D, case=case)
    if kind == "batch":
        opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR, inner_shift=0.25, inner_tol=0.2)
        b = kpcg.Batch([(p["X"], p["theta"], p["noise"], p["idx"]) for p in D["problems"]], options=opt)
        b.set_tiling(8)  # a fixed tiling: the autotuner's choice may differ from run to run
        S["V"] = b.block([p["V"] for p in D["problems"]], torch.float32)
        S["R"] = b.block([p["R"] for p in D["problems"]], torch.float32)
        S["handle"] = b
        return S
    if kind == "solve":
        # the handle stands at other hyperparameters; the step under way moves it to new ones
        opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR, inner_tol=0.1)
        s = kpcg.Solver(D["X"], D["theta"] + 0.05, 2 * D["noise"], ard=True, options=opt)
        s.precond(kpcg.KPCG_PREC_NYSTROM, len(D["idx"]), D["idx"])
    elif kind == "grad":
        opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR, inner_shift=0.25, inner_tol=0.2)
        s = kpcg.Solver(D["X"], D["theta"] + 0.05, 2 * D["noise"], ard=True, options=opt)
        s.precond(kpcg.KPCG_PREC_NYSTROM, len(D["idx"]), D["idx"])
    elif kind == "predict":
        opt = kpcg.default_options(precision=kpcg.KPCG_DF64)
        s = kpcg.Solver(D["X"], D["theta"], D["noise"], ard=True, options=opt)
        s.precond(kpcg.KPCG_PREC_NYSTROM, len(D["idx"]), D["idx"])
        S["alpha"] = s.solve(D["y"], tol=1e-11)[0]
    elif kind == "laplace":
        opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR, inner_tol=1e-4)
        s = kpcg.Solver(D["X"], D["theta"], D["noise"], ard=True, options=opt)
        s.precond(kpcg.KPCG_PREC_NYSTROM, len(D["idx"]), D["idx"])
    else:
        s = kpcg.Solver(D["X"], D["theta"], D["noise"], ard=True)
    S["handle"] = s
    return S


def run(state):
    case, h = state["case"], state["handle"]
    kind = case["kind"]
    if kind == "mv32":
        return h.matvec_f32(state["V"], impl=case["impl"])
    if kind == "mv64":
        return h.matvec_f64(state["V"], impl=case["impl"])
    if kind == "solve":
        h.set_theta(state["theta"], state["noise"])
        return h.solve(state["y"], tol=case["tol"])[0]
    if kind == "grad":
        h.set_theta(state["theta"], state["noise"])
        g, alpha, _ = h.grad(state["y"], state["probes"], tol=case["tol"], want_alpha=True)
        return {"grad": g, "alpha": alpha}
    if kind == "predict":
        mean, var, _ = h.predict(state["Xs"], state["alpha"], tol=case["tol"])
        return {"mean": mean, "var": var}
    if kind == "laplace":
        f, a, _, _ = h.laplace(state["y"], cg_tol=case["tol"])
        return {"f": f, "a": a}
    return {"kv": h.matvec_f32(state["V"], case["c"]),
            "pc": h.precond_apply_f32(state["R"], case["c"])}


def _product(n, d, c, b):
    """Bytes and operations of one product: each distinct entry of K once (2 d operations for the
    distance, one exp), 2 n^2 c for the contraction."""
    return 4.0 * n * d + 2.0 * b * n * c, 0.5 * n * (n + 1) * (2 * d + 1) + 2.0 * n * n * c


def work(case):
    kind = case["kind"]
    if kind == "batch":
        by = fl = 0.0
        for n, d in _batch_shapes(case):
            m = min(512, max(64, n // 8))
            p = _product(n, d, case["c"], 4)
            by += p[0] + 8.0 * n * m + 8.0 * n * case["c"]
            fl += p[1] + 4.0 * n * m * case["c"]
        return {"bytes": by, "flops": fl}
    n, d = case["n"], case["d"]
    if kind in ("mv32", "mv64"):
        by, fl = _product(n, d, case["c"], 4 if kind == "mv32" else 8)
        return {"bytes": by, "flops": fl}
    # whole calls: the preconditioner's n m^2 and one product with every right-hand side (how
    # many iterations a solve needs is the method's, not a size)
    m = case["m"]
    c = {"grad": case.get("t", 0) + 1, "predict": case.get("ns", 1)}.get(kind, 1)
    by, fl = _product(n, d, c, 8)
    if kind != "predict":
        fl += 1.0 * n * m * m
    if kind == "grad":
        fl += 2.0 * n * n * c * (d + 1)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ 64-bit values
def _kernel(A, B, theta):
    """K(A, B) of Eq. 1 in FP64, A and B float32 inputs."""
    il = torch.as_tensor(np.exp(-theta[:-1]), device=DEV)
    a, b = A.double() * il, B.double() * il
    q = torch.zeros((a.shape[0], b.shape[0]), device=DEV, dtype=torch.float64)
    for r in range(a.shape[1]):
        t = a[:, r, None] - b[None, :, r]
        q.addcmul_(t, t)
    return q.mul_(-0.5).add_(float(theta[-1])).exp_()


def _times(X, theta, noise, V):
    V = V.double()
    out = noise * V
    step = max(1, int(2.5e8 // max(1, X.shape[0])))
    for i in range(0, X.shape[0], step):
        out[i:i + step] += _kernel(X[i:i + step], X, theta) @ V
    return out


def _chol(X, theta, noise):
    K = _kernel(X, X, theta)
    K.diagonal().add_(noise)
    return torch.linalg.cholesky(K)


def exact(case, seed):
    D, kind = _data(case, seed), case["kind"]
    if kind == "batch":
        ld, c = max(p["X"].shape[0] for p in D["problems"]), case["c"]
        kv = torch.zeros((len(D["problems"]) * c, ld), device=DEV, dtype=torch.float64).t()
        pc = torch.zeros_like(kv)
        for k, p in enumerate(D["problems"]):
            n, nz = p["X"].shape[0], p["noise"] * 1.25
            kv[:n, k * c:(k + 1) * c] = _times(p["X"], p["theta"], nz, p["V"])
            U = p["X"][torch.as_tensor(p["idx"], device=DEV)]
            kxu, R = _kernel(p["X"], U, p["theta"]), p["R"].double()
            L = torch.linalg.cholesky(nz * _kernel(U, U, p["theta"]) + kxu.t() @ kxu)
            pc[:n, k * c:(k + 1) * c] = (R - kxu @ torch.cholesky_solve(kxu.t() @ R, L)) / nz
        return {"kv": kv, "pc": pc}
    X, theta, noise = D["X"], D["theta"], D["noise"]
    if kind in ("mv32", "mv64"):
        return _times(X, theta, noise, D["V"])
    if kind == "solve":
        return torch.cholesky_solve(D["y"][:, None], _chol(X, theta, noise))[:, 0]
    if kind == "predict":
        L, ks = _chol(X, theta, noise), _kernel(X, D["Xs"], theta)
        a = torch.cholesky_solve(D["y"][:, None], L)
        w = torch.linalg.solve_triangular(L, ks, upper=False)
        return {"mean": (ks.t() @ a)[:, 0], "var": math.exp(theta[-1]) - (w * w).sum(0)}
    if kind == "grad":
        L, R = _chol(X, theta, noise), D["probes"]
        a = torch.cholesky_solve(D["y"][:, None], L)
        W = torch.cholesky_solve(R, L)
        K = _kernel(X, X, theta)
        il, out = np.exp(-theta[:-1]), []
        Xd = X.double()
        for r in range(X.shape[1] + 1):
            G = K if r == X.shape[1] else K * ((Xd[:, r, None] - Xd[None, :, r]) * il[r]).square_()
            out.append(-0.5 * (W * (G @ R)).sum() / R.shape[1] + 0.5 * (a * (G @ a)).sum())
        out.append(noise * (-0.5 * (W * R).sum() / R.shape[1] + 0.5 * (a * a).sum()))
        return {"grad": torch.stack(out), "alpha": a[:, 0]}
    # probit Laplace mode by Newton's method on the dense system
    K, y = _kernel(X, X, theta), D["y"]
    f = torch.zeros_like(y)
    for _ in range(12):
        z = y * f
        ratio = math.sqrt(2.0 / math.pi) / torch.special.erfcx(-z / math.sqrt(2.0))
        g, W = y * ratio, ratio * (z + ratio)
        sw = W.sqrt()
        b = W * f + g
        L = sw[:, None] * K * sw[None, :]
        L.diagonal().add_(1.0)
        v = (sw * (K @ b))[:, None]
        a = b - sw * torch.cholesky_solve(v, torch.linalg.cholesky(L))[:, 0]
        f_new = K @ a
        done = float((f_new - f).abs().max()) < 1e-13
        f = f_new
        if done:
            break
    return {"f": f, "a": a}
