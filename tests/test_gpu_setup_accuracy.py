"""The Nystrom set-up's inner matrix M = noise K_UU + K_UX K_XU keeps FP64 accuracy.

M is nearly singular here (kappa 2e7 to 4e10 with these sizes), so the apply amplifies
an error in M far above all others if its right-hand side is a unit vector: K_UX e_i is a
row of K_XU, without rounding.  The yardstick is the same formula with M formed and factored in
FP64 on the CPU, both against extended precision.  The device adds in another order and
applies an explicit inverse: 8 times the yardstick, where a relative error of 2^-48
in K_UX K_XU gives 15 to 40 times (computed with such errors put into M).  The amplitude s2 moves
the scale of the set-up's digits over a power of two and far from 1.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LD = np.longdouble


def _factor(A):
    L = A.copy()
    for j in range(len(L)):
        L[j, j] = np.sqrt(L[j, j])
        L[j + 1:, j] /= L[j, j]
        L[j + 1:, j + 1:] -= np.outer(L[j + 1:, j], L[j + 1:, j])
    return np.tril(L)


def _solve(L, B):
    x = B.copy()
    for j in range(len(L)):
        x[j] /= L[j, j]
        x[j + 1:] -= np.outer(L[j + 1:, j], x[j])
    for j in range(len(L) - 1, -1, -1):
        x[j] /= L[j, j]
        x[:j] -= np.outer(L[j, :j], x[j])
    return x


@pytest.mark.parametrize("n,d,m,ell,noise,s2", [
    (3000, 3, 60, 1.0, 1e-3, 1.0), (3000, 3, 60, 1.0, 1e-3, 0.9), (3000, 3, 60, 1.0, 1e-3, 3e7),
    (3000, 3, 60, 1.0, 1e-3, 1e-9), (9000, 2, 40, 0.6, 1e-4, 1.0), (3000, 2, 48, 0.7, 1e-4, 2.5)])
def test_inner_matrix(n, d, m, ell, noise, s2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, d, 11, dist="normal", ell=ell, s2=s2, noise=noise * s2)
    idx = synthetic.inducing_subset(n, m, seed=3)
    amp = np.exp(LD(p.log_theta[-1]))
    Y = p.X.astype(LD) * np.exp(-LD(p.log_theta[0]))

    def K(A, B):
        return amp * np.exp(-sum((A[:, r][:, None] - B[:, r][None]) ** 2 for r in range(d)) / 2)

    kxu, kuu = K(Y, Y[idx]), K(Y[idx], Y[idx])
    at = np.array([0, 1, 7, n // 3, n - 1, idx[0], idx[m // 2], idx[-1]])
    R = np.zeros((n, len(at)))
    R[at, np.arange(len(at))] = 1.0
    nz = LD(p.noise)
    ref = (R.astype(LD) - kxu @ _solve(_factor(nz * kuu + kxu.T @ kxu), kxu[at].T)) / nz
    k64 = kxu.astype(np.float64)
    S = np.zeros((m, m))
    for i in range(0, n, 512):
        S += k64[i:i + 512].T @ k64[i:i + 512]
    u = _solve(np.linalg.cholesky(p.noise * kuu.astype(np.float64) + S), k64[at].T.copy())
    yard = (R.astype(LD) - kxu @ u.astype(LD)) / nz
    opt = kpcg.default_options(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, m, idx)
        Z = s.precond_apply(torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t()).cpu().numpy()

    def err(z):
        e = np.linalg.norm((z - ref).astype(np.float64), axis=0)
        return (e / np.linalg.norm(ref.astype(np.float64), axis=0)).max()

    assert err(Z) <= 8.0 * err(yard), (err(Z), err(yard))


@pytest.mark.parametrize("n,d,m,ell,noise", [(65536, 8, 16, 0.6, 1e-3), (65536, 8, 12, 0.6, 1e-2),
                                             (65536, 12, 16, 1.0, 1e-3)])
def test_narrow_kernel(n, d, m, ell, noise):
    """Many entries far below the one of size 1: what is cut off each of them must not add up
    over the n rows.  Six to fifteen units of 1e-15 missing on M's diagonal (the squares
    of the digits below 2^-32) show as 13 to 27 times the yardstick, which works on K_XU
    as the library keeps it, in FP32 pairs."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, d, 11, dist="normal", ell=ell, s2=1.0, noise=noise)
    idx = synthetic.inducing_subset(n, m, seed=3)
    Y = p.X.astype(LD) * np.exp(-LD(p.log_theta[0]))

    def K(A, B):
        return np.exp(-sum((A[:, r][:, None] - B[:, r][None]) ** 2 for r in range(d)) / 2)

    kxu, kuu = K(Y, Y[idx]), K(Y[idx], Y[idx])
    at = np.array([0, 1, 7, n // 3, n - 1, idx[0], idx[m // 2], idx[-1]])
    R = np.zeros((n, len(at)))
    R[at, np.arange(len(at))] = 1.0
    ref = (R.astype(LD) - kxu @ _solve(_factor(LD(noise) * kuu + kxu.T @ kxu), kxu[at].T)) / LD(noise)
    k64 = kxu.astype(np.float64)
    hi = k64.astype(np.float32)
    k64 = hi.astype(np.float64) + (k64 - hi).astype(np.float32)
    S = np.zeros((m, m))
    for i in range(0, n, 512):
        S += k64[i:i + 512].T @ k64[i:i + 512]
    u = _solve(np.linalg.cholesky(noise * kuu.astype(np.float64) + S), k64[at].T.copy())
    yard = (R.astype(LD) - k64.astype(LD) @ u.astype(LD)) / LD(noise)
    opt = kpcg.default_options(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, m, idx)
        Z = s.precond_apply(torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t()).cpu().numpy()

    def err(z):
        e = np.linalg.norm((z - ref).astype(np.float64), axis=0)
        return (e / np.linalg.norm(ref.astype(np.float64), axis=0)).max()

    assert err(Z) <= 8.0 * err(yard), (err(Z), err(yard))
