"""K_UX K_XU of the Nystrom set-up over the sizes where its work split changes.

Tiles are 128 x 64 (the last one ragged), rows come in groups of 128, split over
CTAs while m is small and in blocks of about 49152 / ceil(m/128) rows.  The FP64
apply is compared with its formula on the oracle's kernel in FP64; the amplitude
s2 moves the fixed-point scale.  The inner matrix has a condition number kappa
below 2e5, so the FP64 parts are accurate to ~ kappa 2^-53 = 2e-11 and the
apply's compensated FP32 sums, 2^-44 of sums over n rows, to well under 1e-9
(the bound of the applies' test, at kappa 1e6).
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# n, m, s2
CASES = [(1, 1, 1.0), (65, 63, 3.7), (127, 64, 1e-3), (129, 65, 1.0), (1030, 127, 250.0),
         (513, 128, 1.0), (1025, 129, 0.02), (9000, 40, 1.0), (2047, 191, 1e4),
         (6500, 1000, 1.0)]


@pytest.mark.parametrize("n,m,s2", CASES)
def test_setup_sum(n, m, s2):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, 6, 11, dist="normal", ell=0.7, s2=s2, noise=0.3 * s2)
    idx = synthetic.inducing_subset(n, m, seed=3)
    R = synthetic.rng(5).standard_normal((n, min(n, 2)))  # one row: one column
    ell, amp = oracle.split_theta(p.log_theta, p.d, p.ard)
    X = p.X.astype(np.float64) / ell
    def K(a, b):
        q = (a**2).sum(1)[:, None] + (b**2).sum(1)[None] - 2.0 * a @ b.T
        return amp * np.exp(-0.5 * np.maximum(q, 0.0))
    kxu, kuu = K(X, X[idx]), K(X[idx], X[idx])
    M = p.noise * kuu + kxu.T @ kxu
    assert np.linalg.cond(M) < 2e5
    ref = (R - kxu @ np.linalg.solve(M, kxu.T @ R)) / p.noise
    opt = kpcg.default_options(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, m, idx)
        Rd = torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t()
        Z = s.precond_apply(Rd).cpu().numpy()
    assert np.linalg.norm(Z - ref) / np.linalg.norm(ref) <= 1e-9
