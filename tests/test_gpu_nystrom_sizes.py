"""Nystrom applies over the sizes where their work split changes.

The projection takes column groups of 32, 64, 128 or 256 inducing points and row
ranges of 32 to 512 rows, the back products 1, 4, 8, 9 or 16 columns at a time.
P^-1 R is compared with its formula (the inversion lemma of Sec. 3.1) on the
oracle's kernel blocks in FP64.  The data are spread out (l = 1 in six
dimensions) with noise 0.1, so the inner matrix has a condition number below 1e6
and its FP64 solve is accurate to ~1e6 x 2^-53 = 1e-10; the FP32 apply rounds
its result (2^-24) and its compensated sums (2^-44, amplified as above).
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CASES = [(1, 1, 1), (40, 31, 3), (129, 32, 4), (300, 33, 5), (513, 64, 8), (700, 65, 9),
         (1030, 128, 2), (1030, 129, 16), (2050, 256, 17), (1500, 257, 33)]


@pytest.fixture(scope="module")
def kpcg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as k
    from paper_1602_06693_gb300 import build
    build.build()
    return k


def _case(n, m, c, shift):
    p = synthetic.make_problem(n, 6, 11, dist="normal", ell=1.0, noise=0.1)
    idx = synthetic.inducing_subset(n, m, seed=3)
    R = synthetic.rng(5).standard_normal((n, c))
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    X = p.X.astype(np.float64) / ell
    def K(a, b):
        return s2 * np.exp(-0.5 * ((a[:, None, :] - b[None, :, :]) ** 2).sum(-1))
    nz = p.noise * (1.0 + shift)
    kxu, kuu = K(X, X[idx]), K(X[idx], X[idx])
    M = nz * kuu + kxu.T @ kxu
    assert np.linalg.cond(M) < 1e6
    ref = (R - kxu @ np.linalg.solve(M, kxu.T @ R)) / nz
    return p, idx, R, ref


def _err(a, ref):
    return float(np.linalg.norm(a - ref) / np.linalg.norm(ref))


@pytest.mark.parametrize("n,m,c", CASES)
def test_fp64_apply(kpcg, n, m, c):
    p, idx, R, ref = _case(n, m, c, 0.0)
    opt = kpcg.default_options(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, m, idx)
        Rd = torch.from_numpy(np.ascontiguousarray(R.T)).cuda().t()
        Z = s.precond_apply(Rd).cpu().numpy()
    assert _err(Z, ref) <= 1e-9


@pytest.mark.parametrize("n,m,c", CASES)
def test_batched_fp32_apply(kpcg, n, m, c):
    # two problems of different sizes, the second without a preconditioner
    p, idx, R, ref = _case(n, m, c, 0.25)
    q = synthetic.make_problem(70, 3, 2, noise=0.1)
    opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR, inner_shift=0.25)
    with kpcg.Batch([(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, idx),
                     (torch.from_numpy(q.X).cuda(), q.log_theta, q.noise, None)],
                    options=opt) as b:
        R2 = synthetic.rng(6).standard_normal((70, c)).astype(np.float32)
        Z = b.precond_apply_f32(b.block([R.astype(np.float32), R2], torch.float32), c)
        z, z2 = (t.cpu().numpy() for t in b.unblock(Z, c))
    assert _err(z, ref) <= 1e-6
    assert np.array_equal(z2, R2)
