"""The vector steps of PCG over the sizes where their work split changes.

One cluster of 1, 2, 4 or 8 CTAs runs a column's step: 256 rows per CTA and
batch element, batches of 8 per thread, and from 24577 rows on the steps are
separate kernels.  Each column is its own CG: a zero column costs no iteration,
doubling a column doubles every vector and scalar exactly (powers of two), and
the certified residual meets the tolerance in every column.  Doubled columns
share iterations; their products may round differently next to other columns,
by 2^-24 of the inner solve's correction, so the solutions agree to the
tolerance times the condition number, below 1e-8 x 1e3 with this noise.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-8


@pytest.mark.parametrize("precision", ["KPCG_FP64", "KPCG_TC_IR"])
@pytest.mark.parametrize("n", [2, 255, 257, 513, 1025, 2049, 16384, 16385, 24577])
def test_columns(n, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, 4, 7, dist="normal", ell=0.2, noise=0.5)
    b = synthetic.rng(9).standard_normal(n)
    B = np.stack([b, np.zeros(n), 2.0 * b, synthetic.rng(10).standard_normal(n)])
    opt = kpcg.default_options(precision=getattr(kpcg, precision))
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        Bd = torch.from_numpy(np.ascontiguousarray(B)).cuda().t()
        X, it, info, st = s.solve(Bd, tol=TOL)
        K = s.matvec_f64(X.contiguous() if X.dim() == 1 else X, impl=0)
        x = X.cpu().numpy()
        r = (Bd - K).cpu().numpy()
    assert st == 0 and info.max_rel_res <= TOL
    assert np.all(x[:, 1] == 0.0) and it[1] == 0
    nb = np.linalg.norm(B.T, axis=0)
    for k in (0, 2, 3):
        # the product itself is FP64-class: 1e-13 of ||K|| ||x||
        assert np.linalg.norm(r[:, k]) <= 1.01 * TOL * nb[k]
    assert abs(int(it[0]) - int(it[2])) <= 1
    assert np.linalg.norm(x[:, 2] - 2.0 * x[:, 0]) <= 1e-5 * np.linalg.norm(x[:, 2])


@pytest.mark.parametrize("n,c", [(300, 1), (2500, 5)])
def test_replayed_chunks(n, c):
    """A fresh handle's buffers move between its first inner solves and a used one's do
    not, so the recorded iterations are replayed from different points on: every kernel is
    deterministic, the results are equal bit by bit."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, 4, 7, dist="normal", ell=1.0, noise=1e-3)
    idx = synthetic.inducing_subset(n, 32, seed=3)
    B = torch.from_numpy(np.ascontiguousarray(synthetic.rng(9).standard_normal((c, n)))).cuda().t()
    opt = kpcg.default_options(precision=kpcg.KPCG_TC_IR)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, 32, idx)
        runs = [s.solve(B, tol=TOL) for _ in range(3)]
    X, it, info, st = runs[0]
    assert st == 0 and info.outer_steps >= 3 and info.max_rel_res <= TOL
    for Y, jt, jnfo, _ in runs[1:]:
        assert np.array_equal(jt, it) and jnfo.iters_total == info.iters_total
        assert torch.equal(Y, X)
