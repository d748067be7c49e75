"""The FP64 products on both sides of the sizes where another kernel takes them.

Few rows go to the plain or double-float kernels, more to the fixed-point one; beyond its
range three and four columns go to the symmetric FP64 kernel from 2000 rows on, the plain
one takes 5 to 7 columns as eight.  Bounds norm-wise against |K_y| |V|: FP64 products
2^-46 as in the other sizes, double-float entries are good to 2^-44 of the largest: 2^-43.
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _check(n, d, c, impl, ell, tol):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, d, 7, dist="normal", ell=ell, s2=1.7, noise=1e-3)
    V = synthetic.rng(8).standard_normal((n, c))
    l, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    ref = oracle.kyv(p.X, l, s2, p.noise, V)
    big = oracle.kyv(p.X, l, s2, p.noise, np.abs(V))
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, ard=p.ard) as s:
        Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t()
        O = s.matvec_f64(Vd, impl=impl).cpu().numpy()
    assert (np.linalg.norm(O - ref, axis=0) <= tol * np.linalg.norm(big, axis=0)).all()


@pytest.mark.parametrize("n", [8, 9, 16, 17])
@pytest.mark.parametrize("d,c", [(8, 1), (3, 7), (16, 16), (8, 17), (12, 25)])
def test_fp64_few_rows(n, d, c):
    _check(n, d, c, 0, 2.0, 2.0 ** -46)


@pytest.mark.parametrize("n,d,c", [
    (96, 8, 3), (97, 8, 3), (256, 8, 4), (257, 8, 4), (16, 8, 5), (17, 8, 8), (511, 12, 1),
    (512, 14, 4), (1536, 12, 5), (1537, 11, 16), (32, 14, 9), (33, 14, 17), (48, 13, 8),
    (49, 13, 5), (2048, 16, 2), (2049, 13, 1)])
def test_double_float_lines(n, d, c):
    _check(n, d, c, 1, 2.0, 2.0 ** -43)


@pytest.mark.parametrize("n,d,c", [
    (300, 4, 3), (300, 4, 5), (2000, 8, 3), (2001, 8, 3), (2001, 8, 4), (2001, 8, 5), (700, 16, 6),
    (700, 16, 7), (700, 3, 9), (700, 3, 19), (300, 20, 3), (300, 20, 7), (300, 20, 9)])
def test_beyond_the_fixed_point_range(n, d, c):
    _check(n, d, c, 0, 0.1, 2.0 ** -46)
