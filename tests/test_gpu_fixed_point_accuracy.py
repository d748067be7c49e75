"""Accuracy of the FP64-accurate product (matvec_f64 impl 0) against extended precision.

References are sums of FP64 scaled inputs' kernel entries in long double.  A row's error
is held against (|K_y| |V|)_i:
 * narrow kernels at large n, where n small entries meet one of size 1: an FP64 sum in
   chains of ~2^9 terms rounds at 2^-53 2^4.5, so 2^-48.  Vectors of one sign let every
   bias of the small entries add up, a constant one with all its digits set also that of
   products of low digits;
 * broad kernels over the column widths and passes, norm-wise: 2^-53 in each entry's
   exponent (of size ~4, and from inputs rounded at 2^-53) and in the sums: 2^-50.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LD = np.longdouble


@pytest.fixture(scope="module")
def kpcg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as k
    from paper_1602_06693_gb300 import build
    build.build()
    return k


def _rows(X, theta, rows):
    """Rows of K in long double."""
    Y = X.astype(LD) / np.exp(theta[:-1]).astype(LD)
    q = np.zeros((len(rows), X.shape[0]), dtype=LD)
    for r in range(X.shape[1]):
        q += (Y[rows, r][:, None] - Y[None, :, r]) ** 2
    return np.exp(-q / 2) * np.exp(LD(theta[-1]))


def _product(kpcg, X, theta, noise, V, impl):
    with kpcg.Solver(torch.from_numpy(X).cuda(), theta, noise) as s:
        Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t()
        return s.matvec_f64(Vd, impl=impl).cpu().numpy().reshape(V.shape)


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("n,d,ell", [(65536, 16, 0.62), (40001, 12, 0.62)])
def test_narrow_kernel(kpcg, impl, n, d, ell):
    rng = synthetic.rng(5)
    X = np.clip(rng.standard_normal((n, d)), -4.0, 4.0).astype(np.float32)  # scaled: within 8
    theta = np.concatenate([np.full(d, np.log(ell)), [0.0]])
    V = np.stack([np.ones(n), np.full(n, 1.0 / 3.0), 0.5 + rng.random(n)], axis=1)
    O = _product(kpcg, X, theta, 1e-3, V, impl)
    rows = np.array([0, 1, 77, n // 2, n - 2, n - 1])
    K = _rows(X, theta, rows)
    ref = K @ V.astype(LD) + LD(1e-3) * V[rows].astype(LD)
    err = np.abs((O[rows].astype(LD) - ref) / ref).astype(np.float64)  # all terms are positive
    assert err.max() <= 2.0 ** -48, err


@pytest.mark.parametrize("n,d,c", [(65, 12, 8), (129, 16, 2), (1000, 8, 24), (1025, 5, 25),
                                   (1100, 9, 49), (1100, 14, 1)])
def test_broad_kernel(kpcg, n, d, c):
    p = synthetic.make_problem(n, d, 7, dist="normal", ell=2.5, s2=1.7, noise=1e-3)
    theta = np.concatenate([np.full(d, np.log(2.5)), [p.log_theta[-1]]])
    assert np.allclose(p.log_theta, theta, rtol=1e-12)
    V = synthetic.rng(8).standard_normal((n, c))
    V[:, 0] = 1.0 / 3.0
    O = _product(kpcg, p.X, p.log_theta, p.noise, V, 0)
    K = _rows(p.X, p.log_theta, np.arange(n))
    ref = K @ V.astype(LD) + LD(p.noise) * V.astype(LD)
    big = K @ np.abs(V).astype(LD)
    err = np.linalg.norm((O - ref).astype(np.float64), axis=0) / np.linalg.norm(
        big.astype(np.float64), axis=0)
    assert err.max() <= 2.0 ** -50, err
