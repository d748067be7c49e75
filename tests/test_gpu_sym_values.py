"""Infinities, NaN and sums that leave FP32's range on the way in the symmetric
tensor-core product (matvec_f32 impl 6).

The kernel is broad, no entry underflows: an infinity in V reaches every row, a NaN
too.  In the last case the 256-column tiles 0 and 8 add 3e38 each to a row, tile 16 takes 3e38
away: the partials and the result are FP32 numbers, the running sum is not.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def kpcg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as k
    from paper_1602_06693_gb300 import build
    build.build()
    return k


@pytest.mark.parametrize("n", [130, 900, 5000])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_values_that_are_not_finite(kpcg, n, bad):
    p = synthetic.make_problem(n, 4, 3, dist="normal", ell=5.0, noise=1e-2)
    V = synthetic.rng(4).standard_normal((n, 2))
    V[n // 2, 1] = bad
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().float().t()
        O = s.matvec_f32(Vd, impl=6).cpu().numpy()
    assert np.isfinite(O[:, 0]).all()
    assert np.isnan(O[:, 1]).all() if np.isnan(bad) else (O[:, 1] == bad).all()


def test_sum_beyond_the_range(kpcg):
    n, noise = 17 * 256, 1e-2
    p = synthetic.make_problem(n, 4, 3, dist="normal", ell=100.0, noise=noise)
    V = np.zeros(n)
    for tile, v in ((0, 3e38), (8, 3e38), (16, -3e38)):
        V[256 * tile:256 * (tile + 1)] = v / 256
    at = np.flatnonzero(V)
    X = p.X.astype(np.float64) / 100.0
    K = np.exp(-0.5 * ((X[:, None] - X[None, at]) ** 2).sum(2))
    ref = K @ V[at] + noise * V
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        O = s.matvec_f32(torch.from_numpy(V).cuda().float(), impl=6).double().cpu().numpy()
    assert np.abs(O - ref).max() <= 2e-5 * 9e38  # the kernel's parity bound
