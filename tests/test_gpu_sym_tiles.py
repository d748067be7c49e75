"""The symmetric tensor-core product (matvec_f32 impl 6) at the edges of its tiles:
row tiles of 128, column tiles of 256 (their second half absent, ragged or full) and one or
several row tiles per work item.  Tolerance: 2e-5 of the norm, that of every FP32
product here (entries ~2^-22 from ex2.approx plus |arg| 2^-24, summed in FP32).
"""
import numpy as np
import pytest

import oracle
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


@pytest.mark.parametrize("n,d,c", [
    (129, 3, 1), (255, 10, 1), (256, 8, 2), (257, 11, 1), (383, 20, 1), (384, 8, 1), (385, 8, 3),
    (513, 14, 1), (1025, 8, 1), (3000, 16, 1)])
def test_tile_edges(kpcg, n, d, c):
    p = synthetic.make_problem(n, d, 4, dist="normal", ell=2.0, s2=1.3, noise=1e-2)
    V = synthetic.rng(9).standard_normal((n, c)).astype(np.float32)
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    ref = oracle.kyv(p.X, ell, s2, p.noise, V.astype(np.float64))
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        O = s.matvec_f32(torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t(), impl=6)
        O2 = s.matvec_f32(torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t(), impl=6)
    assert torch.equal(O, O2)
    O = O.cpu().numpy().astype(np.float64)
    for k in range(c):
        assert np.linalg.norm(O[:, k] - ref[:, k]) <= 2e-5 * np.linalg.norm(ref[:, k])
