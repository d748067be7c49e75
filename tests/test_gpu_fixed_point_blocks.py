"""Blocks of FP64 columns whose last pass is a narrow one.

The fixed-point product takes a block in passes of equal width, at most 24 columns; from
530 columns on the last pass can have one or two.  Every column is compared with
the oracle, against 2^-46 |K_y| |V| as in the other widths.
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("n,d,c", [(130, 4, 530), (130, 4, 553), (65, 14, 577), (130, 4, 529)])
def test_narrow_last_pass(impl, n, d, c):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, d, 7, dist="normal", ell=2.0, s2=1.7, noise=1e-3)
    V = synthetic.rng(8).standard_normal((n, c))
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    ref = oracle.kyv(p.X, ell, s2, p.noise, V)
    big = oracle.kyv(p.X, ell, s2, p.noise, np.abs(V))
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, ard=p.ard) as s:
        Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t()
        O = s.matvec_f64(Vd, impl=impl).cpu().numpy()
    err = np.linalg.norm(O - ref, axis=0) / np.linalg.norm(big, axis=0)
    assert err.max() <= 2.0 ** -46, (int(err.argmax()), err.max())
