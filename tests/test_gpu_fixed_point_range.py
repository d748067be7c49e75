"""The FP64-accurate product at the ends of FP64's range.

A power of two on V changes the exponents of the products and sums only, so the result
carries it exactly as long as it is a normal number itself, also where s^2 brings back
into range what V alone would take out of it.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("log2_s2,power", [(-40, 1018), (60, -1074), (0, 900), (0, -900)])
@pytest.mark.parametrize("c", [1, 3])
def test_power_of_two_on_v(log2_s2, power, c):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    n = 300
    p = synthetic.make_problem(n, 3, 7, dist="normal", ell=3.0, s2=2.0 ** log2_s2, noise=1e-3)
    V = synthetic.rng(8).integers(1, 16, (n, c)).astype(np.float64)
    W = np.ldexp(V, power)
    assert np.array_equal(np.ldexp(W, -power), V)
    noise = p.noise * 2.0 ** log2_s2
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, noise) as s:
        def product(A):
            return s.matvec_f64(torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t(),
                                impl=0).cpu().numpy()
        O, Q = product(V), product(W)
    ref = np.ldexp(O, power)
    assert np.isfinite(ref).all() and (np.abs(ref) > 2.0 ** -1020).all()
    assert np.array_equal(Q, ref)
