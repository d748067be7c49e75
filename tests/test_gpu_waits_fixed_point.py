"""Bounded waits of the fixed-point kernels: the FP64-class product and the sum of the
Nystrom set-up.

As for the other tensor-core kernels, the options' test hook lets a wait run out under
a 2 ms limit: the call reports KPCG_ERR_TIMEOUT, the flag is cleared with the report and
the handle stays usable.
"""
import numpy as np
import pytest

import oracle
import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STALL = dict(wait_stall=1, wait_limit_ns=2_000_000)


@pytest.fixture(scope="module")
def kpcg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as k
    from paper_1602_06693_gb300 import build
    build.build()
    return k


def _timeout(kpcg, call):
    with pytest.raises(kpcg.KpcgError) as e:
        call()
    assert e.value.name == "KPCG_ERR_TIMEOUT"


# impl 0 takes the product at every width, impl 1 for three and more columns or d > 10
@pytest.mark.parametrize("impl,d,c", [(0, 8, 1), (0, 14, 3), (1, 8, 3), (1, 14, 1)])
def test_product(kpcg, impl, d, c):
    p = synthetic.make_problem(3000, d, 5, dist="normal", ell=3.0, noise=1e-2)
    V = synthetic.rng(3).standard_normal((p.n, c))
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    ref = oracle.kyv(p.X, ell, s2, p.noise, V)
    Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t()
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, ard=p.ard) as s:
        s.set_options(kpcg.default_options(**STALL))
        for _ in range(2):
            _timeout(kpcg, lambda: s.matvec_f64(Vd, impl=impl))
        s.set_options(kpcg.default_options())
        O = s.matvec_f64(Vd, impl=impl).cpu().numpy().reshape(p.n, c)
    # the oracle's sums of 3000 terms, 2^-53 sqrt(n) of them
    assert np.linalg.norm(O - ref) <= 1e-13 * np.linalg.norm(ref)


def test_setup(kpcg):
    p = synthetic.make_problem(3000, 6, 5, dist="normal", ell=1.0, noise=1e-1)
    idx = synthetic.inducing_subset(p.n, 200, seed=3)
    R = torch.from_numpy(synthetic.rng(5).standard_normal(p.n)).cuda()
    X = torch.from_numpy(p.X).cuda()
    opt = dict(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(X, p.log_theta, p.noise, options=kpcg.default_options(**opt)) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, 200, idx)
        want = s.precond_apply(R)
    with kpcg.Solver(X, p.log_theta, p.noise, options=kpcg.default_options(**opt, **STALL)) as s:
        for _ in range(2):
            _timeout(kpcg, lambda: s.precond(kpcg.KPCG_PREC_NYSTROM, 200, idx))
        s.set_options(kpcg.default_options(**opt))
        s.precond(kpcg.KPCG_PREC_NYSTROM, 200, idx)
        assert torch.equal(s.precond_apply(R), want)


@pytest.mark.parametrize("precision,max_iter", [("KPCG_FP32", 100000), ("KPCG_FP64", 0)])
def test_last_residual_of_a_solve(kpcg, precision, max_iter):
    """The residual of what a solve returns is its last product, and the only one of these
    two: FP32 iterations take the FP32 kernel, and without a budget nothing iterates."""
    p = synthetic.make_problem(1500, 8, 5, dist="normal", ell=3.0, noise=1e-1)
    y = torch.from_numpy(p.y).cuda()
    opt = dict(precision=getattr(kpcg, precision), max_iter=max_iter)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        s.set_options(kpcg.default_options(**opt, **STALL))
        _timeout(kpcg, lambda: s.solve(y, tol=1e-4))
        s.set_options(kpcg.default_options())
        s.matvec_f64(y, impl=0)  # the flag is cleared
        x, _, info, st = s.solve(y, tol=1e-8)
        assert st == 0 and info.max_rel_res <= 1e-8


@pytest.mark.parametrize("n,fixed", [(50, False), (256, False), (257, True), (2048, True),
                                     (2049, False)])
def test_where_the_double_float_product_takes_it(kpcg, n, fixed):
    """One column, d <= 10: only a few row tiles go to the fixed-point kernel, which the test
    hook of the waits tells from the double-float ones; fewer or more are slower there."""
    p = synthetic.make_problem(n, 8, 5, dist="normal", ell=3.0, noise=1e-2)
    V = torch.from_numpy(synthetic.rng(3).standard_normal(n)).cuda()
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, ard=p.ard) as s:
        s.set_options(kpcg.default_options(**STALL))
        if fixed:
            _timeout(kpcg, lambda: s.matvec_f64(V, impl=1))
        else:
            s.matvec_f64(V, impl=1)
