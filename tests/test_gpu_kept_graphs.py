"""Inner iterations replayed from a graph over the outer steps of a solve, for every inner
operator and preconditioner: equal bit by bit to the same solve without graphs (profiling turns
them off); every kernel is deterministic."""
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


def _precond(kpcg, s, kind, n):
    idx = synthetic.inducing_subset(n, 40, seed=3)
    if kind == "pitc":
        s.precond_pitc(40, idx, 64)
    elif kind == "block":
        s.precond(kpcg.KPCG_PREC_BLOCK_JACOBI, 64)
    elif kind != "none":
        s.precond(getattr(kpcg, "KPCG_PREC_" + kind.upper()), 40, idx)


CASES = [(prec, kind, c, 0) for prec in ("KPCG_FP32_IR", "KPCG_FP32X_IR", "KPCG_TC_IR", "KPCG_TCX_IR")
         for kind, c in (("nystrom", 1), ("none", 5))]
CASES += [("KPCG_TC_IR", kind, 2, 0) for kind in ("fitc", "pitc", "block")]
CASES += [("KPCG_TCX_IR", "nystrom", 2, 1), ("KPCG_TCX_IR", "fitc", 1, 1)]


@pytest.mark.parametrize("precision,kind,c,inner_f64", CASES)
def test_solve(kpcg, precision, kind, c, inner_f64):
    n = 700
    p = synthetic.make_problem(n, 6, 7, dist="normal", ell=2.0, noise=1e-2)
    B = torch.from_numpy(np.ascontiguousarray(synthetic.rng(9).standard_normal((c, n)))).cuda().t()
    out = []
    for profile in (0, 1):
        opt = kpcg.default_options(precision=getattr(kpcg, precision), inner_f64=inner_f64,
                                   profile=profile)
        with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
            _precond(kpcg, s, kind, n)
            runs = [s.solve(B, tol=1e-10) for _ in range(2)]
        for X, it, info, st in runs:
            assert st == 0 and info.max_rel_res <= 1e-10 and info.outer_steps >= 2
            out.append((X.cpu().numpy(), np.array(it)))
    for X, it in out[1:]:
        assert np.array_equal(X, out[0][0]) and np.array_equal(it, out[0][1])


@pytest.mark.parametrize("precision", ["KPCG_FP32_IR", "KPCG_TC_IR"])
@pytest.mark.parametrize("kind", ["nystrom", "none"])
def test_laplace(kpcg, precision, kind):
    n = 700
    p = synthetic.make_problem(n, 6, 7, dist="normal", ell=2.0, noise=1.0)
    y = torch.from_numpy(np.where(np.sin(p.X.astype(np.float64)).sum(1) > 0, 1.0, -1.0)).cuda()
    out = []
    for profile in (0, 1):
        opt = kpcg.default_options(precision=getattr(kpcg, precision), inner_tol=1e-4, profile=profile)
        with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
            _precond(kpcg, s, kind, n)
            s.solve(y, tol=1e-6)  # the handle takes up the profiling option
            f, a, info, st = s.laplace(y, cg_tol=1e-10)
            assert st == 0
            out.append((f.cpu().numpy(), a.cpu().numpy()))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
