"""The fixed-point tensor-core product behind the FP64 products.

matvec_f64 impl 0 and 1 take it (impl 1 for d > 10, three and more columns, or few
rows) while the scaled inputs stay in its range, else the FP64 or double-float
kernels.  Each result is compared with the oracle column by column, against
2^-46 |K_y| |V|: the entries are good to 2^-50 or better and the double-float ones
to 2^-44 of the largest, the sums of up to 1100 terms (the oracle's too) round at
2^-53 sqrt(n) or better.
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


def _check(kpcg, p, V, impl, tol=2.0 ** -46, noise=None):
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    V2 = V.reshape(p.n, -1)
    ref = oracle.kyv(p.X, ell, s2, p.noise, V2)
    big = oracle.kyv(p.X, ell, s2, p.noise, np.abs(V2))
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, ard=p.ard) as s:
        # a wider leading dimension than n
        buf = torch.full((V2.shape[1], p.n + 5), float("nan"), dtype=torch.float64, device="cuda")
        buf[:, :p.n] = torch.from_numpy(np.ascontiguousarray(V2.T)).cuda()
        out = torch.full((V2.shape[1], p.n + 3), 7.0, dtype=torch.float64, device="cuda")
        s.matvec_f64(buf[:, :p.n].t(), impl=impl, out=out[:, :p.n].t())
        assert bool((out[:, p.n:] == 7.0).all())
        O = out[:, :p.n].t().cpu().numpy()
    for k in range(V2.shape[1]):
        assert np.linalg.norm(O[:, k] - ref[:, k]) <= tol * np.linalg.norm(big[:, k]), k


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("n,d,c", [
    (1, 1, 1), (2, 16, 2), (63, 3, 3), (64, 8, 1), (65, 12, 8), (127, 13, 9), (128, 8, 2),
    (129, 16, 16), (193, 11, 17), (1000, 8, 24), (1025, 5, 25), (1100, 9, 49), (1100, 14, 1)])
def test_sizes_and_columns(kpcg, impl, n, d, c):
    p = synthetic.make_problem(n, d, 7, dist="normal", ell="loguniform", s2=1.7, noise=1e-3)
    _check(kpcg, p, synthetic.rng(8).standard_normal((n, c)), impl)


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("span", [1e-4, 1.0, 9.0, 30.0, 400.0])
def test_range_of_the_inputs(kpcg, impl, span):
    """From inputs that all coincide to ones beyond the fixed-point range (the scaled
    inputs reach about 0.85 span / 2)."""
    p = synthetic.make_problem(600, 4, 9, dist="uniform", ell=1.0, noise=1e-3)
    p.X = np.ascontiguousarray(p.X * np.float32(span))
    p.X[5] = p.X[300]  # a repeated point
    # the levels dropped at a scale S cost 2^-59 S^2 (S <= 8 for impl 0, 64 for impl 1)
    _check(kpcg, p, synthetic.rng(8).standard_normal((600, 3)), impl,
           2.0 ** -46 if impl == 0 else 2.0 ** -43)


@pytest.mark.parametrize("impl", [0, 1])
def test_scales_of_the_columns(kpcg, impl):
    p = synthetic.make_problem(500, 8, 3, dist="normal", ell=2.0, noise=1e-2)
    V = synthetic.rng(4).standard_normal((500, 6))
    V[:, 1] *= 1e300
    V[:, 2] *= 1e-300
    V[:, 3] = 0.0
    V[:, 4] = 1.0
    V[:, 5] *= np.exp(8.0 * synthetic.rng(5).standard_normal(500))
    V[:, 1] /= 1e3
    with np.errstate(over="ignore"):
        ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
        ref = oracle.kyv(p.X, ell, s2, p.noise, V)
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        O = s.matvec_f64(torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t(), impl=impl).cpu().numpy()
    for k in range(6):
        # the digits of a column are cut 2^-56 below its largest value
        bound = 2.0 ** -46 * (np.abs(V[:, k]).sum() + 500 * np.abs(V[:, k]).max())
        assert np.abs(O[:, k] - ref[:, k]).max() <= bound, k


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_values_that_are_not_finite(kpcg, impl, bad):
    p = synthetic.make_problem(300, 6, 3, dist="normal", ell=2.0, noise=1e-2)
    V = synthetic.rng(4).standard_normal((300, 3))
    V[17, 1] = bad
    ell, s2 = oracle.split_theta(p.log_theta, p.d, p.ard)
    good = oracle.kyv(p.X, ell, s2, p.noise, V[:, [0, 2]])
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        O = s.matvec_f64(torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t(), impl=impl).cpu().numpy()
    assert np.abs(O[:, [0, 2]] - good).max() <= 1e-11
    assert np.isnan(O[:, 1]).all() if np.isnan(bad) else (O[:, 1] == bad).all()


def test_solve_replays_it_from_a_graph(kpcg):
    """The double-float PCG at d = 14 iterates with it, plainly and from a graph."""
    p = synthetic.make_problem(700, 14, 3, dist="normal", ell=3.0, noise=1e-2)
    y = torch.from_numpy(p.y).cuda()
    out = []
    for profile in (0, 1):
        opt = kpcg.default_options(precision=kpcg.KPCG_DF64, profile=profile)
        with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise, options=opt) as s:
            x, _, info, st = s.solve(y, tol=1e-10)
            assert st == 0 and info.max_rel_res <= 1e-10
            out.append(x.cpu().numpy())
    assert np.array_equal(out[0], out[1])
