"""Columns with few values in the FP64 products: a unit vector gives a column of K.

Up to 32 values the product sums FP64 entries, good relative to each entry however small:
its exponent sum t^2 (t = y_i - y_j, y the scaled inputs) comes from inputs with three
roundings each and a sum of d terms, 6 2^-53 |t| (|y_i| + |y_j|) + d 2^-53 t^2, below
2^-50 of sum |t| (|y_i| + |y_j|); entry and sum round a few more times.
"""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LD = np.longdouble


@pytest.mark.parametrize("impl", [0, 1])
@pytest.mark.parametrize("n,d", [(20, 4), (700, 4), (300, 13)])
def test_few_values(impl, n, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    p = synthetic.make_problem(n, d, 7, dist="normal", ell=0.6, s2=1.7, noise=1e-3)
    r = synthetic.rng(8)
    V = np.zeros((n, 7))
    V[0, 0] = 1.0
    V[n - 1, 1] = 1.0
    V[n // 2, 2] = -1e200
    V[r.choice(n, min(n, 31), replace=False), 3] = 1.0 + r.random(min(n, 31))
    V[r.choice(n, min(n, 32), replace=False), 4] = 1.0 + r.random(min(n, 32))
    V[:, 6] = r.standard_normal(n)  # an ordinary column beside them
    with kpcg.Solver(torch.from_numpy(p.X).cuda(), p.log_theta, p.noise) as s:
        Vd = torch.from_numpy(np.ascontiguousarray(V.T)).cuda().t()
        O = [s.matvec_f64(Vd, impl=impl).cpu().numpy() for _ in range(2)]
        W = Vd.clone(memory_format=torch.preserve_format)
        s.matvec_f64(W, impl=impl, out=W)  # in place
    assert np.array_equal(O[0], O[1]) and np.array_equal(O[0], W.cpu().numpy())
    Y = p.X.astype(LD) * np.exp(-LD(p.log_theta[0])) / np.sqrt(LD(2))
    t = Y[:, None, :] - Y[None, :, :]
    K = np.exp(LD(p.log_theta[-1]) - (t ** 2).sum(2)) + LD(p.noise) * np.eye(n)
    a = np.abs(Y) + 0.5  # the library centres the inputs
    rel = 2.0 ** -50 * (8 + (np.abs(t) * (a[:, None] + a[None])).sum(2))
    ref, bound = K @ V.astype(LD), (K * rel) @ np.abs(V).astype(LD)
    assert K.min() < 2.0 ** -100 or n == 20
    for k in range(6):
        bad = np.abs(O[0][:, k] - ref[:, k]) > bound[:, k]
        assert not bad.any(), (k, int(bad.sum()))
    big = K @ np.abs(V[:, 6]).astype(LD)
    assert np.abs(O[0][:, 6] - ref[:, 6]).max() <= 2.0 ** -46 * big.max()
