"""The Nystrom apply on more rows than 65535 of its longest row ranges.

One inducing point u: P^-1 r = (r - k (k.r) / (noise + k.k)) / noise with k = K_XU, s^2 = 1.
k.k is of the size of n, so the formula's FP64 rounding, 2^-53 per entry and in sums of a few
thousand partials, stays below 1e-12 of r / noise.
"""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("c", [1, 2])
def test_fp64_apply_long(c):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    n, noise = 65535 * 512 + 1000, 0.1
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(n, 1, generator=g, device="cuda").clamp_(-4.0, 4.0)
    R = torch.randn(c, n, generator=g, device="cuda", dtype=torch.float64).t()
    opt = kpcg.default_options(precision=kpcg.KPCG_FP64)
    with kpcg.Solver(X, [0.0, 0.0], noise, options=opt) as s:
        s.precond(kpcg.KPCG_PREC_NYSTROM, 1, [n // 2])
        Z = s.precond_apply(R)
    x = X[:, 0].double()
    k = torch.exp(-0.5 * (x - x[n // 2]) ** 2)
    M = noise + (k * k).sum()
    for j in range(c):
        r = R[:, j]
        ref = (r - k * ((k * r).sum() / M)) / noise
        assert ((Z[:, j] - ref).abs().max() <= 1e-12 * ref.abs().max()).item()
