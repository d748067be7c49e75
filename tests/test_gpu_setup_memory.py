"""What a preconditioner holds after its set-up: K_XU (FP32 pairs) and a few m x m matrices,
not the row blocks of digits the set-up's sum works on (82 MB at this size).  A batch
keeps one preconditioner per problem."""
import numpy as np
import pytest

import synthetic

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_setup_gives_its_scratch_back():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1602_06693_gb300 as kpcg
    from paper_1602_06693_gb300 import build
    build.build()
    n, m = 20000, 256
    p = synthetic.make_problem(n, 6, 5, dist="normal", ell=1.0, noise=1e-1)
    idx = synthetic.inducing_subset(n, m, seed=3)
    X = torch.from_numpy(p.X).cuda()
    held = []
    for _ in range(2):  # the first time loads the kernels
        with kpcg.Solver(X, p.log_theta, p.noise) as s:
            torch.cuda.synchronize()
            free = torch.cuda.mem_get_info()[0]
            s.precond(kpcg.KPCG_PREC_NYSTROM, m, idx)
            torch.cuda.synchronize()
            held.append(free - torch.cuda.mem_get_info()[0])
    # 41 MB of K_XU, 13 MB of split partials, three m x m matrices and whole 2 MB pages
    assert held[1] <= 8 * n * m + (28 << 20), held
