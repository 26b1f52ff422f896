"""Histories too long for the usual place beside the pair buffer: lbfgs_minimize_batched_noalloc
keeps them on chip where two CTAs still fit on an SM, and gives the results of
lbfgs_minimize_batched, which has them in its workspace."""
import numpy as np
import pytest

from paper_2510_25938_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


# (N, m) on both sides of every step of the ring's chunk (128 atoms: m = 27, 28 .. 32; 256: 13 .. 17)
@pytest.mark.parametrize("n,m", [(128, 24), (128, 27), (128, 28), (128, 30), (128, 32), (65, 32),
                                 (100, 31), (256, 12), (256, 13), (256, 14), (256, 15), (256, 16),
                                 (256, 17), (129, 16)])
@pytest.mark.parametrize("prec", [2, 0])
def test_same_results(lj, n, m, prec):
    n_cand = 330                       # more than two CTAs an SM
    x0 = torch.as_tensor(I.fcc_fragments(n_cand, n, 0.03, n).reshape(-1), device="cuda")
    got = []
    for noalloc in (False, True):
        x = x0.clone()
        e = torch.empty(n_cand, dtype=torch.float64, device="cuda")
        st = torch.empty(n_cand, dtype=torch.int32, device="cuda")
        kw = dict(n_cand=n_cand, uniform_n=n,
                  params=lj.LbfgsParams(m=m, prec=prec, gtol=1e-5, max_iter=40))
        if noalloc:
            lj.lbfgs_minimize_batched_noalloc(x, e, st, **kw)
        else:
            ctx = lj.Ctx(0)
            lj.lbfgs_minimize_batched(ctx, x, e, st, **kw)
            torch.cuda.synchronize()
            ctx.close()
        got.append([v.cpu().numpy() for v in (x, e, st)])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
