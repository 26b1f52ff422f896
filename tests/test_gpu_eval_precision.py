"""FP32 evaluations of large clusters: a gradient in a large batch, whose candidates have a
thread per atom group, is as exact as in a small one, whose sums are split over
many threads."""
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


@pytest.mark.parametrize("n,n_cand", [(400, 800), (600, 700)])
def test_fp32_gradient_error_does_not_depend_on_the_batch(lj, n, n_cand):
    """Relative errors against the FP64 evaluation of the same inputs.  Both are means
    over 10^5 components and more (0.3% of sampling), so that 10% is left for the
    different splits; one sum over all atoms was 25 to 40% worse."""
    few = 60
    x = I.fcc_fragments(n_cand, n, 0.05, 1).reshape(-1).astype(np.float32)
    xd = torch.as_tensor(x, device="cuda")
    e = torch.empty(n_cand, dtype=torch.float64, device="cuda")
    ctx = lj.Ctx(0)

    def gradient(count, dtype):
        xc = xd[:3 * n * count].to(dtype)
        g = torch.empty_like(xc)
        prec = lj.LJ_PREC_FP32 if dtype == torch.float32 else lj.LJ_PREC_FP64
        lj.lj_energy_grad_batched(ctx, xc, e, g, n_cand=count, uniform_n=n, prec=prec)
        return g.double()

    exact = gradient(n_cand, torch.float64)
    many, part = gradient(n_cand, torch.float32), gradient(few, torch.float32)
    torch.cuda.synchronize()
    ctx.close()
    exact_few = exact[:part.numel()]
    err_many = (many - exact).norm() / exact.norm()
    err_few = (part - exact_few).norm() / exact_few.norm()
    assert err_many <= 1.1 * err_few
