"""The double-float tier of a mixed quench resolves its last line search: it converges, and one
FP64 evaluation confirms it."""
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


@pytest.mark.parametrize("morse", [True, False])
@pytest.mark.parametrize("n,n_cand", [(38, 1500), (150, 800), (400, 800)])
def test_double_float_convergence_is_confirmed(lj, n, n_cand, morse):
    """Displaced fcc fragments.  Energies of the tier are exact to about a fifth of what its
    gradient-only search allows between two points, so that a few trials in a
    thousand are turned away and none of the quenches; 2% of the evaluations are left
    for those that need another FP64 step."""
    x = torch.as_tensor(I.fcc_fragments(n_cand, n, 0.04, 5).reshape(-1), device="cuda")
    e = torch.empty(n_cand, dtype=torch.float64, device="cuda")
    st = torch.empty(n_cand, dtype=torch.int32, device="cuda")
    stats = lj.new_stats()
    ctx = lj.Ctx(0)
    lj.lbfgs_minimize_batched(ctx, x, e, st, stats=stats, n_cand=n_cand, uniform_n=n,
                              params=lj.LbfgsParams(
                                  potential=lj.LJ_POT_MORSE if morse else lj.LJ_POT_LJ, rho=6.0,
                                  switch_gtol=1e-4))
    torch.cuda.synchronize()
    ctx.close()
    assert (st == lj.LJ_CAND_CONVERGED).all()
    assert lj.stats_dict(stats)["evals64"] <= 1.02 * n_cand
