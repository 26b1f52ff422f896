"""Mixed quenches of 257 to 512 atoms have a build for few candidates and one for many, and
in an uneven batch the device chooses: a candidate's result does not depend on it."""
import numpy as np
import pytest

from paper_2510_25938_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KEEP = 6                       # compared candidates of 300 atoms, first in every batch


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


def _quench(lj, noalloc, morse, x, off=None, n=0):
    cand = off.size - 1 if off is not None else x.size // (3 * n)
    kw = dict(uniform_n=n) if off is None else dict(
        atom_offset=torch.as_tensor(off, device="cuda"), max_n=int(np.diff(off).max()))
    kw["params"] = lj.LbfgsParams(m=5, potential=lj.LJ_POT_MORSE if morse else lj.LJ_POT_LJ)
    xd = torch.as_tensor(x, device="cuda").clone()
    e = torch.empty(cand, dtype=torch.float64, device="cuda")
    st = torch.full((cand,), -1, dtype=torch.int32, device="cuda")
    if noalloc:
        lj.lbfgs_minimize_batched_noalloc(xd, e, st, n_cand=cand, **kw)
    else:
        ctx = lj.Ctx(0)
        lj.lbfgs_minimize_batched(ctx, xd, e, st, n_cand=cand, **kw)
        torch.cuda.synchronize()
        ctx.close()
    assert (st == lj.LJ_CAND_CONVERGED).all()
    return xd.cpu().numpy(), e.cpu().numpy()


@pytest.mark.parametrize("noalloc", [False, True])
@pytest.mark.parametrize("morse", [False, True])
def test_same_result_from_either_build(lj, morse, noalloc):
    n = 300
    x = I.fcc_fragments(200, n, 0.04, 9).reshape(-1)
    few, many = x[:3 * n * KEEP], x
    xf, ef = _quench(lj, noalloc, morse, few, n=n)
    xm, em = _quench(lj, noalloc, morse, many, n=n)
    assert np.array_equal(em[:KEEP], ef) and np.array_equal(xm[:xf.size], xf)
    # uneven: few and many of 300 among 200 small ones
    small = I.fcc_fragments(200, 20, 0.04, 9).reshape(-1)
    for big in (KEEP, 200):
        off = I.offsets_from_sizes(np.array([n] * big + [20] * 200))
        xu, eu = _quench(lj, noalloc, morse, np.concatenate([x[:3 * n * big], small]), off)
        assert np.array_equal(eu[:KEEP], ef) and np.array_equal(xu[:xf.size], xf)
