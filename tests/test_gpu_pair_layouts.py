"""The minimiser's evaluations and recursion at the sizes where their layouts
change: half pairs (odd and even N), ring chunks with remainders, tiles, the
chunks of the recursion's vectors and the teams of every bucket."""
import numpy as np
import pytest

import oracle as O
from paper_2510_25938_gb300 import inputs as I
from tests.helpers import energy_scale, morse_bounds, numpy_energy_grad

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [2, 3, 4, 13, 21, 22, 31, 32, 33, 42, 43, 63, 64, 65, 66, 85, 86, 113, 127, 128, 129, 130,
         170, 171, 255, 256, 257]
GTOL = 1e-5       # FP64 energies of these sizes resolve it


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


def _minimise(lj, x, off, hi, team=0, **kw):
    ctx = lj.Ctx(0)
    ctx.set_option(lj.LJ_OPT_LBFGS_TEAM, team)
    n = off.size - 1
    xd = torch.as_tensor(x, device="cuda").clone()
    e = torch.empty(n, dtype=torch.float64, device="cuda")
    st = torch.empty(n, dtype=torch.int32, device="cuda")
    lj.lbfgs_minimize_batched(ctx, xd, e, st, n_cand=n,
                              atom_offset=torch.as_tensor(off, device="cuda"), max_n=hi,
                              params=lj.LbfgsParams(gtol=GTOL, **kw))
    torch.cuda.synchronize()
    ctx.close()
    return xd.cpu().numpy(), e.cpu().numpy(), st.cpu().numpy()


def _batch():
    off = I.offsets_from_sizes(SIZES)
    x = np.concatenate([I.fcc_fragments(1, n, 0.04, n).reshape(-1) for n in SIZES])
    return x, off


@pytest.mark.parametrize("morse", [False, True])
@pytest.mark.parametrize("team", [0, 32, 64, 128, 256, 512])
def test_fp64_energy_of_every_layout(lj, team, morse):
    """No iteration: the FP64 evaluation's energy against the oracle, to 64
    roundings of the terms (no cancellation assumed)."""
    x, off = _batch()
    pot = dict(potential=lj.LJ_POT_MORSE if morse else lj.LJ_POT_LJ, rho=6.0)
    _, e, _ = _minimise(lj, x, off, SIZES[-1], team, prec=lj.LJ_PREC_FP64, max_iter=0, **pot)
    ref, _ = O.eval_batch(x, off.size - 1, atom_off=off, rho=6.0,
                          potential=O.OBJ_MORSE if morse else O.OBJ_LJ)
    for c in range(off.size - 1):
        s = x[3 * off[c]:3 * off[c + 1]]
        tol = morse_bounds(s, rho=6.0, u=2.0 ** -53)[0] if morse else \
            64 * 2.0 ** -53 * energy_scale(s)
        assert abs(e[c] - ref[c]) <= tol, SIZES[c]


@pytest.mark.parametrize("prec", [0, 2])
@pytest.mark.parametrize("team,m", [(0, 10), (0, 1), (0, 2), (0, 32), (32, 10), (64, 3), (128, 10),
                                    (256, 5)])
def test_minima_of_every_layout(lj, prec, team, m):
    """Converged, and the returned points are minima with the returned energies."""
    x, off = _batch()
    xm, e, st = _minimise(lj, x, off, SIZES[-1], team, prec=prec, m=m)
    assert (st == lj.LJ_CAND_CONVERGED).all(), [SIZES[c] for c in np.nonzero(st)[0]]
    for c in range(off.size - 1):
        er, gr = numpy_energy_grad(xm[3 * off[c]:3 * off[c + 1]])
        assert np.abs(gr).max() < GTOL * (1 + 1e-6), SIZES[c]
        assert abs(e[c] - er) <= 1e-12 * abs(er), SIZES[c]
