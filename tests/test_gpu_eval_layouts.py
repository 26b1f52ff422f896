"""Evaluations of batches between one cluster and a GPU full of them: several candidates
with several parts each in a CTA, partial last CTAs, and the packed uneven layout at its
largest clusters."""
import numpy as np
import pytest

import oracle as O
from paper_2510_25938_gb300 import inputs as I
from tests.helpers import energy_scale, grad_scale_terms, morse_bounds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TERMS = 64          # roundings of a pair term, as in test_gpu_eval_ring.py


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


def _check(lj, sizes, f32, morse, uniform, eps=1.0, sigma=1.0):
    off = I.offsets_from_sizes(sizes)
    x = sigma * np.concatenate([I.fcc_fragments(1, int(k), 0.05, i).reshape(-1)
                                for i, k in enumerate(sizes)])
    if f32:
        x = x.astype(np.float32).astype(np.float64)
    u = 2.0 ** -24 if f32 else 2.0 ** -53
    xd = torch.as_tensor(x, device="cuda").to(torch.float32 if f32 else torch.float64)
    n_cand = len(sizes)
    e = torch.empty(n_cand, dtype=torch.float64, device="cuda")
    g = torch.empty_like(xd)
    kw = dict(uniform_n=int(sizes[0])) if uniform else dict(
        atom_offset=torch.as_tensor(off, device="cuda"), max_n=int(max(sizes)))
    ctx = lj.Ctx(0)
    lj.lj_energy_grad_batched(ctx, xd, e, g, n_cand=n_cand, eps=eps, sigma=sigma,
                              prec=lj.LJ_PREC_FP32 if f32 else lj.LJ_PREC_FP64,
                              potential=lj.LJ_POT_MORSE if morse else lj.LJ_POT_LJ, rho=6.0, **kw)
    torch.cuda.synchronize()
    ctx.close()
    e, g = e.cpu().numpy(), g.double().cpu().numpy()
    er, gr = O.eval_batch(x, n_cand, atom_off=off, eps=eps, sigma=sigma, rho=6.0,
                          potential=O.OBJ_MORSE if morse else O.OBJ_LJ)
    # every candidate of small batches, else both ends and a stride between
    pick = range(n_cand) if n_cand <= 400 else sorted(
        {*range(60), *range(n_cand - 60, n_cand), *range(0, n_cand, n_cand // 200)})
    for c in pick:
        s = slice(3 * off[c], 3 * off[c + 1])
        if sizes[c] < 2:
            assert e[c] == 0 and not g[s].any()
        elif morse:
            eb, gb = morse_bounds(x[s], eps, sigma, rho=6.0, u=u)
            assert abs(e[c] - er[c]) <= eb, c
            assert (np.abs(g[s] - gr[s]) <= gb + u * np.abs(gr[s])).all(), c
        else:
            assert abs(e[c] - er[c]) <= TERMS * u * energy_scale(x[s], eps, sigma), c
            assert np.linalg.norm(g[s] - gr[s]) <= TERMS * u * grad_scale_terms(x[s], eps, sigma), c


# (N, candidates) of every kind of layout that the rule chooses: packed, packed with parts,
# parts over a CTA, parts over several CTAs
SHAPES = [(2, 1000), (4, 5000), (5, 301), (8, 2501), (13, 203), (13, 3001), (20, 601), (25, 5003),
          (30, 601), (38, 41), (38, 801), (45, 2501), (60, 43), (60, 1201), (100, 11), (100, 301),
          (150, 151), (300, 11), (300, 61)]


@pytest.mark.parametrize("f32,morse", [(True, False), (False, False), (True, True), (False, True)])
@pytest.mark.parametrize("n,n_cand", SHAPES)
def test_uniform(lj, n, n_cand, f32, morse):
    _check(lj, [n] * n_cand, f32, morse, True)


@pytest.mark.parametrize("morse", [False, True])
@pytest.mark.parametrize("lo,hi,n_cand", [(0, 8, 5001), (2, 25, 2503), (0, 53, 1501), (0, 60, 1501),
                                          (3, 68, 1203), (3, 69, 1203)])
def test_uneven_packed_fp32(lj, lo, hi, n_cand, morse):
    sizes = I.uneven_sizes(n_cand, lo, hi, hi)
    sizes[-1] = hi
    _check(lj, sizes, True, morse, False)


@pytest.mark.parametrize("f32", [True, False])
@pytest.mark.parametrize("morse", [False, True])
@pytest.mark.parametrize("sizes", [[38] * 4100, [51] * 2000, [127] * 700, [13] * 301, [150] * 3,
                                   "0-9", "2-150"])
def test_eps_and_sigma(lj, sizes, morse, f32):
    """eps = 1.7, sigma (re) = 1.3 in every variant of the kernels."""
    uniform = not isinstance(sizes, str)
    if not uniform:
        lo, hi = (int(v) for v in sizes.split("-"))
        sizes = I.uneven_sizes(14000 if hi < 10 else 60, lo, hi, hi)
    _check(lj, sizes, f32, morse, uniform, eps=1.7, sigma=1.3)
