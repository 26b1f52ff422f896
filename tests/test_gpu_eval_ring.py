"""lj_energy_grad_batched against the oracle where its layout changes: groups
with missing atoms, split last shifts, several candidates a CTA, several parts
and CTAs a candidate, unaligned groups, and the ends of the FP64 range."""
import numpy as np
import pytest

import oracle as O
from paper_2510_25938_gb300 import inputs as I
from tests.helpers import energy_scale, grad_scale_terms, morse_bounds

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# per-term bounds against the no-cancellation scales: 64 roundings of the
# arithmetic's unit (r2 ~4, its inverse 2, the 6th and 12th powers multiply)
TERMS = 64
RHO = 6.0


@pytest.fixture(scope="module")
def lj():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2510_25938_gb300 import build
    build.build()
    from paper_2510_25938_gb300 import lj_bh
    return lj_bh


def _evaluate(lj, x, n_cand, n, off, f32, morse, shift):
    dt = torch.float32 if f32 else torch.float64
    buf = torch.zeros(x.size + shift, dtype=dt, device="cuda")
    out = torch.full_like(buf, 7.0)
    buf[shift:] = torch.as_tensor(x, dtype=dt)
    e = torch.empty(n_cand, dtype=torch.float64, device="cuda")
    kw = dict(uniform_n=n) if off is None else dict(
        atom_offset=torch.as_tensor(off, device="cuda"), max_n=n)
    ctx = lj.Ctx(0)
    lj.lj_energy_grad_batched(ctx, buf[shift:], e, out[shift:], n_cand=n_cand,
                              prec=lj.LJ_PREC_FP32 if f32 else lj.LJ_PREC_FP64,
                              potential=lj.LJ_POT_MORSE if morse else lj.LJ_POT_LJ, rho=RHO, **kw)
    torch.cuda.synchronize()
    ctx.close()
    assert (out[:shift] == 7.0).all()
    return e.cpu().numpy(), out[shift:].double().cpu().numpy()


def _check(x, off, e, g, f32, morse):
    u = 2.0 ** -24 if f32 else 2.0 ** -53
    er, gr = O.eval_batch(x, off.size - 1, atom_off=off,
                          potential=O.OBJ_MORSE if morse else O.OBJ_LJ, rho=RHO)
    for c in range(off.size - 1):
        s = slice(3 * off[c], 3 * off[c + 1])
        if off[c + 1] - off[c] < 2:
            assert e[c] == 0 and not g[s].any()
            continue
        if morse:
            eb, gb = morse_bounds(x[s], rho=RHO, u=u)
            assert abs(e[c] - er[c]) <= eb, c
            assert (np.abs(g[s] - gr[s]) <= gb + u * np.abs(gr[s])).all(), c
        else:
            assert abs(e[c] - er[c]) <= TERMS * u * energy_scale(x[s]), c
            assert np.linalg.norm(g[s] - gr[s]) <= TERMS * u * grad_scale_terms(x[s]), c


def _starts(n, count, seed):
    """Jittered fcc fragments: well separated atoms at every size."""
    return I.fcc_fragments(count, n, 0.05, seed).reshape(-1)


# (N, candidates): one group and fewer; the FP32 groups of eight (N = 38) and
# of four; even rings (a split shift); the sizes at which the FP64 group grows
# (512, 513, 768, 769) and the largest; few candidates (parts, clusters of CTAs)
UNIFORM = [(1, 40000), (2, 40000), (3, 40000), (7, 30000), (8, 20000), (38, 4000), (40, 4001),
           (41, 3000), (51, 2000), (52, 2000), (127, 700), (129, 700), (300, 300), (512, 160),
           (513, 160), (768, 40), (769, 40), (1024, 160), (13, 1), (38, 1), (38, 200), (150, 3),
           (500, 2), (1024, 1), (257, 30)]


@pytest.mark.parametrize("f32,morse", [(True, False), (False, False), (True, True), (False, True)])
@pytest.mark.parametrize("n,n_cand", UNIFORM)
def test_eval_ring_uniform(lj, n, n_cand, f32, morse):
    x = _starts(n, n_cand, n)
    if f32:
        x = x.astype(np.float32).astype(np.float64)
    e, g = _evaluate(lj, x, n_cand, n, None, f32, morse, 0)
    # every candidate where that is quick, else the first and last tiles
    pick = np.arange(n_cand)
    if n_cand * n * n > 4_000_000:
        pick = np.unique(np.r_[:min(n_cand, 70), max(0, n_cand - 70):n_cand])
        pick = pick[:max(2, 12_000_000 // (n * n))] if n > 400 else pick
    at = (pick[:, None] * 3 * n + np.arange(3 * n)).reshape(-1)
    _check(x[at], np.arange(pick.size + 1) * n, e[pick], g[at], f32, morse)


@pytest.mark.parametrize("f32,morse", [(True, False), (False, False), (True, True), (False, True)])
@pytest.mark.parametrize("lo,hi,n_cand", [(0, 20, 70), (2, 150, 60), (90, 400, 12), (500, 1024, 3),
                                          (0, 9, 14000), (3, 52, 5000)])
def test_eval_ring_uneven(lj, lo, hi, n_cand, f32, morse):
    sizes = I.uneven_sizes(n_cand, lo, hi, hi)
    sizes[-1] = hi
    off = I.offsets_from_sizes(sizes)
    x = np.concatenate([_starts(int(k), 1, i) for i, k in enumerate(sizes)])
    if f32:
        x = x.astype(np.float32).astype(np.float64)
    e, g = _evaluate(lj, x, n_cand, hi, off, f32, morse, 0)
    _check(x, off, e, g, f32, morse)


@pytest.mark.parametrize("f32", [True, False])
@pytest.mark.parametrize("n_cand", [50, 12000])
def test_eval_ring_bad_size(lj, n_cand, f32):
    """A candidate above max_n gets a NaN energy and no gradient; the others are
    what they are without it."""
    sizes = np.full(n_cand, 5)
    sizes[7] = 12
    off = I.offsets_from_sizes(sizes)
    x = np.concatenate([_starts(int(k), 1, i) for i, k in enumerate(sizes)])
    if f32:
        x = x.astype(np.float32).astype(np.float64)
    e, g = _evaluate(lj, x, n_cand, 9, off, f32, False, 0)
    assert np.isnan(e[7]) and (g[3 * off[7]:3 * off[8]] == 7.0).all()
    keep = np.r_[0:7, 8:n_cand]
    xs = np.concatenate([x[3 * off[c]:3 * off[c + 1]] for c in keep])
    gs = np.concatenate([g[3 * off[c]:3 * off[c + 1]] for c in keep])
    _check(xs, np.arange(keep.size + 1) * 5, e[keep], gs, f32, False)


@pytest.mark.parametrize("n", [38, 40, 100])
@pytest.mark.parametrize("shift", [1, 2, 3, 4])
def test_eval_ring_unaligned_buffers(lj, n, shift):
    x = _starts(n, 3000, n).astype(np.float32).astype(np.float64)
    base = _evaluate(lj, x, 3000, n, None, True, False, 0)
    got = _evaluate(lj, x, 3000, n, None, True, False, shift)
    assert np.array_equal(base[0], got[0]) and np.array_equal(base[1], got[1])


def test_eval_f64_range(lj):
    """Dimers from overflow to underflow of r^2 and of its inverse."""
    r = np.array([1e-60, 1e-30, 0.3, 1.0, 1.5, 1e10, 1e60, 1e154, 1e160])
    x = np.zeros((r.size, 2, 3))
    x[:, 1, 1] = r
    e, g = _evaluate(lj, x.reshape(-1), r.size, 2, None, False, False, 0)
    assert not np.isfinite(e[:2]).any()
    for k in range(2, 5):
        s6 = r[k] ** -6
        assert abs(e[k] - 4 * s6 * (s6 - 1)) <= TERMS * 2.0 ** -53 * 4 * s6 * (s6 + 1)
        ref = 24 * s6 * (2 * s6 - 1) / r[k]
        assert abs(-g[6 * k + 4] - ref) <= TERMS * 2.0 ** -53 * 24 * s6 * (2 * s6 + 1) / r[k]
        assert g[6 * k + 1] == -g[6 * k + 4]
    assert np.allclose(e[5:7], -4 * r[5:7] ** -6, rtol=1e-14, atol=0)
    assert (e[7:] == 0).all() and np.isfinite(g[30:]).all()
