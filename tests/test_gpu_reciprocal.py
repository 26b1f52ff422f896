"""The FP64 pair reciprocal is the correctly rounded one.  Dimers on an axis, far
enough apart (r > 512: s^6 < 2^-54) that s^6 - 1 is -1: their energy is -4 s^6 and
their force 24 (s^2 s^6) r, products of the reciprocal alone that numpy repeats
whatever operations are fused, so both are equal bit for bit."""
import numpy as np
import pytest

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


def _distances():
    """Random significands over many exponents, and r^2 next to powers of two."""
    rng = np.random.default_rng(5)
    parts = [np.exp(rng.uniform(np.log(1024.0), np.log(1e8), 300_000))]
    for to in (0.0, np.inf):
        edge = np.sqrt(2.0 ** np.arange(21.0, 41.0))
        for _ in range(40):
            parts.append(edge)
            edge = np.nextafter(edge, to)
    return np.concatenate(parts)


def _reference(z):
    r2 = z * z
    s2 = 1.0 / r2                       # numpy's division rounds correctly
    s6 = s2 * s2 * s2
    # the significand of all ones is the reciprocal's one exception
    frac = r2.view(np.uint64) & np.uint64((1 << 52) - 1)
    return -4.0 * s6, -24.0 * ((s2 * s6) * z), frac != np.uint64((1 << 52) - 1)


def test_evaluation(lj):
    z = _distances()
    e_ref, f_ref, ok = _reference(z)
    x = np.zeros((z.size, 2, 3))
    x[:, 1, 2] = z
    xd = torch.as_tensor(x.reshape(-1), device="cuda")
    e = torch.empty(z.size, dtype=torch.float64, device="cuda")
    g = torch.empty_like(xd)
    ctx = lj.Ctx(0)
    lj.lj_energy_grad_batched(ctx, xd, e, g, n_cand=z.size, uniform_n=2, prec=lj.LJ_PREC_FP64)
    torch.cuda.synchronize()
    ctx.close()
    g = g.cpu().numpy().reshape(-1, 2, 3)[:, :, 2]
    assert np.array_equal(e.cpu().numpy()[ok], e_ref[ok])
    assert np.array_equal(g[ok, 0], f_ref[ok]) and np.array_equal(g[ok, 1], -f_ref[ok])


def test_minimiser(lj):
    z = _distances()
    e_ref, _, ok = _reference(z)
    x = np.zeros((z.size, 2, 3))
    x[:, 1, 2] = z
    xd = torch.as_tensor(x.reshape(-1), device="cuda")
    e = torch.empty(z.size, dtype=torch.float64, device="cuda")
    st = torch.empty(z.size, dtype=torch.int32, device="cuda")
    ctx = lj.Ctx(0)
    lj.lbfgs_minimize_batched(ctx, xd, e, st, n_cand=z.size, uniform_n=2,
                              params=lj.LbfgsParams(prec=lj.LJ_PREC_FP64, max_iter=0))
    torch.cuda.synchronize()
    ctx.close()
    assert np.array_equal(e.cpu().numpy()[ok], e_ref[ok])
