"""Morse evaluations keep the precision of their type: the exponent's error is
what rho amplifies."""
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


def test_fp64_dimers(lj):
    """Dimers on an axis at the steepest range, rho = 64: the root of r^2 is the coordinate
    itself, the exponent one rounding, exp is within an ulp (CUDA's bound: 2 u) and every
    other operation adds at most u."""
    rho, u = 64.0, 2.0 ** -53
    z = np.random.default_rng(3).uniform(0.95, 1.2, 100_000)
    x = np.zeros((z.size, 2, 3))
    x[:, 1, 2] = z
    xd = torch.as_tensor(x.reshape(-1), device="cuda")
    e = torch.empty(z.size, dtype=torch.float64, device="cuda")
    g = torch.empty_like(xd)
    ctx = lj.Ctx(0)
    lj.lj_energy_grad_batched(ctx, xd, e, g, n_cand=z.size, uniform_n=2, prec=lj.LJ_PREC_FP64,
                              potential=lj.LJ_POT_MORSE, rho=rho)
    torch.cuda.synchronize()
    ctx.close()
    m = np.exp((rho - rho * z).astype(np.longdouble))
    er, gr = m * (m - 2), 2 * rho * m * (m - 1)
    e = e.cpu().numpy()
    g = g.cpu().numpy().reshape(-1, 2, 3)[:, :, 2]
    # m off by 2 u, m - 2 and m - 1 rounded, two (gradient: four) products and a quotient
    assert (np.abs(e - er) <= u * m * (2 * m + 2 * np.abs(m - 2) + 2 * np.abs(m - 2))).all()
    bound = 2 * rho * u * m * (2 * m + 2 * np.abs(m - 1) + 5 * np.abs(m - 1))
    assert (np.abs(g[:, 0] - gr) <= bound).all() and (g[:, 1] == -g[:, 0]).all()


def test_fp32_energies_have_no_bias(lj):
    """The exponent's slope (rho / re) log2 e is not an FP32 number: its rounding, 4.1e-8 of
    it at rho = 6, would move every energy the same way.  Over many dimers the other
    roundings average out: the error of the exponent ln m per unit of it stays below
    half of that."""
    rho = 6.0
    z = np.random.default_rng(4).uniform(1.2, 1.8, 400_000).astype(np.float32)
    x = np.zeros((z.size, 2, 3), dtype=np.float32)
    x[:, 1, 2] = z
    e = torch.empty(z.size, dtype=torch.float64, device="cuda")
    ctx = lj.Ctx(0)
    lj.lj_energy_grad_batched(ctx, torch.as_tensor(x.reshape(-1), device="cuda"), e, None,
                              n_cand=z.size, uniform_n=2, prec=lj.LJ_PREC_FP32,
                              potential=lj.LJ_POT_MORSE, rho=rho)
    torch.cuda.synchronize()
    ctx.close()
    t = rho * (1.0 - z.astype(np.float64))               # -1.2 .. -4.8
    m = 1.0 - np.sqrt(1.0 + e.cpu().numpy())            # m (m - 2) = E, m < 1
    slope = np.polyfit(t, np.log(m) - t, 1)[0]
    assert abs(slope) <= 2e-8
