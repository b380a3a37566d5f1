"""The medium gradient of the levels that are left over where four do not divide a sweep: their terms
are multiplied and summed in FP64, so that a site whose terms cancel keeps what is left of them."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sim_cls():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03172_gb300 import build
    build.build()
    from paper_1704_03172_gb300.sim import LBSim
    return LBSim


# eta^2 = 1/4, tau = 1 and small whole pressures: every population, rho and gsum is exact in FP32, and
# only the products and the sum of the terms are not.  The residuals of times 0 and 1 are chosen so
# that a receiver's terms cancel to their last bits; those of later times are zero.
# Tolerance: the sum is exact to FP64; what is rounded is the result, to FP32 (6e-8).
@pytest.mark.parametrize("nx,ny", [(40, 33), (700, 801)])  # one CTA per SM and two
@pytest.mark.parametrize("nt", [2, 3, 6, 11])
def test_leftover_terms_that_cancel(sim_cls, oracle_mod, nx, ny, nt):
    rng = np.random.default_rng(nx + nt)
    p0 = rng.integers(1, 8, (ny, nx)).astype(np.float32)
    c = np.full((ny, nx), 0.5, np.float32)
    xs = np.arange(3, nx - 3, 5)
    rec = np.stack([xs, 4 + np.arange(len(xs)) * 3 % (ny - 8)], 1).astype(np.int32)
    kw = dict(c_ref=1.0, tau=1.0)
    sim = sim_cls(c, lattice=5, collision="bgk", **kw)
    sim.set_receivers(rec, nt)
    sim.init_pressure(p0)
    sim.record_rho(nt)
    sim.step(nt)
    p = sim.traces(nt).cpu().numpy().astype(np.float64)[:2]
    rho = p / 0.125                       # c_s^2 = eta^2 / 2
    dj = np.zeros((nt, len(rec)), np.float32)
    dj[1] = rng.uniform(1, 2, len(rec))
    # at a receiver: dJ/d(eta^2) = R1 (rho1 / 2 - rho0 / 8) + R0 rho0 / 2
    rest = dj[1].astype(np.float64) * (rho[1] / 2 - rho[0] / 8)
    dj[0] = -rest / (rho[0] / 2)
    left = rest + dj[0].astype(np.float64) * rho[0] / 2
    g = sim.adjoint(dj, nt)[0].cpu().numpy().astype(np.float64)[rec[:, 1], rec[:, 0]]
    sim.close()
    P = oracle_mod.Problem(5, nx, ny, c, receivers=rec, mrt=False, periodic=False, **kw)
    ref = oracle_mod.adjoint(P, oracle_mod.init_pressure(P, p0.astype(np.float64)), nt,
                             dj.astype(np.float64))[0][rec[:, 1], rec[:, 0]]
    np.testing.assert_allclose(ref, left * 2 * 0.5, rtol=1e-6, atol=1e-12)  # dJ/dc = dJ/d(eta^2) 2 eta / c_ref
    assert np.all(np.abs(left) < 1e-6 * np.abs(rest) + 1e-30)
    np.testing.assert_allclose(g, ref, rtol=2e-7, atol=1e-12)
