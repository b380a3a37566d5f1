"""Values that overflow on their way out of a zero-ghost grid: lost across the face, as with one step
per launch, and not brought back by the launches of several steps, which compute sites beyond it too.

Sites along the four faces hold populations of up to 2.6e38, so that what they send out is infinite while
what they keep is not.  States are equal bit for bit, NaN for NaN."""
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


# Pulled populations (the bits of FP32 values, exact in BF16) of a site at each face whose collision
# sends an infinite value out through it and finite ones everywhere else, and which stays finite for the
# steps that follow; tau = 1/2 and 0.505 (D2Q5), 0.505 (D2Q9), c = c_ref.  D2Q5 has none at the top.
HOT = {5: dict(left=[0x7d4c0000, 0xff200000, 0x7eec0000, 0x7eb80000, 0x7f1c0000],
               right=[0xfd780000, 0xfe9c0000, 0xff0c0000, 0x7f240000, 0xff0c0000],
               bottom=[0xfd5c0000, 0xff000000, 0x7f100000, 0xff1c0000, 0xfec00000]),
       9: dict(left=[0xfeec0000, 0xfcf00000, 0xfed40000, 0x7f700000, 0x7e080000, 0x7e180000, 0xfeb00000,
                     0xff380000, 0x7ce80000],
               right=[0xff500000, 0x7f140000, 0xfe380000, 0x7e000000, 0xfeb40000, 0xfeac0000, 0x7e5c0000,
                      0x7e9c0000, 0xfe800000],
               bottom=[0x7e900000, 0xfe440000, 0xfe240000, 0x7d8c0000, 0xff3c0000, 0x7df40000, 0xfdec0000,
                       0x7f140000, 0x7eec0000],
               top=[0xfeb00000, 0x7c4c0000, 0x7f2c0000, 0x7d940000, 0x7ed80000, 0xff180000, 0xfeb00000,
                    0xfe240000, 0x7d580000])}


def _sites(s):
    return dict(left=s[:, 15:-15:30, 0], right=s[:, 20:-15:30, -1], bottom=s[:, 0, 15:-15:30],
                top=s[:, -1, 20:-15:30])


def _state(Q, nx, ny):
    import torch
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    s = torch.randn(Q, ny, nx, device="cuda", generator=g)
    for face, bits in HOT[Q].items():
        _sites(s)[face][:] = torch.tensor(np.array(bits, np.uint32).view(np.float32)).cuda()[:, None]
    return s


# (steps; the first, from a pulled state, goes alone)
@pytest.mark.parametrize("Q,tau,storage,nx,ny,steps,launches", [
    (5, 0.5, "f32", 130, 97, 4, 2), (5, 0.505, "f32", 301, 203, 5, 2),  # tiles
    (5, 0.505, "bf16", 131, 100, 4, 2),
    (5, 0.505, "f32", 2011, 1800, 5, 2), (5, 0.505, "bf16", 2010, 1801, 5, 2),  # wavefront
    (5, 0.5, "f32", 2700, 2100, 7, 2),  # six steps
    (9, 0.505, "f32", 1531, 703, 5, 2), (9, 0.505, "bf16", 1200, 703, 3, 2)])
@pytest.mark.parametrize("sponge", [0, 7])
def test_overflow_leaves_through_the_faces(sim_cls, Q, tau, storage, nx, ny, steps, launches, sponge):
    import torch
    g0, out = _state(Q, nx, ny), []
    for how in ("direct", "auto"):
        sim = sim_cls(np.ones((ny, nx), np.float32), lattice=Q, tau=tau, storage=storage,
                      boundary="zero", sponge_width=sponge, sponge_sigma_max=1e-3, c_ref=1.0,
                      step_kernel=how)
        sim.set_state(g0)
        before = sim.info()[6]
        sim.step(steps)
        assert sim.info()[6] - before == (steps if how == "direct" else launches)
        out.append(sim.state().clone())
        sim.close()
    for face in HOT[Q]:  # (some of the sites stayed finite: what left them is gone)
        assert torch.isfinite(_sites(out[0])[face]).all(0).any(), face
    torch.testing.assert_close(out[1], out[0], rtol=0, atol=0, equal_nan=True)
