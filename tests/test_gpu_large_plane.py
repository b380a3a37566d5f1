"""D3Q7 grids whose planes hold more than 2^31 sites: two steps per launch against one, bit for bit.

Rows beyond the 2^31st site of a plane lie further from its start than 32 bits reach.  A source and
receivers around that row; 60 GB of BF16 populations."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_fused_steps_beyond_2_31_sites_of_a_plane():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 110 << 30:
        pytest.skip("needs 110 GB of free device memory")
    from paper_1704_03172_gb300 import build
    build.build()
    from paper_1704_03172_gb300.sim import LBSim
    nx, ny, steps = 992, 2170000, 9  # (rows of less than 1024 sites: the register-streaming step)
    row = (1 << 31) // nx            # the first whose offset needs more than 32 bits
    rng = np.random.default_rng(1)
    rec = np.stack([rng.integers(480, 500, 300), rng.integers(row - 8, row + 9, 300), np.zeros(300)], 1)
    rec = np.concatenate([rec, [(490, 0, 0), (490, ny - 1, 0)]]).astype(np.int32)
    c = torch.full((1, ny, nx), 0.7, device="cuda")
    torch.cuda.synchronize()
    out = []
    for how, launches in (("direct", steps), ("auto", 1 + 4)):
        sim = LBSim(c, lattice=7, storage="bf16", c_ref=1.0, step_kernel=how)
        sim.set_source(490, row, 0, 1.0 + np.arange(steps))
        sim.set_receivers(rec, steps)
        sim.init_pressure(None)
        before = sim.info()[6]
        sim.step(steps)
        assert sim.info()[6] - before == launches
        out.append(sim.traces(steps).cpu().numpy())
        sim.close()
        torch.cuda.empty_cache()
    assert np.count_nonzero(out[0].any(0)) > 50  # receivers that the wave has reached
    np.testing.assert_array_equal(out[0], out[1])
