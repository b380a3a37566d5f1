"""Grids on which one step per launch measured faster than several keep it (fuse_steps in csrc/wave.cu,
sweep3_pays in csrc/sweep3.cu); their neighbours on the other side of each line fuse."""
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


def _launches(sim_cls, shape, calls, nrec=0, **kw):
    """Kernels that steps in calls of the given lengths launch, after one from the initial state."""
    import torch
    sim = sim_cls(torch.full(shape, 0.8, device="cuda"), c_ref=1.0, **kw)
    if nrec:
        rng = np.random.default_rng(nrec)
        sim.set_receivers(np.stack([rng.integers(0, n, nrec) for n in shape[::-1]], 1), sum(calls) + 1)
    sim.init_pressure(None)
    sim.step(1)
    before = sim.info()[6]
    for n in calls:
        sim.step(n)
    sim.sync()
    n = sim.info()[6] - before
    sim.close()
    return n


# 8 steps: FP16 counts its scales' update, and after two steps the launch that mends
@pytest.mark.parametrize("storage,coll,nx,ny,boundary,launches", [
    ("f16", "bgk", 1471, 700, "periodic", 16), ("f16", "mrt", 1493, 2258, "periodic", 16),
    ("f16", "bgk", 1472, 700, "periodic", 12), ("f16", "bgk", 1471, 700, "zero", 12),
    ("bf16", "mrt", 2017, 1861, "periodic", 8), ("bf16", "bgk", 1669, 2200, "periodic", 8),
    ("bf16", "mrt", 2018, 1861, "periodic", 2), ("bf16", "mrt", 2017, 1861, "zero", 2)])
def test_seam_of_odd_16_bit_rows(sim_cls, storage, coll, nx, ny, boundary, launches):
    assert _launches(sim_cls, (ny, nx), [8], storage=storage, collision=coll,
                     boundary=boundary) == launches
