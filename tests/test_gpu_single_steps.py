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


# D3Q7: the receivers' blocks take no planes' time (a share of the launch's slots once, which left
# 45 of 304 CTAs: 468 us a step against 122 with few receivers; now 143)
def test_many_receivers_leave_the_sweep_its_ctas(sim_cls):
    import torch
    n, times = 256, []
    rng = np.random.default_rng(1)
    for nrec in (64, 160000):
        sim = sim_cls(torch.full((n, n, n), 0.8, device="cuda"), lattice=7, c_ref=1.0)
        sim.set_receivers(rng.integers(0, n, (nrec, 3)), 200)
        sim.init_pressure(None)
        sim.step(21)
        best = 1e9
        for _ in range(5):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record(sim.stream)
            sim.step(20)
            e1.record(sim.stream)
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        times.append(best)
        sim.close()
    assert times[1] < 2 * times[0], times


# and those of both steps are recorded, in more blocks than the sweep has slots
def test_many_receivers_are_recorded(sim_cls):
    import torch
    nx, ny, nz, nrec, steps = 256, 250, 256, 170000, 5
    rng = np.random.default_rng(2)
    rec = np.stack([rng.integers(0, n, nrec) for n in (nx, ny, nz)], 1)
    g0, out = torch.randn(7, nz, ny, nx, device="cuda"), []
    for how in ("direct", "auto"):
        sim = sim_cls(torch.full((nz, ny, nx), 0.8, device="cuda"), lattice=7, c_ref=1.0, tau=0.7,
                      step_kernel=how)
        sim.set_receivers(rec, steps)
        sim.set_state(g0)
        before = sim.info()[6]
        sim.step(steps)
        assert sim.info()[6] - before == (steps if how == "direct" else 3)
        out.append(sim.traces(steps).clone())
        sim.close()
    assert torch.equal(out[0], out[1])


# flat and periodic D3Q7 grids, and many receivers on small ones
@pytest.mark.parametrize("storage,nx,ny,nz,boundary,nrec,launches", [
    ("bf16", 238, 68, 129, "zero", 10, 8), ("bf16", 208, 139, 74, "periodic", 10, 8),
    ("bf16", 208, 227, 82, "periodic", 10, 8), ("bf16", 192, 103, 417, "periodic", 10, 8),
    ("bf16", 128, 128, 128, "periodic", 10, 8), ("f32", 184, 254, 62, "periodic", 10, 8),
    ("bf16", 256, 256, 256, "zero", 60000, 8), ("f32", 135, 229, 106, "zero", 100000, 8),
    ("bf16", 96, 96, 96, "zero", 10, 4), ("bf16", 112, 294, 301, "zero", 10, 4),
    ("bf16", 164, 211, 179, "periodic", 10, 4), ("f32", 135, 229, 106, "zero", 1000, 4),
    ("f32", 256, 256, 256, "zero", 160000, 4)])
def test_d3q7_shapes(sim_cls, storage, nx, ny, nz, boundary, nrec, launches):
    assert _launches(sim_cls, (nz, ny, nx), [8], nrec, lattice=7, storage=storage,
                     boundary=boundary) == launches


# odd periodic FP32 rows: the seam costs less there, but not nothing
@pytest.mark.parametrize("lattice,nx,ny,boundary,calls,launches", [
    (9, 297, 4006, "periodic", [8], 8), (9, 1183, 1183, "periodic", [8], 8),
    (9, 1415, 1413, "periodic", [8], 2), (9, 1184, 1183, "periodic", [8], 2), (9, 1183, 1183, "zero", [8], 2),
    (5, 1923, 1924, "periodic", [2, 3], 5), (5, 1923, 1924, "periodic", [8], 2),
    (5, 1924, 1924, "periodic", [2, 3], 3), (5, 2345, 2345, "periodic", [2, 3], 3)])
def test_seam_of_odd_fp32_rows(sim_cls, lattice, nx, ny, boundary, calls, launches):
    assert _launches(sim_cls, (ny, nx), calls, lattice=lattice, tau=0.6, boundary=boundary) == launches


# D2Q5 grids on tiles: two steps alone do not pay for a launch of tiles
@pytest.mark.parametrize("storage,nx,ny,fused", [("f32", 614, 117, 2), ("bf16", 991, 996, 2),
                                                  ("f32", 1900, 557, 3)])  # (eight: 4 and 4)
def test_two_steps_of_a_small_grid(sim_cls, storage, nx, ny, fused):
    kw = dict(storage=storage, boundary="periodic", collision="bgk")
    assert _launches(sim_cls, (ny, nx), [2, 2, 1], **kw) == 5
    assert _launches(sim_cls, (ny, nx), [3, 8], **kw) == fused
