"""Which launches lb_step takes, by its counter, and the fused forms that only large grids reach: the
D2Q9 BF16 wavefront on periodic grids, six D2Q5 steps at every kind of edge, rho of every level on
the tape, and the wavefront sweep of the adjoint with what is left of it.

Steps are compared with one launch per step bit for bit (csrc/wave.cuh); the adjoint with the FP64
oracle, within 1e-4 in relative L2 as the other FP32 adjoint tests."""
import numpy as np
import pytest

from paper_1704_03172_gb300 import workloads as W

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


def _sim(sim_cls, Q, coll, tau, storage, boundary, nx, ny, sponge, how):
    rng = np.random.default_rng(nx + ny)
    c = np.where(np.arange(ny)[:, None] > ny // 2, 1.0, 0.6) * np.ones((ny, nx))
    sim = sim_cls(c.astype(np.float32), lattice=Q, collision=coll, tau=tau,
                  s=W.mrt_rates(Q, W.DEFAULT_SEED + 2), storage=storage, boundary=boundary,
                  sponge_width=sponge, c_ref=1.0, w_ref=(0.0, 0.01, 0.24), step_kernel=how)
    rec = np.concatenate([np.stack([rng.integers(0, nx, 40), rng.integers(0, ny, 40)], 1),
                          [(0, 0), (nx - 1, ny - 1), (nx - 1, 0), (0, ny - 1)]]).astype(np.int32)
    return sim, rec


def _stepped(sim, steps):
    before = sim.info()[6]
    sim.step(steps)
    return sim.info()[6] - before


# 23 steps: one from the pulled state and 22 in launches of K.  (launches of 6: 6, 6, 6, 4)
@pytest.mark.parametrize("Q,coll,tau,storage,boundary,nx,ny,sponge,launches", [
    (9, "bgk", 0.6, "bf16", "periodic", 1202, 903, 0, 1 + 11),
    (9, "mrt", 0.5, "bf16", "periodic", 1120, 400, 7, 1 + 11),
    (9, "bgk", 0.6, "bf16", "periodic", 2600, 2501, 0, 1 + 6),
    (9, "mrt", 0.5, "bf16", "periodic", 3002, 2200, 9, 1 + 6),
    (5, "bgk", 0.5, "f32", "periodic", 2600, 2300, 0, 1 + 4),
    (5, "bgk", 0.8, "f32", "periodic", 2601, 2300, 6, 1 + 4),
    (5, "bgk", 0.5, "f32", "zero", 2701, 2103, 0, 1 + 4),
    (5, "bgk", 0.8, "f32", "zero", 57, 82001, 5, 1 + 4),
    (5, "mrt", 0.5, "f32", "periodic", 2000, 1803, 6, 1 + 6),
    (5, "mrt", 0.5, "bf16", "periodic", 2000, 1803, 0, 1 + 6)])
def test_large_grids(sim_cls, Q, coll, tau, storage, boundary, nx, ny, sponge, launches):
    import torch
    steps, out = 23, []
    g = torch.Generator(device="cuda").manual_seed(nx)
    g0 = torch.randn(Q, ny, nx, device="cuda", generator=g)
    wav = np.random.default_rng(1).normal(size=steps - 4)
    for how in ("direct", "auto"):
        sim, rec = _sim(sim_cls, Q, coll, tau, storage, boundary, nx, ny, sponge, how)
        sim.set_source(nx // 3, ny // 2, wav)
        sim.set_receivers(rec, steps)
        sim.set_state(g0)
        assert _stepped(sim, steps) == (steps if how == "direct" else launches)
        out.append((sim.state().clone(), sim.traces(steps).clone()))
        sim.close()
    assert torch.equal(out[0][0], out[1][0])
    assert torch.equal(out[0][1], out[1][1])


# The tapes are equal if the gradients are: the same sweep reads them.  launches: 1 + 2 of four, of
# six and four, 1 + 5 of two and (FP16) for each launch the scales after it and the mended launch
@pytest.mark.parametrize("coll,tau,storage,nx,ny,nt,launches", [
    ("mrt", 0.5, "f32", 2011, 1800, 9, 3), ("bgk", 0.5, "f32", 2700, 2100, 11, 3),
    ("bgk", 0.8, "bf16", 2010, 1801, 9, 3), ("mrt", 0.5, "f16", 1031, 489, 11, 2 + 15)])
def test_tape_of_every_level(sim_cls, coll, tau, storage, nx, ny, nt, launches):
    import torch
    out = []
    wav = np.random.default_rng(2).normal(size=nt)
    dj = np.random.default_rng(3).normal(size=(nt, 44)).astype(np.float32)
    p0 = W.gaussian_pulse(nx, ny, nx // 2, ny // 3, 40.0, 1.0).astype(np.float32)
    for how in ("direct", "auto"):
        sim, rec = _sim(sim_cls, 5, coll, tau, storage, "zero", nx, ny, 8, how)
        sim.set_source(nx // 3, ny // 2, wav)
        sim.set_receivers(rec, nt)
        sim.init_pressure(p0)
        sim.record_rho(nt)
        n = _stepped(sim, nt)
        if how == "auto":
            assert n == launches
        out.append([x.clone() for x in sim.adjoint(dj, nt)[:2]])
        sim.close()
    assert out[0][0].abs().max() > 0
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


# D2Q5 grids above the tiles' line, tall and narrow: 9 .. 11 levels are two launches of the wavefront
# sweep and one to three single ones
@pytest.mark.parametrize("coll,boundary,nt,every", [
    ("bgk", "zero", 9, 0), ("mrt", "zero", 11, 6), ("bgk", "periodic", 10, 5), ("mrt", "periodic", 9, 0)])
def test_wavefront_adjoint(sim_cls, oracle_mod, coll, boundary, nt, every):
    nx, ny, tau, sponge = 57, 62000, 0.5, 5 if boundary == "zero" else 0
    sim, rec = _sim(sim_cls, 5, coll, tau, "f32", boundary, nx, ny, sponge, "auto")
    src = (rec[3, 0] + 1) % nx, rec[3, 1]  # next to a receiver
    wav = np.random.default_rng(5).normal(size=nt)
    rng = np.random.default_rng(6)
    p0 = rng.normal(size=(ny, nx)).astype(np.float32)
    sim.set_source(int(src[0]), int(src[1]), wav)
    sim.set_receivers(rec, nt)
    sim.init_pressure(p0)
    sim.checkpoint_every(every) if every else sim.record_rho(nt)
    sim.step(nt)
    dj = rng.normal(size=(nt, len(rec))).astype(np.float32)
    gc, gs, g0 = sim.adjoint(dj, nt, want_g0=True)
    P = oracle_mod.Problem(5, nx, ny, np.where(np.arange(ny)[:, None] > ny // 2, 1.0, 0.6).astype(
        np.float32) * np.ones((ny, nx), np.float32), c_ref=1.0, tau=tau, mrt=coll == "mrt",
        s=W.mrt_rates(5, W.DEFAULT_SEED + 2) if coll == "mrt" else None,
        periodic=boundary == "periodic", sponge_width=sponge, sponge_sigma_max=0.1,
        source=(int(src[0]), int(src[1]), wav), receivers=rec)
    oc, os_, og = oracle_mod.adjoint(P, oracle_mod.init_pressure(P, p0.astype(np.float64)), nt,
                                     dj.astype(np.float64))
    assert _rel(gc.cpu().numpy(), oc) < 1e-4
    assert _rel(gs.cpu().numpy(), os_) < 1e-4
    assert _rel(g0.cpu().numpy(), np.asarray(og).reshape(g0.shape)) < 1e-4
    sim.close()
