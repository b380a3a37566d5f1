"""lb_footprint bounds what a context holds: every buffer it asks its allocator for and keeps."""
import numpy as np
import pytest

from paper_1704_03172_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,storage,nx,ny,nrec", [
    (5, "f32", 300, 200, 100000), (9, "bf16", 128, 77, 50000), (5, "f16", 64, 40, 3),
    (5, "f16", 1100, 300, 1)])
def test_footprint_bounds_the_allocations(monkeypatch, lattice, storage, nx, ny, nrec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03172_gb300 import build
    build.build()
    from paper_1704_03172_gb300 import lbac
    from paper_1704_03172_gb300.sim import LBSim
    held, real, free = {}, torch.cuda.caching_allocator_alloc, torch.cuda.caching_allocator_delete

    def alloc(size, **kw):
        p = real(size, **kw)
        held[p] = size
        return p

    def delete(p):
        held.pop(p)
        free(p)
    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", delete)
    cfg = lbac.lb_config_default()
    cfg.lattice, cfg.nx, cfg.ny = lattice, nx, ny
    cfg.storage = {"f32": lbac.LB_F32, "bf16": lbac.LB_BF16, "f16": lbac.LB_F16}[storage]
    nt = 5
    est = lbac.lb_footprint(cfg, nt, nrec, 0)
    sim = LBSim(W.two_layer(nx, ny, 1.0, 2.0), lattice=lattice, storage=storage, tau=0.6)  # (indexed)
    rng = np.random.default_rng(nrec)
    sim.set_source(nx // 2, ny // 2, np.ones(nt))
    sim.set_receivers(np.stack([rng.integers(0, nx, nrec), rng.integers(0, ny, nrec)], 1), nt)
    used = sum(held.values())
    sim.close()
    assert 0 < used <= est <= 1.05 * used + 4096, (used, est)
