"""What a served BF16 shot rounds does not depend on the shots beside it that record a rho tape: it counts
only shots without one when it decides whether to keep FP32 between the steps of a launch."""
import numpy as np
import pytest

from paper_1704_03172_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# tb_min_ctas: 0 and a count that only the taped shot reaches (the small one makes 5 CTAs)
@pytest.mark.parametrize("tb", [0, 100])
def test_taped_company_leaves_a_bf16_shot_as_it_is(tb):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1704_03172_gb300 import build
    build.build()
    from paper_1704_03172_gb300.sim import LBServer, LBSim

    def shot(n, nt, **kw):
        c = W.layered_fault_model(n, n, n, n_layers=6, throw=(2.0, n / 16))
        return c, dict(nt=nt, source=(n // 2, 6, W.ricker(nt, 0.05)),
                       receivers=W.line_receivers(16, 6, 4, n - 8), tau=0.5, sponge_width=6,
                       c_ref=5500.0, **kw)

    c, s = shot(256, 400, storage="bf16")
    # 168 MB of states, more than L2 holds, and a tape
    cb, sb = shot(2048, 1500, storage="f32", want_gradient=True,
                  observed=np.zeros((1500, 16), np.float32), checkpoint_every=-1)
    srv = LBServer(max_active=2, rounds_per_pass=8, tb_min_ctas=tb)
    ids = [srv.submit(cb, **sb), srv.submit(c, **s)]
    for i in ids:
        srv.wait(i, 120000)
    big, got = (srv.result(i) for i in ids)
    srv.close()
    assert big["start"] < got["start"] and got["done"] < big["done"]  # in company throughout
    sim = LBSim(c, lattice=5, tau=0.5, storage="bf16", sponge_width=6, c_ref=5500.0,
                step_kernel="direct")
    sim.set_source(*s["source"])
    sim.set_receivers(s["receivers"], s["nt"])
    sim.init_pressure(None)
    sim.step(s["nt"])
    want = sim.traces(s["nt"]).cpu().numpy()
    sim.close()
    np.testing.assert_array_equal(got["traces"], want)
