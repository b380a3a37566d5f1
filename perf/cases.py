"""What a user of this library has it do, as cases that can be timed and checked.

Each case is one pass through the public entry points of ``paper_1704_03172_gb300.sim``:
a forward run (initial pressure and a Ricker source in, receiver traces and the pressure
field out), a gradient through ``LBForward`` (traces, dJ/dc and dJ/dS), or a batch of shots
through ``LBServer``.  Sizes, media, sponges, receivers and step counts are those of the
library's own workloads (the 128^2 periodic pulse, the two-layer, refined-block and layered
models, the served stream) or ragged sizes of the same range; long runs are cut to a few
hundred steps, which every step of a run resembles.

Fields start from a smooth random pressure, so that the whole grid carries waves as it does
in the middle of a run.  ``exact`` restates the scheme in 64-bit PyTorch (Eq. BGK-LB, Eq.
MRT-LB basic, Eq. linear eqm dist, Eq. 0th lattice weight of arXiv:1704.03172) without this
library's code.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1704_03172_gb300 import workloads as W

# The most site updates of one pass (the 8192^2 listed case): drawn cases stay below.
MOST = 8192 * 8192 * 96


def listed():
    return [
        # the periodic Gaussian pulse of the paper's homogeneous tests: a grid far smaller than
        # the GPU, where one step's latency and launch are the time
        dict(name="pulse_128", kind="forward", lattice=5, collision="bgk", tau=1.0,
             storage="f32", boundary="periodic", medium="uniform", nx=128, ny=128, steps=500,
             sponge=0, nrec=16),
        # one seismic shot of a served size, run alone: the states stay in L2
        dict(name="shot_512_layered", kind="forward", lattice=5, collision="bgk", tau=0.5,
             storage="f32", boundary="zero", medium="layered", nx=512, ny=512, steps=600,
             sponge=40, nrec=128),
        # the library's headline workload: two layers, sponge, 512 receivers on a line
        dict(name="two_layer_4096", kind="forward", lattice=5, collision="bgk", tau=0.5,
             storage="f32", boundary="zero", medium="two_layer", nx=4096, ny=4096, steps=200,
             sponge=40, nrec=512),
        # the comparison lattice with general relaxation rates on the same model
        dict(name="two_layer_4096_d2q9_mrt", kind="forward", lattice=9, collision="mrt", tau=0.5,
             storage="f32", boundary="zero", medium="two_layer", nx=4096, ny=4096, steps=100,
             sponge=40, nrec=512),
        # the large layered model with populations stored in 16 bits
        dict(name="layered_8192_bf16", kind="forward", lattice=5, collision="bgk", tau=0.5,
             storage="bf16", boundary="zero", medium="layered", nx=8192, ny=8192, steps=96,
             sponge=40, nrec=512),
        # a smooth model on the device (an inversion's current estimate), odd sizes, MRT
        dict(name="smooth_1531x1187_mrt", kind="forward", lattice=5, collision="mrt", tau=0.5,
             storage="f32", boundary="periodic", medium="smooth", nx=1531, ny=1187, steps=300,
             sponge=0, nrec=64),
        # FP16 storage with its range scales on a ragged layered model
        dict(name="layered_3001x1777_f16", kind="forward", lattice=5, collision="bgk", tau=0.5,
             storage="f16", boundary="zero", medium="layered", nx=3001, ny=1777, steps=200,
             sponge=40, nrec=256),
        # the paper's grid refinement: a slow block under a patch twice as fine
        dict(name="refined_2048", kind="refined", lattice=5, collision="mrt", tau=0.5,
             storage="f32", boundary="zero", nx=2048, ny=2048, steps=200, sponge=40, nrec=256),
        # an inversion's iteration: traces and the gradient with respect to model and source
        dict(name="gradient_2048", kind="gradient", lattice=5, collision="bgk", tau=0.5,
             storage="f32", boundary="zero", medium="smooth", nx=2048, ny=2048, steps=250,
             sponge=40, nrec=256, checkpoint=0),
        # the same with 16-bit storage and checkpoints, for runs whose tape would not fit
        dict(name="gradient_1201x911_bf16_ckpt", kind="gradient", lattice=5, collision="bgk",
             tau=0.5, storage="bf16", boundary="zero", medium="smooth", nx=1201, ny=911, steps=300,
             sponge=40, nrec=128, checkpoint=100),
        # three dimensions
        dict(name="cube_256_d3q7", kind="forward", lattice=7, collision="bgk", tau=0.5,
             storage="f32", boundary="zero", medium="two_layer", nx=256, ny=256, nz=256, steps=60,
             sponge=16, nrec=128),
        # independent shots of mixed sizes and storage, a quarter with gradients, at once
        dict(name="served_24", kind="served", shots=24, side_lo=256, side_hi=1024, steps=400,
             nrec=128, sponge=40),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["forward", "gradient", "refined", "cube", "served"], [10, 3, 1.5, 2, 1.5])[0]
    if kind == "served":
        lo = _log_int(rng, 128, 512)
        return dict(kind="served", shots=rng.randint(4, 28), side_lo=lo,
                    side_hi=_log_int(rng, max(lo, 256), 1024), steps=_log_int(rng, 100, 450),
                    nrec=rng.choice([1, 16, 128, 200]), sponge=rng.choice([0, 20, 40]))
    if kind == "refined":
        n = _log_int(rng, 192, 2048)
        return dict(kind="refined", lattice=rng.choice([5, 5, 9]), collision=rng.choice(["bgk", "mrt"]),
                    tau=0.5, storage="f32", boundary="zero", nx=n, ny=n, steps=_log_int(rng, 20, 200),
                    sponge=rng.choice([8, 20, 40]), nrec=rng.choice([16, 100, 256]))
    if kind == "cube":
        nx, ny, nz = (_log_int(rng, 24, 320) for _ in range(3))
        c = dict(kind="forward", lattice=7, collision="bgk", tau=rng.choice([0.5, 0.5, 0.8]),
                 storage=rng.choice(["f32", "f32", "bf16", "f16"]),
                 boundary=rng.choice(["zero", "zero", "periodic"]),
                 medium=rng.choice(["uniform", "two_layer", "layered", "smooth"]), nx=nx, ny=ny,
                 nz=nz, sponge=rng.choice([0, 4, 16]), nrec=rng.choice([1, 32, 128]))
        c["steps"] = max(1, min(_log_int(rng, 4, 300), MOST // (8 * nx * ny * nz)))
        return c
    nx, ny = _log_int(rng, 96, 4096), _log_int(rng, 96, 4096)
    c = dict(kind=kind, lattice=rng.choice([5, 5, 5, 9]), collision=rng.choice(["bgk", "bgk", "mrt"]),
             tau=rng.choice([0.5, 0.5, 0.5, 0.7, 1.0]),
             storage=rng.choice(["f32", "f32", "f32", "bf16", "bf16", "f16"]),
             boundary=rng.choice(["zero", "zero", "periodic"]),
             medium=rng.choice(["two_layer", "layered", "smooth"]), nx=nx, ny=ny,
             sponge=rng.choice([0, 16, 40]), nrec=rng.choice([1, 64, 200, 512]))
    if kind == "gradient":
        c["checkpoint"] = rng.choice([0, 0, 60, 100]) if c["storage"] != "f16" else 0
        c["steps"] = max(8, min(_log_int(rng, 40, 300), MOST // (8 * nx * ny)))
        return c
    c["steps"] = max(1, min(_log_int(rng, 4, 600), MOST // (2 * nx * ny)))
    how = rng.random()  # the ways to run it: as it comes, in place, or several steps a launch
    if how < 0.2 and c["storage"] != "f16":
        c["streaming"] = "aa"
    elif how < 0.35 and c["lattice"] == 5 and c["storage"] != "f16":
        c["time_block"] = rng.choice([2, 4, 8])
    elif how < 0.4 and c["lattice"] == 9 and c["storage"] == "f32":
        c["time_block"] = rng.choice([2, 4])
    return c


# ---------------------------------------------------------------------------- inputs --
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _shape(case):
    return (case["ny"], case["nx"]) if case.get("nz", 1) <= 1 else (case["nz"], case["ny"], case["nx"])


def _smooth(shape, seed, cells):
    """A smooth random field in about [-1, 1] with features of `cells` cells."""
    coarse = [max(2, -(-n // cells) + 1) for n in shape]
    f = torch.rand([1, 1] + coarse, generator=_gen(seed), device="cuda") * 2 - 1
    mode = "bilinear" if len(shape) == 2 else "trilinear"
    return torch.nn.functional.interpolate(f, size=list(shape), mode=mode, align_corners=True)[0, 0]


def _medium(case, seed):
    """(sound-speed map, c_ref).  Smooth models live on the device; the others are the arrays
    that a program reads from a model file, in host memory."""
    shape, kind = _shape(case), case["medium"]
    if kind == "smooth":
        return 0.75 + 0.2 * _smooth(shape, seed, 48), 1.0
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        return np.full(shape, 1.0, np.float32), 1.0
    if kind == "two_layer":
        c = np.full(shape, 1.0, np.float32)
        c[shape[0] // 2:] = 2.0
        return c, 2.0
    layers = 20  # dipping interfaces, speeds as in the layered model
    depth = torch.arange(shape[0], device="cuda", dtype=torch.float32)
    x = torch.arange(shape[-1], device="cuda", dtype=torch.float32) - shape[-1] / 2
    layer = torch.zeros((shape[0], shape[-1]), dtype=torch.int64, device="cuda")
    for d, s in zip(np.sort(rng.uniform(0, shape[0], layers - 1)), rng.uniform(-0.1, 0.1, layers - 1)):
        layer += depth[:, None] > float(d) + float(s) * x[None, :]
    speeds = torch.tensor(rng.uniform(1500.0, 5500.0, layers), dtype=torch.float32, device="cuda")
    c = speeds[layer].cpu().numpy()
    if len(shape) == 3:
        c = np.ascontiguousarray(np.broadcast_to(c[:, None, :], shape))
    return c, 5500.0


def _source(case, seed):
    """(site, wavelet): the paper's wavelet, its amplitude varied by the seed."""
    amp = 0.02 * (1.0 + 0.5 * np.random.default_rng(seed + 1).random())
    wav = (amp * W.ricker(case["steps"], 0.02)).astype(np.float32)
    site = (case["nx"] // 2, case["ny"] // 4)
    return (site + (case["nz"] // 3,) if case.get("nz", 1) > 1 else site), wav


def _receivers(case):
    n, lo = case["nrec"], min(case["sponge"], case["nx"] // 4)
    rec = W.line_receivers(n, case["ny"] // 4, lo, case["nx"] - 2 * lo)
    if case.get("nz", 1) > 1:
        rec = np.concatenate([rec, np.full((n, 1), case["nz"] // 3)], axis=1)
    return rec


def _rates(lattice):
    return W.mrt_rates(lattice, W.DEFAULT_SEED + 2)


W_REF = (0.0, 0.01, 0.24)  # the D2Q9 weights of the two-layer workload


def _scheme(case):
    d = dict(lattice=case["lattice"], collision=case["collision"], tau=case["tau"],
             storage=case["storage"], boundary=case["boundary"], sponge_width=case["sponge"],
             sponge_sigma_max=0.1)
    if case["collision"] == "mrt":
        d["s"] = _rates(case["lattice"])
    if case["lattice"] == 9:
        d["w_ref"] = W_REF
    return d


def _shots(case, seed):
    """The served stream's requests: square layered shots, sides, storage and gradients mixed."""
    rng = np.random.default_rng(seed)
    out = []
    for k in range(case["shots"]):
        # the k-th side, evenly over the logarithm of the range, so that every seed's batch
        # costs the same
        f = k / max(1, case["shots"] - 1)
        n = int(round(case["side_lo"] * (case["side_hi"] / case["side_lo"]) ** f))
        c, c_ref = _medium(dict(medium="layered", nx=n, ny=n), seed * 1000 + k)
        grad, nt = k % 4 == 1, case["steps"]
        lo = min(case["sponge"], n // 4)
        y = lo + 8
        d = dict(n=n, c_map=c, c_ref=c_ref, nt=nt, storage="bf16" if k % 2 else "f32",
                 source=(n // 2, y, (1.0 + rng.random()) * W.ricker(nt, W.SERVED_FC)),
                 receivers=W.line_receivers(case["nrec"], y, lo, n - 2 * lo), grad=grad)
        if grad:
            d["observed"] = (1e-2 * _smooth((nt, case["nrec"]), seed * 1000 + k, 16)).cpu().numpy()
        out.append(d)
    return out


def _patch(case):
    """The refined-block workload at this case's size: slow block, patch, source, receivers."""
    return W.refined_block_workload(case["nx"], case["nrec"], case["steps"])


def prepare(case, seed):
    from paper_1704_03172_gb300.sim import LBServer, LBSim

    kind = case["kind"]
    if kind == "served":
        return dict(kind=kind, case=case, shots=_shots(case, seed), server=LBServer(max_active=64))
    if kind == "gradient":
        c, c_ref = _medium(case, seed)
        c = torch.as_tensor(c, device="cuda").contiguous().requires_grad_()
        site, wav = _source(case, seed)
        spec = dict(_scheme(case), c_ref=c_ref, nt=case["steps"], source_xy=site,
                    receivers=_receivers(case), checkpoint_every=case["checkpoint"])
        return dict(kind=kind, c=c, wav=torch.tensor(wav, device="cuda").requires_grad_(),
                    spec=spec, dj=_residual(case, seed))
    more = {}
    if kind == "refined":
        wl = _patch(case)
        c, c_ref, more["patch"] = wl["c_map"], wl["c_ref"], wl["patch"]
        if case["lattice"] == 5 and case["collision"] == "mrt":
            more["s"] = wl["s"]
        sx, sy, wav = wl["source"]
        site, rec = (sx, sy), wl["receivers"]
        wav = (1.0 + 0.5 * np.random.default_rng(seed).random()) * wav
    else:
        c, c_ref = _medium(case, seed)
        site, wav = _source(case, seed)
        rec = _receivers(case)
        if "streaming" in case:
            more["streaming"] = case["streaming"]
        if "time_block" in case:
            more["time_block"] = case["time_block"]
    sim = LBSim(c, c_ref=c_ref, **dict(_scheme(case), **more))
    sim.set_source(*site, wav)
    sim.set_receivers(rec, case["steps"])
    return dict(kind=kind, sim=sim, p0=_p0(case, seed), steps=case["steps"])


def _residual(case, seed):
    """dJ/dp at the receivers: what an inversion's misfit gives, band-limited as its data are."""
    return _smooth((case["steps"], case["nrec"]), seed + 7, 16)


def _p0(case, seed):
    return 1e-2 * _smooth(_shape(case), seed + 3, 24)


def run(state):
    kind = state["kind"]
    if kind == "served":
        srv, ids = state["server"], []
        case = state["case"]
        for s in state["shots"]:
            ids.append(srv.submit(s["c_map"], nt=s["nt"], source=s["source"],
                                  receivers=s["receivers"], observed=s.get("observed"),
                                  want_gradient=s["grad"], storage=s["storage"],
                                  c_ref=s["c_ref"], sponge_width=case["sponge"]))
        out = []
        for rid, s in zip(ids, state["shots"]):
            srv.wait(rid)
            r = srv.result(rid)
            # an inversion holds its parameters, and so these gradients, in 32 bits
            out.append([r["traces"]] + ([r["grad_c"], r["grad_src"].astype(np.float32)]
                                        if s["grad"] else []))
        return _by_output(out)
    if kind == "gradient":
        from paper_1704_03172_gb300.sim import LBForward

        traces = LBForward.apply(state["c"], state["wav"], state["spec"])
        gc, gs = torch.autograd.grad(traces, (state["c"], state["wav"]), state["dj"])
        return dict(traces=traces.detach(), grad_c=gc, grad_src=gs)
    sim = state["sim"]
    sim.init_pressure(state["p0"])
    sim.step(state["steps"])
    return dict(traces=sim.traces(state["steps"]), pressure=sim.pressure())


def _by_output(out):
    """The shots' results joined by kind: every trace, then every gradient."""
    grads = [o for o in out if len(o) > 1]
    d = dict(traces=np.concatenate([o[0].reshape(-1) for o in out]))
    if grads:
        d["grad_c"] = np.concatenate([o[1].reshape(-1) for o in grads])
        d["grad_src"] = np.concatenate([o[2].reshape(-1) for o in grads])
    return d


def work(case):
    """The initial pressure, the speeds and the wavelet in, traces and pressure (or
    gradients) out, each once; and the operations of the site updates between them (D2Q5:
    moments 6, equilibrium 13, relaxation 10)."""
    per = {5: 29.0, 7: 41.0, 9: 66.0}
    if case["kind"] == "served":
        sites = grad = 0
        for k in range(case["shots"]):
            f = k / max(1, case["shots"] - 1)
            n = int(round(case["side_lo"] * (case["side_hi"] / case["side_lo"]) ** f))
            sites += n * n
            grad += n * n if k % 4 == 1 else 0
        return dict(bytes=4.0 * (sites + grad + case["shots"] * case["steps"] * case["nrec"]),
                    flops=29.0 * case["steps"] * (sites + 2.0 * grad))
    sites = case["nx"] * case["ny"] * case.get("nz", 1)
    traces = 4.0 * case["steps"] * case["nrec"]
    flops = per[case["lattice"]] * sites * case["steps"]
    if case["kind"] == "gradient":
        return dict(bytes=4.0 * 2 * sites + 2 * traces, flops=3.0 * flops)
    if case["kind"] == "refined":  # the patch: a quarter as many nodes, twice as many steps
        flops *= 1.5
    return dict(bytes=4.0 * 3 * sites + traces, flops=flops)


# ------------------------------------------------------------------ the scheme in 64 bits --
_C = {
    5: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0)],
    7: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)],
    9: [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0),
        (-1, -1, 0), (1, -1, 0)],
}


def _moments(lattice):
    """The rows of M (App. A of the paper) from the velocities."""
    c = np.array(_C[lattice], float)
    x, y, one = c[:, 0], c[:, 1], np.ones(len(c))
    r2 = x * x + y * y
    if lattice == 5:
        return np.array([one, x, y, 5 * r2 - 4, x * x - y * y])
    # rho, j_x, j_y, e, p_xx, eps, q_x, q_y, p_xy
    return np.array([one, x, y, 3 * r2 - 4, x * x - y * y, 4 - 10.5 * r2 + 4.5 * r2 * r2,
                     (3 * r2 - 5) * x, (3 * r2 - 5) * y, x * y])


def _weights(lattice, e2):
    """(w_i as fields, c_s^2) from eta^2."""
    if lattice == 9:
        w1, w5 = W_REF[1] * e2, W_REF[2] * e2
        return [1 - 4 * (w1 + w5)] + [w1] * 4 + [w5] * 4, e2 * (2 * W_REF[1] + 4 * W_REF[2])
    q = lattice
    return [1 - e2] + [e2 / (q - 1)] * (q - 1), e2 * (2.0 / (q - 1))


def _ratio(lattice):
    """w_i / c_s^2 of the moving populations (independent of eta)."""
    if lattice == 9:
        c2 = 2 * W_REF[1] + 4 * W_REF[2]
        return [0.0] + [W_REF[1] / c2] * 4 + [W_REF[2] / c2] * 4
    return [0.0] + [0.5] * (lattice - 1)


def _damping(shape, width):
    d = None
    for axis, n in enumerate(shape):
        i = torch.arange(n, device="cuda")
        m = torch.minimum(i, n - 1 - i)
        m = m.reshape([-1 if k == axis else 1 for k in range(len(shape))])
        d = m.expand(shape) if d is None else torch.minimum(d, m)
    r = (width - d).clamp(min=0).double() / max(width, 1)
    return 1 - 0.1 * r * r


class _Scheme:
    """One step g(t) -> g(t + 1) in 64 bits, and the pressure of a state."""

    def __init__(self, case, shape, site):
        self.q, self.shape, self.site = case["lattice"], shape, tuple(reversed(site))
        self.periodic = case["boundary"] == "periodic"
        self.damp = _damping(shape, case["sponge"]) if case["sponge"] > 0 else None
        self.tau, self.mrt = case["tau"], case["collision"] == "mrt"
        if self.mrt:
            M = _moments(self.q)
            C = np.linalg.inv(M) @ np.diag(_rates(self.q)) @ M
            C[np.abs(C) < 1e-14] = 0.0
            self.C = C

    def step(self, g, e2, S):
        w, _ = _weights(self.q, e2)
        a, c = _ratio(self.q), _C[self.q]
        rho = sum(g)
        j = [sum(c[i][k] * g[i] for i in range(self.q) if c[i][k]) for k in range(len(self.shape))]
        d = []  # g - g^eq
        for i in range(self.q):
            eq = w[i] * rho
            for k in range(len(self.shape)):
                if c[i][k]:
                    eq = eq + a[i] * c[i][k] * j[k]
            d.append(g[i] - eq)
        out = []
        for i in range(self.q):
            if self.mrt:
                h = g[i] - sum(self.C[i, k] * d[k] for k in range(self.q) if self.C[i, k])
            else:
                h = g[i] - d[i] / self.tau
            if S is not None:
                one = torch.zeros_like(h)
                one[self.site] = 1.0
                h = h + one * w[i] * S
            if self.damp is not None:
                h = h * self.damp
            out.append(self.stream(h, c[i]))
        return out

    def stream(self, h, c):
        for k, axis in enumerate(range(len(self.shape) - 1, -1, -1)):
            if not c[k]:
                continue
            if self.periodic:
                h = torch.roll(h, c[k], axis)
            else:
                n = self.shape[axis]
                z = torch.zeros_like(h.narrow(axis, 0, 1))
                h = (torch.cat([z, h.narrow(axis, 0, n - 1)], axis) if c[k] > 0
                     else torch.cat([h.narrow(axis, 1, n - 1), z], axis))
        return h

    def equilibrium(self, e2, p0):
        w, cs2 = _weights(self.q, e2)
        return [wi / cs2 * p0 for wi in w]


def _eta2(c, c_ref):
    return (torch.as_tensor(c, device="cuda").double() / c_ref) ** 2


def _forward64(case, c, c_ref, site, wav, rec, p0, keep=None):
    """(traces, pressure, eta^2, scheme); keep: a list that receives the state before each step."""
    e2 = _eta2(c, c_ref)
    sch = _Scheme(case, tuple(e2.shape), site)
    g = (sch.equilibrium(e2, p0.double()) if p0 is not None
         else [torch.zeros_like(e2) for _ in range(sch.q)])
    at = tuple(torch.as_tensor(rec[:, k].astype(np.int64), device="cuda")
               for k in range(rec.shape[1] - 1, -1, -1))
    _, cs2 = _weights(sch.q, e2)
    rows = []
    for n in range(len(wav)):
        if keep is not None:
            keep.append(g)
        rows.append(sum(gi[at] for gi in g) * cs2[at])
        g = sch.step(g, e2, float(wav[n]))
    return torch.stack(rows), sum(g) * cs2, e2, sch, at


def _gradient64(case, c, c_ref, site, wav, rec, dj=None, observed=None):
    """(traces, dJ/dc, dJ/dS): the chain rule through every step, last step first."""
    keep = []
    traces, _, e2, sch, at = _forward64(case, c, c_ref, site, wav, rec, None, keep)
    dj = traces - observed if dj is None else dj
    e2 = e2.requires_grad_()
    lam = [torch.zeros_like(e2) for _ in range(sch.q)]
    ge, gs = torch.zeros_like(e2), torch.zeros(len(wav), dtype=torch.float64, device="cuda")
    for n in range(len(wav) - 1, -1, -1):
        g = [x.detach().requires_grad_() for x in keep.pop()]
        S = torch.tensor(float(wav[n]), dtype=torch.float64, device="cuda", requires_grad=True)
        _, cs2 = _weights(sch.q, e2)
        p = sum(gi[at] for gi in g) * cs2[at]
        out = sch.step(g, e2, S)
        r = torch.autograd.grad(out + [p], g + [e2, S], lam + [dj[n].double()])
        lam, ge, gs[n] = list(r[:sch.q]), ge + r[sch.q], r[sch.q + 1]
    cc = torch.as_tensor(c, device="cuda").double()
    return traces, ge * 2 * cc / (c_ref * c_ref), gs


def exact(case, seed):
    kind = case["kind"]
    if kind == "refined":
        return None
    if kind == "served":
        out = []
        for s in _shots(case, seed):
            sub = dict(lattice=5, collision="bgk", tau=0.5, boundary="zero", sponge=case["sponge"])
            x, y, wav = s["source"]
            args = (sub, s["c_map"], s["c_ref"], (x, y), wav, s["receivers"])
            if s["grad"]:
                r = _gradient64(*args, observed=torch.tensor(s["observed"], device="cuda").double())
                out.append([v.detach().cpu().numpy() for v in r])
            else:
                out.append([_forward64(*args, None)[0].cpu().numpy()])
        return _by_output(out)
    c, c_ref = _medium(case, seed)
    site, wav = _source(case, seed)
    rec = _receivers(case)
    if kind == "gradient":
        if case["nx"] * case["ny"] * case["steps"] * case["lattice"] * 8 > 120e9:
            return None
        t, gc, gs = _gradient64(case, c, c_ref, site, wav, rec, dj=_residual(case, seed))
        return dict(traces=t, grad_c=gc.detach(), grad_src=gs)
    with torch.no_grad():
        traces, p, *_ = _forward64(case, c, c_ref, site, wav, rec, _p0(case, seed))
    return dict(traces=traces, pressure=p)
