// sweep3.cu -- host side of the fused D3Q7 steps (kernel: sweep3.cuh).
#include <cuda_runtime.h>

#include <algorithm>

#include "lb_kernels.cuh"
#include "lb_runtime.h"
#include "sweep3.cuh"

using namespace lbk;
using namespace lbrt;
using namespace lbsweep3;

bool sweep3_supported(const lb_ctx *c) {
    return c->Q == 7 && !c->refined && !c->aa && !c->slab_nyg &&
           (c->cfg.storage == LB_F32 || c->cfg.storage == LB_BF16);
}

namespace {

// Tiles and chunks of a launch, and about what it takes: `rounds` planes one after another, of which a
// CTA computes `rows` rows each.
struct Plan {
    SweepArgs w;
    long long rounds;
    int rows;
    bool one_wave;
};

Plan plan_of(const lb_ctx *ctx) {
    Plan p;
    SweepArgs &w = p.w;
    w.per = ctx->cfg.boundary == LB_PERIODIC ? 1 : 0;
    w.rec_blocks = 0;
    // tiles evened out; their sides multiples of 8 columns (whole 32-byte sectors in FP32) where
    // one tile does not take the row
    const int most = kMaxX / 8 * 8;
    w.tx = ctx->nx <= kMaxX ? 1 : (ctx->nx + most - 1) / most;
    w.outx = round_up((ctx->nx + w.tx - 1) / w.tx, w.tx == 1 ? 2 : 8);
    w.ty = (ctx->ny3 + kMaxY - 1) / kMaxY;
    w.outy = (ctx->ny3 + w.ty - 1) / w.ty;
    // chunks of planes: a CTA takes its planes and two more, and about two planes' time to start;
    // two CTAs share an SM.  The receivers' blocks, which come first, are short: they count nothing here
    // (256^3 with 160000 receivers: 143 us a step, 468 when they were taken off the slots)
    const long long tiles = (long long)w.tx * w.ty, slots = 2 * sm_count();
    p.rounds = -1;
    w.chunks = 1;
    for (int n = 1; n <= ctx->nz; n++) {
        const long long waves = (tiles * n + slots - 1) / slots;
        const long long c = waves * ((ctx->nz + n - 1) / n + 4);
        if (p.rounds < 0 || c < p.rounds) p.rounds = c, w.chunks = n;
        if (waves > 4) break;
    }
    p.rows = std::min(w.outy + 2 * kHaloY, kRegY);
    p.one_wave = tiles * w.chunks <= slots;
    return p;
}

}  // namespace

// Where both states stay in L2 the one-step kernels are as fast or faster (us a step, one / two per
// launch: FP32 96^3 10.4 / 11.5, 128^3 20.2 / 21.5, 192^3 74.8 / 55.4, 320^3 309 / 212; staged BF16
// 1100 x 40 x 40 13.3 / 15.7, 320^3 290 / 162), so FP32 and staged grids have a line in sites.  Odd
// periodic grids, whose rows are not whole lanes at the seam, keep single steps.
//
// Otherwise the estimates below decide, in us: a step of the one-step kernel by the warps' segments of a
// row (128 sites, BF16 256) that it reads, filled or not, and a launch of two by its rounds of planes,
// their rows and the receivers, whose second pressure costs 49 loads.  They are fits to 110 grids of
// 0.2 to 17 million sites, good to 15 %; what they decide, us a step, one / two per launch: BF16 96^3
// 12.7 / 12.2, periodic 12.6 / 14.8; 112 x 294 x 301 131 / 57; 238 x 68 x 129 15.2 / 20.2;
// 208 x 227 x 82 29.5 / 28.2, periodic 28.0 / 34.9; 256^3 107 / 109, with 60000 receivers 108 / 117; FP32
// periodic 184 x 254 x 62 31.5 / 33.5; 96 x 269 x 126 34.4 / 34.3.  Several waves of CTAs overlap, and
// the estimate of a launch does not hold for them: they stay with the line in sites.
bool sweep3_pays(const lb_ctx *c) {
    const bool per = c->cfg.boundary == LB_PERIODIC, bf = c->cfg.storage == LB_BF16;
    if (per && c->nx % 2 != 0) return false;
    if ((long long)c->ny * c->pitch < (bf && !c->staged ? 800000 : 3000000)) return false;
    if (c->staged) return true;
    const Plan p = plan_of(c);
    if (!p.one_wave) return true;
    const int seg = bf ? 256 : 128;
    const double sites = 1e-6 * c->nx * c->ny, read = 1e-6 * round_up(c->nx, seg) * c->ny;
    double one, round;  // a step; a round of planes
    if (bf) {
        one = 0.97 * (2.5 + (per ? 3.6 : 4.0) * read + 2.4 * sites);
        round = per ? 1.2 + 0.125 * p.rows : 0.9 + 0.113 * p.rows;
    } else {
        one = std::max(8.0 * read, 9.8 * sites);
        round = per ? 0.7 + 0.155 * p.rows : 0.4 + 0.135 * p.rows;
    }
    return p.rounds * round + 0.45e-3 * c->nrec < 2 * one;
}

// Two steps with the caller's arguments (a.in must not be raw); the receivers' two rows when
// a.trace_row is set.
lb_status sweep3_launch(lb_ctx *ctx, const StepArgs &a) {
    SweepArgs w = plan_of(ctx).w;
    w.rec_blocks = a.trace_row ? (ctx->nrec + kThreadsZ - 1) / kThreadsZ : 0;
    const bool bf = ctx->cfg.storage == LB_BF16;
    const int smem = bf ? (int)sizeof(SharedZ<__nv_bfloat16>) : (int)sizeof(SharedZ<float>);
    void (*fn)(const StepArgs, const SweepArgs) =
        bf ? sweep3_kernel<__nv_bfloat16> : sweep3_kernel<float>;
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess)
        e = launch_pdl(fn, dim3(w.rec_blocks + w.tx * w.ty * w.chunks), dim3(kThreadsZ), smem, ctx->stream,
                       a, w);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "3-D sweep launch");
    return LB_OK;
}
