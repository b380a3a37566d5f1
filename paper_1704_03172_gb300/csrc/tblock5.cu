// tblock5.cu -- host side of the D2Q5 BF16 blocks with FP32 between their steps
// (cfg.time_block > 1; kernels: tblock5.cuh).
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "lb_kernels.cuh"
#include "lb_runtime.h"
#include "tblock5.cuh"

using namespace lbk;
using namespace lbrt;
using namespace lbtb5;

namespace {
Tb5Fn pick(int K, bool mrt) {
    switch (K) {
        case 2: return pick_k<2, __nv_bfloat16>(mrt);
        case 4: return pick_k<4, __nv_bfloat16>(mrt);
        case 6: return pick_k<6, __nv_bfloat16>(mrt);
        case 8: return pick_k<8, __nv_bfloat16>(mrt);
        case 16: return pick_k<16, __nv_bfloat16>(mrt);
        default: return nullptr;
    }
}
}  // namespace

// K fused D2Q5 steps with the caller's arguments (a.in must not be raw); receivers when
// a.trace_row is set and the row lists exist.
lb_status tb5_launch_args(lb_ctx *ctx, const StepArgs &a, int K) {
    const bool mrt = ctx->cfg.collision == LB_MRT, per = ctx->cfg.boundary == LB_PERIODIC;
    Tb5Fn fn = pick(K, mrt);
    if (!fn) return fail(ctx, LB_EINVAL, "time_block %d not supported for this storage", K);
    static int occ[17] = {0};  // resident CTAs per SM by K (the same for every variant)
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    if (!occ[K]) {
        int nb = 0;
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)((size_t)4 * K * (kWS + 2) * sizeof(float)));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kWS,
                                                      (size_t)4 * K * (kWS + 2) * sizeof(float));
        occ[K] = std::max(1, nb);
    }
    const int OUT = kWS - 2 * K;
    const int strips = (ctx->nx + OUT - 1) / OUT;
    // rows per CTA: the chunks of one wave of CTAs over the SMs.  A CTA sweeps its H + 2K
    // rows one after another, so a wave of short chunks beats fewer tall ones even though
    // each chunk recomputes 2K warm-up rows (GB300, two-layer 1024^2, K = 8: chunks of at
    // least 8K rows gave 80 CTAs and 60 GLUPS)
    const int slots = std::max(1, occ[K] * std::max(sms, 1));
    const int chunks = std::max(1, slots / strips);
    const int H = std::max(1, (ctx->ny + chunks - 1) / chunks);
    Tb5Args tb;
    tb.row_off = a.trace_row ? ctx->row_off : nullptr;
    tb.rec_x = ctx->row_x;
    tb.rec_id = ctx->row_id;
    tb.H = H;
    tb.per = per ? 1 : 0;
    dim3 grid(strips, (ctx->ny + H - 1) / H);
    const size_t smem = (size_t)2 * K * 2 * (kWS + 2) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "temporal-blocking shared memory");
    e = launch_pdl(fn, grid, dim3(kWS), smem, ctx->stream, a, tb);
    if (e != cudaSuccess) return cuda_fail(ctx, e, "temporal-blocking launch");
    return LB_OK;
}
