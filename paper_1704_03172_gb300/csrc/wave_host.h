// wave_host.h -- the wavefront's kernel instances by storage type (one file each, compiled in
// parallel) as the host side picks them.
#pragma once

#include "lb_runtime.h"
#include "wave.cuh"

namespace lbwave {

struct WavePick {
    WaveFn fn;
    int smem;  // dynamic shared memory per CTA
    int ctas;  // resident CTAs per SM the kernel is cut for
};

// An instance for each boundary: what only the other one needs costs registers, of which the levels
// are short (120 grids: 4 % faster on average).  Six steps are the exception, whose zero-ghost instance
// spills more than the one for either (two-layer 4096^2, 200 steps: 7110 us against 6700).
template <int Q, int CK, int K, bool REC, typename ST, bool ROUND> WavePick pick_one(bool per) {
    return {per ? wave_kernel<Q, CK, K, REC, ST, ROUND, kPeriodic>
                : wave_kernel<Q, CK, K, REC, ST, ROUND, K == 6 ? kEither : kZeroGhost>,
            cta_bytes<Q, K, ST>(), min_ctas<Q, K, ST>()};
}
template <int Q, int K, bool REC, typename ST, bool ROUND> WavePick pick_ck(int ck, bool per) {
    if (ck == kMrt) return pick_one<Q, kMrt, K, REC, ST, ROUND>(per);
    if constexpr (Q == 5) {
        if (ck == kLossless) return pick_one<Q, kLossless, K, REC, ST, ROUND>(per);
    }
    return pick_one<Q, kBgk, K, REC, ST, ROUND>(per);
}
template <int Q, int K, typename ST, bool ROUND> WavePick pick_rec(int ck, bool rec, bool per) {
    return rec ? pick_ck<Q, K, true, ST, ROUND>(ck, per) : pick_ck<Q, K, false, ST, ROUND>(ck, per);
}

WavePick pick_d2q5_f32(int ck, int K, bool rec, bool per);   // wave.cu
WavePick pick_d2q5_bf16(int ck, int K, bool rec, bool per);  // wave_bf16.cu: rounded at every level
WavePick pick_d2q5_f16(int ck, bool rec, bool per);          // wave_f16.cu: two steps
WavePick pick_d2q9_f32(int ck, int K, bool rec, bool per);   // wave9.cu
WavePick pick_d2q9_bf16(int ck, int K, bool rec, bool per);  // wave9_bf16.cu

template <bool ROUND> WaveBatchFn pick_batch(bool mrt, bool per) {
    if (per)
        return mrt ? wave_batch_kernel<true, kServeSteps, ROUND, kPeriodic>
                   : wave_batch_kernel<false, kServeSteps, ROUND, kPeriodic>;
    return mrt ? wave_batch_kernel<true, kServeSteps, ROUND, kZeroGhost>
               : wave_batch_kernel<false, kServeSteps, ROUND, kZeroGhost>;
}
WaveBatchFn pick_batch_fp32(bool mrt, bool per);   // wave.cu: BF16 keeps FP32 between a launch's steps
WaveBatchFn pick_batch_round(bool mrt, bool per);  // wave_bf16.cu: it is rounded at every step

}  // namespace lbwave
