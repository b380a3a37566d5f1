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

template <int Q, int CK, int K, bool REC, typename ST, bool ROUND> WavePick pick_one() {
    return {wave_kernel<Q, CK, K, REC, ST, ROUND>, cta_bytes<Q, K, ST>(), min_ctas<Q, K, ST>()};
}
template <int Q, int K, bool REC, typename ST, bool ROUND> WavePick pick_ck(int ck) {
    if (ck == kMrt) return pick_one<Q, kMrt, K, REC, ST, ROUND>();
    if constexpr (Q == 5) {
        if (ck == kLossless) return pick_one<Q, kLossless, K, REC, ST, ROUND>();
    }
    return pick_one<Q, kBgk, K, REC, ST, ROUND>();
}
template <int Q, int K, typename ST, bool ROUND> WavePick pick_rec(int ck, bool rec) {
    return rec ? pick_ck<Q, K, true, ST, ROUND>(ck) : pick_ck<Q, K, false, ST, ROUND>(ck);
}

WavePick pick_d2q5_f32(int ck, int K, bool rec);   // wave.cu
WavePick pick_d2q5_bf16(int ck, int K, bool rec);  // wave_bf16.cu: rounded at every level
WavePick pick_d2q5_f16(int ck, bool rec);          // wave_f16.cu: two steps
WavePick pick_d2q9_f32(int ck, int K, bool rec);   // wave9.cu
WavePick pick_d2q9_bf16(int ck, int K, bool rec);  // wave9_bf16.cu

template <bool ROUND> WaveBatchFn pick_batch(bool mrt) {
    return mrt ? wave_batch_kernel<true, kServeSteps, ROUND>
               : wave_batch_kernel<false, kServeSteps, ROUND>;
}
WaveBatchFn pick_batch_fp32(bool mrt);   // wave.cu: BF16 shots keep FP32 between a launch's steps
WaveBatchFn pick_batch_round(bool mrt);  // wave_bf16.cu: they round at every step

}  // namespace lbwave
