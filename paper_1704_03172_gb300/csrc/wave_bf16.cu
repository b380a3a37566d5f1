// wave_bf16.cu -- BF16-storage D2Q5 instances of the warp wavefront (wave.cuh).
#include "wave_host.h"

namespace lbwave {
WavePick pick_d2q5_bf16(int ck, int K, bool rec, bool per) {
    return K == 4 ? pick_rec<5, 4, __nv_bfloat16, true>(ck, rec, per)
                  : pick_rec<5, 2, __nv_bfloat16, true>(ck, rec, per);
}
WaveBatchFn pick_batch_round(bool mrt, bool per) { return pick_batch<true>(mrt, per); }
}  // namespace lbwave
