// wave9_bf16.cu -- BF16-storage D2Q9 instances of the warp wavefront (wave.cuh).
#include "wave_host.h"

namespace lbwave {
WavePick pick_d2q9_bf16(int ck, int K, bool rec, bool per) {
    return K == 4 ? pick_rec<9, 4, __nv_bfloat16, true>(ck, rec, per)
                  : pick_rec<9, 2, __nv_bfloat16, true>(ck, rec, per);
}
}  // namespace lbwave
