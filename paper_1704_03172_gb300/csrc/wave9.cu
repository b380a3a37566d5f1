// wave9.cu -- FP32 D2Q9 instances of the warp wavefront (wave.cuh).
#include "wave_host.h"

namespace lbwave {
WavePick pick_d2q9_f32(int ck, int K, bool rec, bool per) {
    return K == 4 ? pick_rec<9, 4, float, false>(ck, rec, per) : pick_rec<9, 2, float, false>(ck, rec, per);
}
}  // namespace lbwave
