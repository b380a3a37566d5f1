// wave_f16.cu -- FP16-storage D2Q5 instances of the warp wavefront (wave.cuh), two steps.
#include "wave_host.h"

namespace lbwave {
WavePick pick_d2q5_f16(int ck, bool rec, bool per) { return pick_rec<5, 2, __half, true>(ck, rec, per); }
}  // namespace lbwave
