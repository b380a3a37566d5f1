// tile.cu -- FP32 instances of the register tiles (tile.cuh).
#include "tile.cuh"

namespace lbtile {
TileFn pick_tile_f32(int ck, bool rec, int ctas, bool per) { return pick_tile<float>(ck, rec, ctas, per); }
}  // namespace lbtile
