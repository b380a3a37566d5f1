// tile_bf16.cu -- BF16-storage instances of the register tiles (tile.cuh).
#include "tile.cuh"

namespace lbtile {
TileFn pick_tile_bf16(int ck, bool rec, int ctas, bool per) { return pick_tile<__nv_bfloat16>(ck, rec, ctas, per); }
}  // namespace lbtile
