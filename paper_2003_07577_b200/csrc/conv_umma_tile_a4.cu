// Tile kernels (tcgen05, split reduction) for 4-bit activations.
#include "conv_umma_tile.cuh"

namespace ebs {
static_assert(NUM_TILE_VARIANTS == NUM_CONV_UMMA_VARIANTS, "tables out of sync");
EBS_DEFINE_TILE_ROW(4)
}  // namespace ebs
