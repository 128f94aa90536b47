// Tile kernels of the fp32-compute path for d = 16 (simt_tiles.cuh).
#include "simt_tiles.cuh"

namespace slim {
namespace simt {
extern const TileKernels kTilesD16F32, kTilesD16Bf16;
const TileKernels kTilesD16F32 = tile_set<float, 16>();
const TileKernels kTilesD16Bf16 = tile_set<bf16, 16>();
}  // namespace simt
}  // namespace slim
