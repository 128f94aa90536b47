// Tile kernels of the fp32-compute path for d = 32 (simt_tiles.cuh).
#include "simt_tiles.cuh"

namespace slim {
namespace simt {
extern const TileKernels kTilesD32F32, kTilesD32Bf16;
const TileKernels kTilesD32F32 = tile_set<float, 32>();
const TileKernels kTilesD32Bf16 = tile_set<bf16, 32>();
}  // namespace simt
}  // namespace slim
