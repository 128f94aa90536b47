// Tile kernels of the fp32-compute path for d = 64 (simt_tiles.cuh).
#include "simt_tiles.cuh"

namespace slim {
namespace simt {
extern const TileKernels kTilesD64F32, kTilesD64Bf16;
const TileKernels kTilesD64F32 = tile_set<float, 64>();
const TileKernels kTilesD64Bf16 = tile_set<bf16, 64>();
}  // namespace simt
}  // namespace slim
