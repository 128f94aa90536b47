// Tile kernels of the fp32-compute path for d = 128 (simt_tiles.cuh).
#include "simt_tiles.cuh"

namespace slim {
namespace simt {
extern const TileKernels kTilesD128F32, kTilesD128Bf16;
const TileKernels kTilesD128F32 = tile_set<float, 128>();
const TileKernels kTilesD128Bf16 = tile_set<bf16, 128>();
}  // namespace simt
}  // namespace slim
