// 16-bit instances of the tile kernel (d2q9_tile.cuh).
#include "d2q9_tile.cuh"

namespace lbmrv {

cudaError_t launch_tile16(int storage, int um, int basis, int nv, const void* src, void* dst,
                          const StepArgs& a, const TileAmps& amps, const TilePlan& p,
                          cudaStream_t st) {
    if (storage == kStoreF16)
        return tile_basis<__half>(um, basis, nv, src, dst, a, amps, p, st);
    return tile_basis<__nv_bfloat16>(um, basis, nv, src, dst, a, amps, p, st);
}

}  // namespace lbmrv
