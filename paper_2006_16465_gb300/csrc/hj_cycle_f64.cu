// Binary64 2D cycle kernels (exact evaluation order, no fused multiply-add); the
// other binary64 kernels and the registry are in hj_cycle1d_f64.cu, so that the
// two compile in parallel.
#include "hj_cycle.cuh"

namespace hj {

static const TileKernelInfo k_tiles2d[] = {
    HJ_K2D(double, double, 1, 8, 4, 1, true),    // 32 x 32
    HJ_K2D(double, double, 1, 16, 2, 1, true),   // 32 x 32, two warps
    HJ_K2D(double, double, 1, 4, 8, 1, true),    // 32 x 32, eight warps
    HJ_K2D(double, double, 1, 16, 1, 1, true),   // 32 x 16
    HJ_K2D(double, double, 1, 8, 1, 1, true),    // 32 x 8
    HJ_K2D(double, double, 1, 16, 4, 1, true),   // 32 x 64
    HJ_K2D(double, double, 2, 8, 4, 1, true),    // 64 x 32
    HJ_K2D(double, double, 2, 8, 8, 1, true),    // 64 x 64
};
const TileKernelInfo *tile_kernels2d_f64(int *n) { *n = sizeof(k_tiles2d) / sizeof(k_tiles2d[0]); return k_tiles2d; }

}  // namespace hj
