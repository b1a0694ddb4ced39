// Binary32 cycle kernels (fused multiply-add chains).
#include "hj_cycle.cuh"

namespace hj {

static const TileKernelInfo k_tiles[] = {
    HJ_K2D(float, float, 2, 16, 1, 2, false),    // 32 x 32
    HJ_K2D(float, float, 2, 8, 2, 2, false),     // 32 x 32, two warps
    HJ_K2D(float, float, 2, 4, 4, 2, false),     // 32 x 32, four warps
    HJ_K2D(float, float, 2, 2, 8, 2, false),     // 32 x 32, eight warps
    HJ_K2D(float, float, 2, 8, 1, 2, false),     // 32 x 16
    HJ_K2D(float, float, 2, 4, 1, 2, false),     // 32 x 8
    HJ_K2D(float, float, 2, 16, 2, 2, false),    // 32 x 64
    HJ_K2D(float, float, 2, 16, 2, 1, false),    // 64 x 32
    HJ_K2D(float, float, 2, 16, 4, 1, false),    // 64 x 64
    HJ_K2D(float, float, 4, 8, 4, 1, false),     // 128 x 32
    HJ_K2D(float, float, 4, 8, 8, 1, false),     // 128 x 64
    HJ_K1D(float, float, 1, 1, 4, false),    // 32
    HJ_K1D(float, float, 2, 1, 4, false),    // 64
    HJ_K1D(float, float, 1, 2, 1, false),    // 64, 2 warps
    HJ_K1D(float, float, 4, 1, 4, false),    // 128
    HJ_K1D(float, float, 2, 2, 1, false),    // 128, 2 warps
    HJ_K1D(float, float, 1, 4, 1, false),    // 128, 4 warps
    HJ_K1D(float, float, 8, 1, 4, false),    // 256
    HJ_K1D(float, float, 4, 2, 1, false),    // 256, 2 warps
    HJ_K1D(float, float, 2, 4, 1, false),    // 256, 4 warps
    HJ_K1D(float, float, 1, 8, 1, false),    // 256, 8 warps
};
static const TileKernelInfo k_classic[] = {HJ_KC2D(float, float, false), HJ_KC1D(float, float, false)};

const TileKernelInfo *tile_kernels_f32(int *n) { *n = sizeof(k_tiles) / sizeof(k_tiles[0]); return k_tiles; }
const TileKernelInfo *classic_kernels_f32(int *n) { *n = 2; return k_classic; }

static const VcKernelInfo k_vc = HJ_KVC(float, float, false, hj::vc2d_rows_kernel<false>, hj::vc2d_rows_kernel<true>);
const VcKernelInfo *vc_kernels_f32() { return &k_vc; }

}  // namespace hj
