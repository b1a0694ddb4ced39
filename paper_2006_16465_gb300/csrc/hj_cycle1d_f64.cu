// Binary64 1D cycle, classic and variable-coefficient kernels (exact evaluation
// order, no fused multiply-add), and the registry of all binary64 cycle kernels.
#include <algorithm>
#include <vector>

#include "hj_cycle.cuh"

namespace hj {

static const TileKernelInfo k_tiles1d[] = {
    HJ_K1D(double, double, 1, 1, 4, true),    // 32
    HJ_K1D(double, double, 2, 1, 4, true),    // 64
    HJ_K1D(double, double, 1, 2, 1, true),    // 64, 2 warps
    HJ_K1D(double, double, 4, 1, 4, true),    // 128
    HJ_K1D(double, double, 2, 2, 1, true),    // 128, 2 warps
    HJ_K1D(double, double, 1, 4, 1, true),    // 128, 4 warps
    HJ_K1D(double, double, 8, 1, 4, true),    // 256
    HJ_K1D(double, double, 4, 2, 1, true),    // 256, 2 warps
    HJ_K1D(double, double, 2, 4, 1, true),    // 256, 4 warps
    HJ_K1D(double, double, 1, 8, 1, true),    // 256, 8 warps
};
static const TileKernelInfo k_classic[] = {HJ_KC2D(double, double, true), HJ_KC1D(double, double, true)};


const TileKernelInfo *tile_kernels2d_f64(int *n);   // hj_cycle_f64.cu

const TileKernelInfo *tile_kernels_f64(int *n) {
    static const std::vector<TileKernelInfo> all = [] {
        int n2 = 0;
        const TileKernelInfo *k2 = tile_kernels2d_f64(&n2);
        std::vector<TileKernelInfo> v(k2, k2 + n2);
        v.insert(v.end(), std::begin(k_tiles1d), std::end(k_tiles1d));
        return v;
    }();
    *n = (int)all.size();
    return all.data();
}
const TileKernelInfo *classic_kernels_f64(int *n) { *n = 2; return k_classic; }

static const VcKernelInfo k_vc = HJ_KVC(double, double, true, nullptr, nullptr);
const VcKernelInfo *vc_kernels_f64() { return &k_vc; }

}  // namespace hj
