// Binary64 2D cycle kernels of a subdomain on a cluster of CTAs (hj_cycle.cuh), in
// a translation unit of their own so that the library's kernels compile in
// parallel.
#include "hj_cycle.cuh"

namespace hj {

static const TileKernelInfo k_clusters[] = {
    HJ_K2DCL(4, 4),   // four CTAs of four warps
    HJ_K2DCL(8, 2),   // two CTAs of eight warps
};
const TileKernelInfo *cluster_kernels_f64(int *n) { *n = sizeof(k_clusters) / sizeof(k_clusters[0]); return k_clusters; }

}  // namespace hj
