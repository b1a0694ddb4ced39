// Binary64: TMA-pipelined cycle kernels (hj_tma.cuh), two copy stages, in a
// translation unit of their own so that the library's kernels compile in
// parallel.
#include "hj_tma.cuh"

namespace hj {

static const PpcKernelInfo k_ppc[] = {
    HJ_KPPC(double, double, 1, 8, 4, 1, true, 2),   // 32 x 32
    HJ_KPPC(double, double, 1, 16, 2, 1, true, 2),   // 32 x 32, two warps
    HJ_KPPC(double, double, 1, 16, 1, 1, true, 2),   // 32 x 16
    HJ_KPPC(double, double, 1, 8, 1, 1, true, 2),   // 32 x 8
    HJ_KPPC(double, double, 1, 16, 4, 1, true, 2),   // 32 x 64
    HJ_KPPC(double, double, 2, 8, 4, 1, true, 2),   // 64 x 32
    HJ_KPPC(double, double, 2, 8, 8, 1, true, 2),   // 64 x 64
};
const PpcKernelInfo *ppc_kernels_f64(int *n) { *n = sizeof(k_ppc) / sizeof(k_ppc[0]); return k_ppc; }

}  // namespace hj
