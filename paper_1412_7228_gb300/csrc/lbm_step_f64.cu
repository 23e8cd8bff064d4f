// lbm_step_f64.cu -- the FP64 instantiations of the fused step kernels (one-step and
// multi-step) for every tile configuration the autotuner may pick; compiled
// as a translation unit of its own so that the two precisions build in parallel.
#include "lbm_step_kernels.cuh"

namespace lbm {
namespace {
// 16 x 8 tiles of 128 threads for small lattices: one node per lane and one
// warp per SM quarter, since the FP64 pipe takes 64 clocks per warp
// instruction of a quarter however few lanes it carries, and the tiles spread
// over more SMs (64^2: 8.9 us per step, 15.2 with 32 x 8 tiles, 13.5 in a
// cluster of 16 CTAs; six 128 x 4 slabs 9.0 and 11.7).
const Entry kF64[] = {
    LBM_CFG(double, 32, 8, 256, 1),  LBM_CFG(double, 64, 8, 256, 1), LBM_CFG(double, 32, 16, 256, 1),
    LBM_CFG(double, 64, 4, 256, 1),  LBM_CFG(double, 32, 8, 256, 2),  LBM_CFG(double, 64, 16, 256, 1),
    LBM_CFG(double, 32, 32, 256, 1), LBM_CFG(double, 16, 8, 128, 1),
};
}  // namespace

const Entry* step_table_f64(int* n) {
    *n = int(sizeof(kF64) / sizeof(kF64[0]));
    return kF64;
}

}  // namespace lbm
