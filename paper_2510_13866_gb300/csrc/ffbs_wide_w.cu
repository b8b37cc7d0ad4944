// ffbs_wide_w.cu -- instantiations of the wide-lattice FFBS kernel that draw from windows of f
// (FP32 Hirsch classes that stream f).
#include "ffbs_launch.cuh"
#include "ffbs_wide.cuh"

namespace hqmc {

// units that a CTA filters before it draws their worldlines
int ffbs_wide_batch(int L) {
    switch (L) {
#define HQMC_CASE(n) \
    case n: return WideGeo<float, n, true>::NB;
        HQMC_WIDE_SIZES(HQMC_CASE)
#undef HQMC_CASE
        default: return 1;
    }
}

cudaError_t ffbs_wide_occupancy_w(int L, int *blocks) {
    switch (L) {
#define HQMC_CASE(n) \
    case n: return wide_occ<float, n, false, false, true>(blocks);
        HQMC_WIDE_SIZES(HQMC_CASE)
#undef HQMC_CASE
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_ffbs_wide_w(int L, const DevState &st, const FfbsLaunch &fl, int grid, cudaStream_t s) {
    switch (L) {
#define HQMC_CASE(n) \
    case n: return wide_go<float, n, false, false, true>(st, fl, grid, s);
        HQMC_WIDE_SIZES(HQMC_CASE)
#undef HQMC_CASE
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace hqmc
