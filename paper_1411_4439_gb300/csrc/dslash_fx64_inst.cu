// Instances of the fixed-point FP64 Dslash (dslash_fx64.cuh) for one spinor
// layout: -DHISQ_LAYOUT=<0 (AoS)|1 (SoA)> -DHISQ_FAMILY=<function name>.
#include <cmath>

#include "dslash_fx64.cuh"

namespace hisq {

template <int EPI>
static cudaError_t fx64_by_rpt(const DslashArgs& a, int rpt, int split, cudaStream_t s) {
    const bool small = a.nrhs <= 4 * rpt;   // blocks of at most 128 threads
    switch (rpt * 10 + split) {
        case 11: return launch_fx64<1, 1, EPI, HISQ_LAYOUT, 256, 2>(a, s);
        case 21: return small ? launch_fx64<2, 1, EPI, HISQ_LAYOUT, 128, 3>(a, s)
                              : launch_fx64<2, 1, EPI, HISQ_LAYOUT, 256, 1>(a, s);
        case 41: return launch_fx64<4, 1, EPI, HISQ_LAYOUT, 256, 1>(a, s);
        case 14: return launch_fx64<1, 4, EPI, HISQ_LAYOUT, 256, 2>(a, s);
        case 24: return launch_fx64<2, 4, EPI, HISQ_LAYOUT, 256, 1>(a, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t HISQ_FAMILY(const DslashArgs& a, int epi, int rpt, int split, cudaStream_t s) {
    switch (epi) {
        case EPI_NONE: return fx64_by_rpt<EPI_NONE>(a, rpt, split, s);
        case EPI_X: return fx64_by_rpt<EPI_X>(a, rpt, split, s);
        case EPI_XY: return fx64_by_rpt<EPI_XY>(a, rpt, split, s);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace hisq
