// Large-N (four-step) row and column kernels, FP64.
#include "cme_large_launch.cuh"

namespace cme {

#define CME_LARGE_SHAPES(X) \
    X(6, 8) X(7, 8) X(8, 8) X(9, 8) X(10, 8) X(8, 4) X(9, 4) X(10, 4)

cudaError_t launch_large_row_fp64(int logN2, int R, const LargeArgs& a, long long rows,
                                  cudaStream_t s, bool pdl)
{
    switch (logN2 * 32 + R) {
#define CME_CASE(LN, RR)                                                                    \
    case LN * 32 + RR:                                                                      \
        return large_row_launch<double, LN, RR>(a, rows, s, pdl);
        CME_LARGE_SHAPES(CME_CASE)
#undef CME_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

cudaError_t launch_large_col_fp64(int logN1, int R, const LargeArgs& a, long long cols,
                                  cudaStream_t s, bool pdl)
{
    switch (logN1 * 32 + R) {
#define CME_CASE(LN, RR)                                                                    \
    case LN * 32 + RR:                                                                      \
        return large_col_launch<double, LN, RR>(a, cols, s, pdl);
        CME_LARGE_SHAPES(CME_CASE)
#undef CME_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace cme
