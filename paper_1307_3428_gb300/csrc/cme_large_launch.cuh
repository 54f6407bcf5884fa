// Launches of the large-N row and column kernels for one transform length and radix.
#pragma once

#include "cme_launch.cuh"
#include "cme_large.cuh"

namespace cme {
inline namespace CME_FP32_VARIANT {

template <typename T, int LN, int R>
cudaError_t large_row_launch(const LargeArgs& a, long long rows, cudaStream_t s, bool pdl)
{
    return launch_pdl(large_row_kernel<T, LN, R>, (unsigned)((rows + a.G - 1) / a.G),
                      Plan<LN, R>::P * a.G, smem_bytes_for<T>(LN, R, a.G), s, pdl, a);
}

template <typename T, int LN, int R, int ST>
cudaError_t large_col_stage(const LargeArgs& a, long long cols, cudaStream_t s, bool pdl)
{
    return launch_pdl(large_col_kernel<T, LN, R, ST>, (unsigned)((cols + a.G - 1) / a.G),
                      Plan<LN, R>::P * a.G, smem_bytes_for<T>(LN, R, a.G), s, pdl, a);
}

template <typename T, int LN, int R>
cudaError_t large_col_launch(const LargeArgs& a, long long cols, cudaStream_t s, bool pdl)
{
    switch (a.stage) {
    case LARGE_START:
        return large_col_stage<T, LN, R, LARGE_START>(a, cols, s, pdl);
    case 0:
        return large_col_stage<T, LN, R, 0>(a, cols, s, pdl);
    case 1:
        return large_col_stage<T, LN, R, 1>(a, cols, s, pdl);
    case 2:
        return large_col_stage<T, LN, R, 2>(a, cols, s, pdl);
    case 3:
        return large_col_stage<T, LN, R, 3>(a, cols, s, pdl);
    case LARGE_FINAL:
        return large_col_stage<T, LN, R, LARGE_FINAL>(a, cols, s, pdl);
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace CME_FP32_VARIANT
}  // namespace cme
