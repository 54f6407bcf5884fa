// Large-N (four-step) row and column kernels, FP32: packed arithmetic, and the choice.
#include "cme_large_launch.cuh"

namespace cme {

#define CME_LARGE_ROWS(X) X(7, 8) X(8, 8) X(9, 8) X(8, 4) X(9, 4)
#define CME_LARGE_COLS(X) X(8, 8) X(9, 8) X(8, 4) X(9, 4)

// Packed arithmetic for 2^15 <= N <= 2^18, scalar (kern_large_fp32_scalar.cu) for the others: a rule on
// N alone, so that the grid-barrier kernel below, which is packed, repeats the sequence's bits.
// us per step, scalar / packed: 2^13 17.1 / 16.8, 8 instances 21.1 / 24.5, 9 21.4 / 28.8; 2^14 18.4 / 17.9,
// 4 instances 23.3 / 23.3, 12 39.4 / 39.7; 2^15 20.4 / 19.3, 2 instances 26.1 / 27.3, 3 25.3 / 24.7,
// 4 27.0 / 25.3, 6 44.6 / 47.0, 8 41 / 38.7; 2^16 29.9 / 30.5, 2 instances 28.9 / 27.8, 3 54.9 / 50.5;
// 2^17 29.9 / 29.2, 2 instances 62.5 / 61.2; 2^18 45.5 / 45.6, 3 instances 114.5 / 114.2; 2^19 96.2 /
// 101.8; 2^20 151.8 / 153.1 (columns of N1 = 1024: 178 registers, two blocks per SM where 164 leave
// three).
static bool packed(const LargeArgs& a)
{
    const int logN = a.logN1 + a.logN2;
    return logN >= 15 && logN <= 18;
}

cudaError_t launch_large_row_fp32(int logN2, int R, const LargeArgs& a, long long rows,
                                  cudaStream_t s, bool pdl)
{
    if (!packed(a))
        return launch_large_row_fp32_scalar(logN2, R, a, rows, s, pdl);
    switch (logN2 * 32 + R) {
#define CME_CASE(LN, RR)                                                                    \
    case LN * 32 + RR:                                                                      \
        return large_row_launch<float, LN, RR>(a, rows, s, pdl);
        CME_LARGE_ROWS(CME_CASE)
#undef CME_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

cudaError_t launch_large_col_fp32(int logN1, int R, const LargeArgs& a, long long cols,
                                  cudaStream_t s, bool pdl)
{
    if (!packed(a))
        return launch_large_col_fp32_scalar(logN1, R, a, cols, s, pdl);
    switch (logN1 * 32 + R) {
#define CME_CASE(LN, RR)                                                                    \
    case LN * 32 + RR:                                                                      \
        return large_col_launch<float, LN, RR>(a, cols, s, pdl);
        CME_LARGE_COLS(CME_CASE)
#undef CME_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

#define CME_GRID_SHAPES(X) X(8, 7) X(8, 8) X(9, 8) X(9, 9)

bool large_grid_fits(int logN1, int logN2, long long blocks, int sms)
{
    switch (logN1 * 32 + logN2) {
#define CME_CASE(L1, L2)                                                                    \
    case L1 * 32 + L2: {                                                                     \
        auto k = large_grid_kernel<float, L1, L2, 8>;                                        \
        constexpr size_t smem = large_grid_smem<float, L1, L2, 8>();                          \
        if (prepare_smem(k, smem) != cudaSuccess) {                                          \
            cudaGetLastError();                                                              \
            return false;                                                                    \
        }                                                                                    \
        int per = 0;                                                                         \
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, Plan<L1, 8>::P, smem) !=  \
            cudaSuccess) {                                                                   \
            cudaGetLastError();                                                              \
            return false;                                                                    \
        }                                                                                    \
        return (long long)per * sms >= blocks;                                               \
    }
        CME_GRID_SHAPES(CME_CASE)
#undef CME_CASE
    default:
        return false;
    }
}

cudaError_t launch_large_grid_fp32(int logN1, int logN2, const LargeArgs& a, long long blocks,
                                   cudaStream_t s)
{
    switch (logN1 * 32 + logN2) {
#define CME_CASE(L1, L2)                                                                    \
    case L1 * 32 + L2: {                                                                     \
        auto k = large_grid_kernel<float, L1, L2, 8>;                                        \
        constexpr size_t smem = large_grid_smem<float, L1, L2, 8>();                          \
        cudaError_t e = prepare_smem(k, smem);                                               \
        if (e != cudaSuccess)                                                                \
            return e;                                                                        \
        cudaLaunchConfig_t cfg = {};                                                         \
        cfg.gridDim = dim3((unsigned)blocks, 1, 1);                                          \
        cfg.blockDim = dim3(Plan<L1, 8>::P, 1, 1);                                           \
        cfg.dynamicSmemBytes = smem;                                                         \
        cfg.stream = s;                                                                      \
        cudaLaunchAttribute at[1];                                                           \
        at[0].id = cudaLaunchAttributeCooperative;                                           \
        at[0].val.cooperative = 1;                                                           \
        cfg.attrs = at;                                                                      \
        cfg.numAttrs = 1;                                                                    \
        return cudaLaunchKernelEx(&cfg, k, a);                                               \
    }
        CME_GRID_SHAPES(CME_CASE)
#undef CME_CASE
    default:
        return cudaErrorInvalidValue;
    }
}

}  // namespace cme
