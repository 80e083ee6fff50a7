// FP32 kernels.  Variants (id, pipeline, radial sites per CTA, ring depth, rows
// staged in shared memory and stored by TMA, min CTAs per SM):
//   1  v1  128  6  no   2   CTA-wide barrier per row (111 KB shared)
//   2  v2  128  6  no   2   producer warp + full/empty mbarriers (111 KB)
//   3  v2  128  4  no   3   as 2 with a 4-deep ring (74 KB) and <= 136 registers
//   4  v3  128  5  yes  2   as 2, rows loaded and stored by tensor-map TMA
//   5  v3  128  4  no   3   as 3, rows loaded by tensor-map TMA
#include "dbm.h"
#define DBM_REAL float
#define DBM_VARIANTS(X) X(1, 1, 128, 6, false, 2) X(2, 2, 128, 6, false, 2) X(3, 2, 128, 4, false, 3) \
    X(4, 3, 128, 5, true, 2) X(5, 3, 128, 4, false, 3)
#define DBM_DEFAULT_VARIANT 4
#define DBM_FALLBACK_VARIANT 2
#define DBM_RING_BATCH 1
#define DBM_BATCH_CONST_SLOTS DBM_BATCH_CONST_FP32  // batch constant table entries (160 B each)
#include "dbm_launch_impl.cuh"

namespace dbm {
cudaError_t launch_direct32(const StepArgs<float> &A, int nsm, cudaStream_t s)
{
    const int log_cols = direct32_log_cols(A.ntheta), cols = 1 << log_cols, rows = 128 >> log_cols;
    const long long blocks = (long long)((A.nr + cols - 1) / cols) * ((A.ntheta + rows - 1) / rows);
    // Three blocks per SM (168 registers) or four (128): a block's time is 0.81
    // of that with four (64^2, one wave: 2.89 against 3.55 us per step), so what
    // counts is the number of waves (256^2: 5.43 against 5.26; 320^2: 6.88 against 7.03).
    const long long waves3 = (blocks + 3 * nsm - 1) / (3 * nsm), waves4 = (blocks + 4 * nsm - 1) / (4 * nsm);
    if (A.c.sector)
        direct32_kernel<true, 3><<<(unsigned)blocks, 128, 0, s>>>(A, log_cols);
    else if (0.81 * waves3 < waves4)
        direct32_kernel<false, 3><<<(unsigned)blocks, 128, 0, s>>>(A, log_cols);
    else
        direct32_kernel<false, 4><<<(unsigned)blocks, 128, 0, s>>>(A, log_cols);
    return cudaGetLastError();
}

cudaError_t launch_batch_direct32(const BatchArgs<float> &B, int nsm, cudaStream_t s)
{
    batch_direct32_kernel<float><<<3 * nsm, 128, 0, s>>>(B);
    return cudaGetLastError();
}

cudaError_t launch_row32(const StepArgs<float> &A, int steps, cudaStream_t s)
{
    row32_kernel<<<(A.nr + Row32::STORED - 1) / Row32::STORED, Row32::WIDTH, 0, s>>>(A, steps);
    return cudaGetLastError();
}

cudaError_t launch_totals(const double *partials, int nblocks, double *totals, cudaStream_t s)
{
    totals_kernel<<<1, 128, 0, s>>>(partials, nblocks, totals);
    return cudaGetLastError();
}

cudaError_t launch_rcp_selftest(const float *x, float *approx, float *ieee, int n, cudaStream_t s)
{
    rcp_selftest_kernel<<<256, 256, 0, s>>>(x, approx, ieee, n);
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(int *status, int arrive, long long limit, cudaStream_t s)
{
    wait_selftest_kernel<<<1, 64, 0, s>>>(status, arrive, limit);
    return cudaGetLastError();
}

cudaError_t launch_batch_advance(long long *T, int k, cudaStream_t s)
{
    batch_advance_kernel<<<1, 32, 0, s>>>(T, k);
    return cudaGetLastError();
}
}  // namespace dbm
