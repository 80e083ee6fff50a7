// FP64 kernels (ALU-bound on GB300).  Variants as in the FP32 unit:
//   1  v1  64  5  no   2
//   2  the direct kernel (dbm_direct64.cuh); as launch information, variant 4's shape
//   3  v2  64  4       3
//   4  v3  64  5  no   2   (tensor-map TMA)
//   5  v3  64  4       3   (tensor-map TMA)
#include "dbm.h"
#define DBM_REAL double
#define DBM_VARIANTS(X) X(1, 1, 64, 5, false, 2) X(2, 3, 64, 5, false, 2) X(3, 2, 64, 4, false, 3) \
    X(4, 3, 64, 5, false, 2) X(5, 3, 64, 4, false, 3)
#define DBM_DEFAULT_VARIANT 2
#define DBM_FALLBACK_VARIANT 2
#define DBM_RING_BATCH 0  // batches run the direct kernel
#define DBM_BATCH_CONST_SLOTS DBM_BATCH_CONST_FP64  // batch constant table entries (464 B each)
#include "dbm_launch_impl.cuh"

namespace dbm {
cudaError_t launch_batch_direct64(const BatchArgs<double> &B, int nsm, int blocks_per_sm, cudaStream_t s)
{
    batch_direct64_kernel<double><<<nsm * blocks_per_sm, 128, 0, s>>>(B, nsm);
    return cudaGetLastError();
}

cudaError_t launch_rcp64_selftest(const double *x, double *fast, double *ieee, int n, cudaStream_t s)
{
    rcp64_selftest_kernel<<<256, 256, 0, s>>>(x, fast, ieee, n);
    return cudaGetLastError();
}

cudaError_t batch_direct64_blocks(int *blocks_per_sm)
{
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, (void *)batch_direct64_kernel<double>, 128, 0);
}

cudaError_t launch_direct64(const Direct64Args &D, cudaStream_t s)
{
    // up to two waves of warps, each has an SM quarter (nearly) to itself and
    // its loads are not hidden by others
    const long long tasks = (long long)D.chunks * D.A.ntheta;
    const unsigned blocks = (unsigned)((D.full + 3) / 4 + 4 / D.per_block * (tasks - D.full));
    if (tasks <= 2 * D.quarters)
        direct64_kernel<true><<<blocks, 128, 0, s>>>(D);
    else
        direct64_kernel<false><<<blocks, 128, 0, s>>>(D);
    return cudaGetLastError();
}
}  // namespace dbm
