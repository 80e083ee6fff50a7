// The FP32 step straight from global memory (one simulation).
#pragma once

#include "dbm_device.cuh"

namespace dbm {

// ---------------------------------------------------------------------------
// A warp updates 32 radial sites of a row; a block's four warps the same 32 of
// four rows (log_cols = 5), or 128 sites of one row (7, grids of fewer rows).
// Where the state stays in L2 and a step takes a few microseconds, what counts
// is the time from the launch to the last store: no ring to fill, no barrier,
// the neighbours' lines shared through L1.
// SECTOR: the sector's wraps and disc centre turn the velocity set, so an
// offset can lead to another plane, back or forth (64 bits, signed).
// ---------------------------------------------------------------------------
template <bool SECTOR> struct DirectOffset { using type = uint32_t; };
template <> struct DirectOffset<true> { using type = long long; };

template <bool SECTOR, int MINB>
__global__ void __launch_bounds__(128, MINB) direct32_kernel(const __grid_constant__ StepArgs<float> A, int log_cols)
{
    const StepConsts<float> &C = A.c;
    const int cols = 1 << log_cols, chunks = (A.nr + cols - 1) >> log_cols;
    const int band = blockIdx.x / chunks, chunk = blockIdx.x - band * chunks;
    const int m = (band << (7 - log_cols)) + (threadIdx.x >> log_cols);
    const int j = (chunk << log_cols) + (threadIdx.x & (cols - 1));
    if (m >= A.ntheta || j >= A.nr) return;
    if (!DBM_DEBUG_CHECK(A.nr <= A.ld && m >= 0 && j >= 0, A.status)) return;
    const int mp = m == 0 ? A.ntheta - 1 : m - 1, mn = m == A.ntheta - 1 ? 0 : m + 1;
    const uint32_t ld = (uint32_t)A.ld;
    const uint32_t own = (uint32_t)m * ld + (uint32_t)j;
    uint32_t left = own - (j > 0 ? 1u : 0u);
    const uint32_t right = own + (j < A.nr - 1 ? 1u : 0u);
    const uint32_t prev = (uint32_t)mp * ld + (uint32_t)j, next = (uint32_t)mn * ld + (uint32_t)j;
    if (C.centre == 2 && j == 0)  // the site across the centre of a full disc
        left = (uint32_t)(m + A.ntheta / 2 < A.ntheta ? m + A.ntheta / 2 : m + A.ntheta / 2 - A.ntheta) * ld;

    const float4 c4 = __ldg(reinterpret_cast<const float4 *>(A.rowtab + (long long)m * 16));
    const float4 s4 = __ldg(reinterpret_cast<const float4 *>(A.rowtab + (long long)m * 16 + 8));
    const float cs[4] = {c4.x, c4.y, c4.z, c4.w}, sn4[4] = {s4.x, s4.y, s4.z, s4.w};
    const float *__restrict__ fin = A.f_in, *__restrict__ lin = A.lam_in;
    float *__restrict__ out = A.f_out;
    const long long plane = A.plane;
    float f[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) f[q] = __ldg(fin + q * plane + own);
    typename DirectOffset<SECTOR>::type rn[8], tn[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        rn[i] = upwind_below(cs, i) ? left : right;
        tn[i] = upwind_below(sn4, i) ? prev : next;
        if constexpr (SECTOR) {
            if (C.centre == 1 && j == 0 && upwind_below(cs, i)) rn[i] += (((i + 4) & 7) - i) * plane;
            if (m == 0 && upwind_below(sn4, i)) tn[i] += (((i + 1) & 7) - i) * plane;
            if (m == A.ntheta - 1 && !upwind_below(sn4, i)) tn[i] += (((i + 7) & 7) - i) * plane;
        }
    }
    A.lam_out[own] = site_update(
        C, f, __ldg(lin + own), A.ld, j, m, __ldg(A.inv_r + j), cs, sn4,
        [&](int q, int i) { return __ldg(fin + q * plane + rn[i]); },
        [&](int q, int i) { return __ldg(fin + q * plane + tn[i]); }, [&](int q, float v) { (out + q * plane)[own] = v; },
        [&](bool inner) { return __ldg(lin + (inner ? left : right)); },
        [&](bool below) { return __ldg(lin + (below ? prev : next)); });
}

}  // namespace dbm
