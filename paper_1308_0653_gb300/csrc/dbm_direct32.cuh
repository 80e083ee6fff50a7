// The FP32 step straight from global memory.
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
__host__ __device__ inline int direct32_log_cols(int ntheta) { return ntheta >= 4 ? 5 : 7; }

template <bool SECTOR> struct DirectOffset { using type = uint32_t; };
template <> struct DirectOffset<true> { using type = long long; };

// The site of one thread.
template <bool SECTOR, typename Args>
__device__ __forceinline__ void direct32_site(const Args &A, const StepConsts<float> &C, int m, int j)
{
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

template <bool SECTOR, int MINB>
__global__ void __launch_bounds__(128, MINB) direct32_kernel(const __grid_constant__ StepArgs<float> A, int log_cols)
{
    const int cols = 1 << log_cols, chunks = (A.nr + cols - 1) >> log_cols;
    const int band = blockIdx.x / chunks, chunk = blockIdx.x - band * chunks;
    const int m = (band << (7 - log_cols)) + (threadIdx.x >> log_cols);
    const int j = (chunk << log_cols) + (threadIdx.x & (cols - 1));
    direct32_site<SECTOR>(A, A.c, m, j);
}

// The same for a batch: persistent blocks (the number of tiles is the slot
// table's) and tiles of 128 sites of all slots in turn.  Three blocks per SM:
// four (128 registers) took 16.4 us per step where three take 14.9 (16 instances
// of 64 to 160 sites squared; the row ring 18.8, see batch_direct32 for the line
// between them).  A table look-up per tile instead of the slots in shared
// memory: 15.4.
template <typename real>  // float
__global__ void __launch_bounds__(128, 3) batch_direct32_kernel(const __grid_constant__ BatchArgs<real> B)
{
    __shared__ DirectSlot<real> slots[32];
    int u = blockIdx.x;
    for (int base = 0; base < B.max_slots; base += 32) {
        DirectSlots<real> group;
        group.load(B, base, slots);
        for (; u < group.end; u += gridDim.x) {
            const DirectSlot<real> &A = slots[group.of(u)];
            if (A.cidx < 0) continue;
            const StepConsts<real> &C = batch_consts<real>((int)__reduce_or_sync(0xffffffffu, (unsigned)A.cidx));
            const int log_cols = direct32_log_cols(A.ntheta);
            const int band = (u - A.first) / A.chunks, chunk = u - A.first - band * A.chunks;
            const int m = (band << (7 - log_cols)) + (threadIdx.x >> log_cols);
            const int j = (chunk << log_cols) + (threadIdx.x & ((1 << log_cols) - 1));
            if (C.sector)
                direct32_site<true>(A, C, m, j);
            else
                direct32_site<false>(A, C, m, j);
        }
        if (group.end == group.total) break;
    }
}

}  // namespace dbm
