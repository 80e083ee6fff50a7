// The FP64 step straight from global memory (one simulation).
#pragma once

#include "dbm_device.cuh"

namespace dbm {

// ---------------------------------------------------------------------------
// A task is 32 radial sites of a row, done by one warp ("full") or by four,
// each lane one ring of one of 8 sites; values come straight from global
// memory: an FP64 site takes some 8000 cycles, so a few warps per SM quarter
// hide the loads, and neighbours come from L1 and L2.
//
// A block is four warps, one per SM quarter: four full tasks, or one to four
// quarters of one.  A quarter takes 0.42 of a full task's time, so quarters carry the
// grids that have fewer warps than the chip has SM quarters, and what whole
// waves of full tasks leave over (see fill_direct64).
//
// Against the row ring with the same update: 2048^2 3.61 -> 3.11 ms per step
// (the ring's two CTAs of two consumer warps leave one warp per SM quarter),
// 64^2 17.6 -> 8.3 us (its 64 one-row items used 128 of 608 quarters), 20000 x
// 1 33.8 -> 20.4 us (313 items on 304 CTAs took two waves).
// ---------------------------------------------------------------------------
struct Direct64Args {
    StepArgs<double> A;
    int chunks;  // ceil(nr / 32)
    int full;    // tasks done by one warp each; the others in quarters
    int quarters;   // SM quarters of the device
    int per_block;  // quarter tasks per block: 1, 2 or 4
};

template <int G, bool AHEAD>
__device__ __forceinline__ void direct64_task(const StepArgs<double> &A, int row, int j_raw)
{
    const int j = min(j_raw, A.nr - 1), m = row;
    if (!DBM_DEBUG_CHECK(j >= 0 && m >= 0 && m < A.ntheta && A.nr <= A.ld, A.status)) return;
    const int mp = m == 0 ? A.ntheta - 1 : m - 1, mn = m == A.ntheta - 1 ? 0 : m + 1;
    const long long at = (long long)m * A.ld + j, dp = (long long)(mp - m) * A.ld, dn = (long long)(mn - m) * A.ld;
    long long dl = j > 0 ? -1 : 0;
    if (A.c.centre == 2 && j == 0) {  // the site across the centre of a full disc
        const int half = A.ntheta / 2;
        dl = (long long)(m + half < A.ntheta ? half : half - A.ntheta) * A.ld;
    }
    const long long dr = j < A.nr - 1 ? 1 : 0;
    const double *f = A.f_in + at, *l = A.lam_in + at;
    const Places64 p{f, f + dl, f + dr, f + dp, f + dn, l, l + dl, l + dr, l + dp, l + dn};
    site_update64<G, 0, AHEAD>(A.c, p, A.plane, A.rowtab + (long long)m * 16, A.inv_r[j], j, m, A.ntheta, j_raw < A.nr,
                     A.f_out + at, A.plane, A.lam_out + at);
}

template <bool AHEAD>
__global__ void __launch_bounds__(128) direct64_kernel(const __grid_constant__ Direct64Args D)
{
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int full_blocks = (D.full + 3) / 4;
    if (b < full_blocks) {
        const int t = 4 * b + warp;
        if (t < D.full) direct64_task<1, AHEAD>(D.A, t / D.chunks, (t % D.chunks) * 32 + lane);
        return;
    }
    // per_block quarter tasks, on warps that take turns from block to block
    const int n = b - full_blocks, groups = 4 / D.per_block;
    if (warp / D.per_block != n % groups) return;
    const int q = n * D.per_block + warp % D.per_block;
    const int t = D.full + q / 4;
    direct64_task<4, AHEAD>(D.A, t / D.chunks, (t % D.chunks) * 32 + (q & 3) * 8 + (lane & 7));
}

}  // namespace dbm
