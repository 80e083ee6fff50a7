// The FP64 step straight from global memory.
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

template <int G, bool AHEAD, typename Args>
__device__ __forceinline__ void direct64_task(const Args &A, const StepConsts<double> &C, int row, int j_raw)
{
    const int j = min(j_raw, A.nr - 1), m = row;
    if (!DBM_DEBUG_CHECK_WARP(j >= 0 && m >= 0 && m < A.ntheta && A.nr <= A.ld, A.status)) return;
    const int mp = m == 0 ? A.ntheta - 1 : m - 1, mn = m == A.ntheta - 1 ? 0 : m + 1;
    const long long at = (long long)m * A.ld + j, dp = (long long)(mp - m) * A.ld, dn = (long long)(mn - m) * A.ld;
    long long dl = j > 0 ? -1 : 0;
    if (C.centre == 2 && j == 0) {  // the site across the centre of a full disc
        const int half = A.ntheta / 2;
        dl = (long long)(m + half < A.ntheta ? half : half - A.ntheta) * A.ld;
    }
    const long long dr = j < A.nr - 1 ? 1 : 0;
    const double *f = A.f_in + at, *l = A.lam_in + at;
    const Places64 p{f, f + dl, f + dr, f + dp, f + dn, l, l + dl, l + dr, l + dp, l + dn};
    site_update64<G, 0, AHEAD>(C, p, A.plane, A.rowtab + (long long)m * 16, A.inv_r[j], j, m, A.ntheta, j_raw < A.nr,
                     A.f_out + at, A.plane, A.lam_out + at);
}

template <bool AHEAD>
__global__ void __launch_bounds__(128) direct64_kernel(const __grid_constant__ Direct64Args D)
{
    const int b = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int full_blocks = (D.full + 3) / 4;
    if (b < full_blocks) {
        const int t = 4 * b + warp;
        if (t < D.full) direct64_task<1, AHEAD>(D.A, D.A.c, t / D.chunks, (t % D.chunks) * 32 + lane);
        return;
    }
    // per_block quarter tasks, on warps that take turns from block to block
    const int n = b - full_blocks, groups = 4 / D.per_block;
    if (warp / D.per_block != n % groups) return;
    const int q = n * D.per_block + warp % D.per_block;
    const int t = D.full + q / 4;
    direct64_task<4, AHEAD>(D.A, D.A.c, t / D.chunks, (t % D.chunks) * 32 + (q & 3) * 8 + (lane & 7));
}

// Whole waves of full tasks; of the rest, quarter tasks where two waves of them
// are enough.
__host__ __device__ inline long long direct64_full(long long tasks, long long quarters)
{
    const long long full = tasks / quarters * quarters;
    return 4 * (tasks - full) > 2 * quarters ? tasks : full;
}

// The same for a batch: persistent warps (the number of tasks is the slot
// table's), tasks over the SMs first, then over their quarters, then over the
// blocks of an SM, so that what whole waves leave over is spread.  Against the
// row ring of items of 16 rows: 28 instances of 128 to 200 sites squared 831 ->
// 631 us per step, 6 of 64 to 200 148 -> 117; 15.1 us per wave of 608 tasks
// where a single 2048^2 takes 14.4.
template <typename real>  // double
__global__ void __launch_bounds__(128) batch_direct64_kernel(const __grid_constant__ BatchArgs<real> B, int nsm)
{
    __shared__ DirectSlot<real> slots[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int tasks = B.n_items[1], full = (int)direct64_full(tasks, 4 * nsm), units = full + 4 * (tasks - full);
    int u = ((int)blockIdx.x / nsm * 4 + warp) * nsm + (int)blockIdx.x % nsm;
    for (int base = 0; base < B.max_slots; base += 32) {
        DirectSlots<real> group;
        group.load(B, base, slots);
        for (; u < units; u += 4 * gridDim.x) {
            const int t = u < full ? u : full + (u - full) / 4;
            if (t >= group.end) break;
            const DirectSlot<real> &A = slots[group.of(t)];
            if (A.cidx < 0) continue;
            const int row = (t - A.first) / A.chunks, col = (t - A.first) % A.chunks * 32;
            if (u < full)
                direct64_task<1, false>(A, batch_consts<real>(A.cidx), row, col + lane);
            else
                direct64_task<4, false>(A, batch_consts<real>(A.cidx), row, col + ((u - full) & 3) * 8 + (lane & 7));
        }
        if (group.end == group.total) break;
    }
}

}  // namespace dbm
