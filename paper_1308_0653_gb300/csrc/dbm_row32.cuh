// Several FP32 steps per launch of a simulation of one theta row (the paper's
// runs: one theta cell of a pi/4 sector with thousands of radial sites).
#pragma once

#include "dbm_device.cuh"

namespace dbm {

// ---------------------------------------------------------------------------
// A single row is a few microseconds of launch and load latency around one
// microsecond of work, so a launch makes K steps.  A block holds WIDTH
// consecutive sites, one per thread, and loads and stores them once.  A site's
// f stay in its thread's registers; its theta neighbours are its own f with the
// velocities turned (row -1 and row 1 are row 0), its radial neighbours come
// through shared memory, double-buffered, one barrier per step.  A block's edge
// sites are wrong by one site more on each side per step (where the edge is no
// boundary), so it stores only the WIDTH - 2 MAX_STEPS in the middle.
//
// A pass goes from one of the two state buffers to the other, as a step does on
// the other paths.  It makes an odd number of steps, so that the state is in the
// buffer that the number of steps says: dbm_step of an even number, captured into
// a caller's graph, can be replayed.  17 + 15 make the 32 of a step graph (400
// steps of 6000 sites 0.402 ms; 0.399 by passes of 16).
// ---------------------------------------------------------------------------
struct Row32 {
    static constexpr int WIDTH = 128;
    static constexpr int MAX_STEPS = 17;
    static constexpr int STORED = WIDTH - 2 * MAX_STEPS;  // sites per block
    // Steps of the next pass with `left` to go: odd, an even rest of two passes in two.
    static int pass_steps(long long left)
    {
        if (left > 2 * MAX_STEPS || (left % 2 != 0 && left > MAX_STEPS)) return MAX_STEPS;
        return (int)(left % 2 != 0 ? left : (left / 2) | 1);
    }
};

static __global__ void __launch_bounds__(Row32::WIDTH, 2)
row32_kernel(const __grid_constant__ StepArgs<float> A, int steps)
{
    constexpr int W = Row32::WIDTH;
    __shared__ float sm[2][NARR][W];
    const StepConsts<float> &C = A.c;
    const int tx = threadIdx.x;
    const int j_raw = blockIdx.x * Row32::STORED - Row32::MAX_STEPS + tx;
    const int j = min(max(j_raw, 0), A.nr - 1);  // threads outside the row repeat a boundary site, unread
    if (!DBM_DEBUG_CHECK(A.ntheta == 1 && A.nr <= A.ld && steps >= 1 && steps <= Row32::MAX_STEPS, A.status)) return;
    const float inv_r = __ldg(A.inv_r + j);
    float cs[4], sn4[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        cs[i] = __ldg(A.rowtab + i);
        sn4[i] = __ldg(A.rowtab + 8 + i);
    }
    float f[NV], y = __ldg(A.lam_in + j);
#pragma unroll
    for (int q = 0; q < NV; ++q) f[q] = __ldg(A.f_in + q * A.plane + j);
    // neighbour columns: the site itself at a radial boundary and at the block's edge
    const int left = tx - (j_raw > 0 && tx > 0 ? 1 : 0), right = tx + (j_raw < A.nr - 1 && tx < W - 1 ? 1 : 0);
    const bool centre0 = C.centre == 1 && j_raw == 0;  // disc centre: the same site, i -> i + 4
    for (int s = 0; s < steps; ++s) {
        float(&buf)[NARR][W] = sm[s & 1];
#pragma unroll
        for (int q = 0; q < NV; ++q) buf[q][tx] = f[q];
        buf[NV][tx] = y;
        __syncthreads();
        float nw[NV];
        const float *rn[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            rn[i] = &buf[0][upwind_below(cs, i) ? left : right];
            if (centre0 && upwind_below(cs, i)) rn[i] += (((i + 4) & 7) - i) * W;
        }
        y = site_update(
            C, f, y, A.ld, j, 0, inv_r, cs, sn4, [&](int q, int i) { return rn[i][q * W]; },
            [&](int q, int i) {  // row -1: i -> i + 1 in a sector; row 1: i -> i - 1
                const float below = C.sector ? f[q + ((i + 1) & 7) - i] : f[q];
                const float above = C.sector ? f[q + ((i + 7) & 7) - i] : f[q];
                return upwind_below(sn4, i) ? below : above;
            },
            [&](int q, float v) { nw[q] = v; }, [&](bool inner) { return buf[NV][inner ? left : right]; },
            [&](bool) { return y; });
#pragma unroll
        for (int q = 0; q < NV; ++q) f[q] = nw[q];
    }
    if (tx >= Row32::MAX_STEPS && tx < W - Row32::MAX_STEPS && j_raw < A.nr) {
#pragma unroll
        for (int q = 0; q < NV; ++q) A.f_out[q * A.plane + j] = f[q];
        A.lam_out[j] = y;
    }
}

}  // namespace dbm
