// Device code of the polar-coordinate discrete-Boltzmann detonation update
// (Lin, Xu, Zhang, Li, arXiv:1308.0653) for sm_103a.
//
// Data layout in HBM (one instance):
//   f[v][theta][ld]   33 planes, row length ld = nr rounded up to 32 elements,
//                     r contiguous (coalesced 128-byte rows)
//   lam[theta][ld]    reaction variable: lambda (FP64) or 1 - lambda (FP32,
//                     see LamStore)
//   rowtab[theta][16] cos(i pi/4 - theta_m), sin(i pi/4 - theta_m), i = 0..7
//   inv_r[ld]         1 / r_j at cell centres
//
// The fused step kernel is persistent: each CTA owns W consecutive radial
// sites (one per thread) of a run of theta rows ("work item") and marches down
// the rows.  A ring of NSTAGE shared-memory row buffers, each holding all 33
// f planes plus lambda for the strip and a 16-byte halo on both radial sides,
// is filled by TMA (tensor-map tiles, cp.async.bulk.tensor, in the default
// variant; per-array cp.async.bulk in the others), completion on an mbarrier
// per buffer.  Row m is computed from buffers m-1, m, m+1, so every f value
// is read from HBM once per step (plus the halo columns and two halo rows per
// item) and written once.  Variant v1 (march) uses one CTA-wide barrier per
// row; v2/v3 (march2) a producer warp and full/empty mbarriers.
#pragma once

#include <cuda.h>  // CUtensorMap (type only; descriptors are encoded by the host runtime)
#include <cuda_runtime.h>
#include <stdint.h>

namespace dbm {

constexpr int NV = 33;    // D2V33 velocities (Sec. II.B)
constexpr int NARR = 34;  // 33 f planes + lambda

// Status bits written by kernels into the instance's status word.
constexpr int ST_WAIT_TIMEOUT = 1;   // an mbarrier wait gave up
constexpr int ST_NONFINITE = 2;      // a moment was NaN / inf (moments kernel)
constexpr int ST_SMEM_ALIGN = 4;     // dynamic shared memory not 128-byte aligned (step skipped)
constexpr int ST_BOUNDS = 8;         // DBM_DEBUG builds: a copy or store failed its bounds check

// DBM_DEBUG builds check every copy the producer issues (tensor coordinates on
// the 16-byte boundary TMA requires, rows inside the grid, bulk extents inside
// the row and 16-byte aligned) and every global store of the update, and skip
// a failing one with ST_BOUNDS set; a skipped copy ends the step through the
// abort path, like an expired wait.  Release builds compile the checks out.
// Code whose warps vote or shuffle further on asks by whole warps (_WARP): a
// lane that left alone would be waited for.
#ifdef DBM_DEBUG
#define DBM_DEBUG_CHECK(cond, status_ptr) (dbm::debug_check((cond), (status_ptr)))
#define DBM_DEBUG_CHECK_WARP(cond, status_ptr) (!dbm::warp_any(!dbm::debug_check((cond), (status_ptr))))
#else
#define DBM_DEBUG_CHECK(cond, status_ptr) (true)
#define DBM_DEBUG_CHECK_WARP(cond, status_ptr) (true)
#endif
__device__ __forceinline__ bool debug_check(bool ok, int *status)
{
    if (!ok) atomicOr(status, ST_BOUNDS);
    return ok;
}

// Whether x holds in any lane, asked by all 32: the same answer in each.  Lanes
// that each read for themselves a flag that another warp may be setting could
// part, and those that went on would wait for the others in the next vote, shuffle
// or warp barrier without end.
__device__ __forceinline__ bool warp_any(bool x) { return __any_sync(0xffffffffu, x); }

template <typename real> struct Halo;
template <> struct Halo<float> { static constexpr int value = 4; };   // 16 bytes
template <> struct Halo<double> { static constexpr int value = 2; };  // 16 bytes

// Powers of the ring speeds for the FP64 update; nothing for FP32.
template <typename real> struct RingPowers {};
template <> struct RingPowers<double> {
    double v3_6[4], v3_2[4], v4_24[4], v4_6[4], v5_24[4];  // v^3/6, v^3/2, v^4/24, v^4/6, v^5/24
};

// Per-instance constants of the update (host-computed in double, rounded to
// real).  A single-instance launch reads them from its parameter block (the
// constant bank, as instruction operands); a batched launch reads them from
// a constant-memory table indexed by the item's slot.
template <typename real>
struct StepConsts : RingPowers<real> {
    real cr_scale;        // dt / dr
    real ct_scale;        // dt / dtheta
    real decay;           // exp(-dt / tau)
    real one_m_decay;     // 1 - exp(-dt / tau)
    real dt, Q, omega1, omega2, m_exp, n_exp, T_th;
    real inv_dt;          // 1 / dt
    real v[4], v2[4];     // ring speeds and their squares
    real Fc[4][4];        // F_k(T) = T (Fc[k][0] + T (Fc[k][1] + T (Fc[k][2] + T Fc[k][3])))
    int reaction_energy;  // 0 explicit R, 1 consistent R
    int general_pow;      // 0: m = n = 1 (P^m = P), 1: pow()
    int sector;           // 1: pi/4 sector, theta wrap rotates velocities by one direction
    int centre;           // disc centre at r = 0: 1 in a sector (ghost j = -1 is j = 0 with
                          // i -> i+4), 2 on a full grid (ghost is j = 0 of row m + ntheta/2)
};

// Step arguments of one instance and one ping-pong parity.  The tensor maps
// describe this parity's input f as a 3-D tensor (ld, ntheta, 33) and lambda
// as 2-D (ld, ntheta), with a box of one row of W + 2 HALO columns; they are
// used by the tensor-TMA variants.
template <typename real>
struct StepArgs {
    CUtensorMap tm_f;     // 128 B, 64-byte aligned
    CUtensorMap tm_lam;
    CUtensorMap tm_out;   // this parity's output f, box of one row of 32 columns (FP32)
    const real *f_in;
    real *f_out;
    const real *lam_in;
    real *lam_out;
    const real *rowtab;   // [ntheta][16]
    const real *inv_r;    // [ld]
    int *status;          // sticky status word
    long long plane;      // ntheta * ld (elements between f planes)
    int nr, ntheta, ld;
    int strips;           // ceil(nr / W)
    int rows_per_item;    // theta rows per work item
    int segs;             // ceil(ntheta / rows_per_item)
    int items;            // strips * segs
#ifdef DBM_DEBUG
    int stop_loads;       // > 0: a CTA's producer stops after that many rows (dbm_selftest_stop_loads)
#endif
    StepConsts<real> c;
};

// Constant-memory table of the batched launches' per-slot constants (one
// per precision translation unit, defined there).
template <typename real> __device__ const StepConsts<real> &batch_consts(int i);

// ---------------------------------------------------------------------------
// PTX helpers (mbarrier + TMA bulk copy)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// A tensor map read from global memory (the batch slot table, written by host
// copies) must be made visible to the tensor-map proxy before the first
// tensor copy that uses it.
__device__ __forceinline__ void fence_tensormap_acquire(const CUtensorMap *map)
{
    asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(map) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait: gives up after ~2^31 SM cycles (about a second) and reports false.
constexpr long long kWaitLimitCycles = 1LL << 31;

__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  long long limit = kWaitLimitCycles)
{
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > limit) return false;
    }
    return true;
}

// As mbar_try_wait, without suspending: only asks.
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Barrier over the first `nthreads` threads only (id 1; id 0 is __syncthreads).
__device__ __forceinline__ void named_bar_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// Tensor TMA: tile of a 3-D / 2-D tensor map at coordinates (x, y[, z]),
// x innermost; out-of-range elements are filled with zeros.
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z,
                                            uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            smem_addr(dst)),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(smem_addr(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_addr(dst)),
        "l"(map), "r"(x), "r"(y), "r"(smem_addr(bar))
        : "memory");
}

// Tensor TMA store of a tile from shared memory; parts outside the map are
// left out.  Completion by bulk groups of the issuing thread.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, const void *src, int x, int y, int z)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(map),
                 "r"(smem_addr(src)), "r"(x), "r"(y), "r"(z)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_addr(dst)),
        "l"(src), "r"(bytes), "r"(smem_addr(bar))
        : "memory");
}

template <typename real> __device__ __forceinline__ real expm1_(real x);
template <> __device__ __forceinline__ float expm1_<float>(float x) { return expm1f(x); }
template <> __device__ __forceinline__ double expm1_<double>(double x) { return expm1(x); }

template <typename real> __device__ __forceinline__ real pow_(real x, real y);
template <> __device__ __forceinline__ float pow_<float>(float x, float y) { return powf(x, y); }
template <> __device__ __forceinline__ double pow_<double>(double x, double y) { return pow(x, y); }

// ---------------------------------------------------------------------------
// Explicitly rounded arithmetic.  Every operation of the site update is an
// IEEE round-to-nearest intrinsic (no contraction, no reassociation), so the
// update is the same bit pattern in every kernel variant, in batched and
// single launches, and in graph replays.
// ---------------------------------------------------------------------------
template <typename real> struct Op;
template <> struct Op<float> {
    static __device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
    static __device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
    static __device__ __forceinline__ float sub(float a, float b) { return __fsub_rn(a, b); }
    static __device__ __forceinline__ float div(float a, float b) { return __fdiv_rn(a, b); }
    // 1/x for normal, finite x of moderate size (densities, temperatures):
    // the hardware's approximate reciprocal refined by one Newton-Raphson
    // step for f(r) = 1/r - x, r1 = r0 + r0 (1 - x r0).  Branch-free; its
    // error against the correctly rounded reciprocal is checked on the GPU.
    static __device__ __forceinline__ float rcp(float x)
    {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        const float e = __fmaf_rn(-x, r, 1.0f);
        return __fmaf_rn(r, e, r);
    }
};
template <> struct Op<double> {
    static __device__ __forceinline__ double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
    static __device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ double add(double a, double b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ double sub(double a, double b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ double div(double a, double b) { return __ddiv_rn(a, b); }
    static __device__ __forceinline__ double rcp(double x) { return __ddiv_rn(1.0, x); }
};

// ---------------------------------------------------------------------------
// Unbiased rounding of the FP32 reaction variable.  Lambda grows by small
// amounts per step (1e-5 is typical), a few hundred float ulps, and rounding
// each new value to nearest drops the same fraction of an ulp step after step
// while that amount changes slowly: over 20 000 steps of the 2048^2 implosion
// that bias alone left lambda 1.7e-4 behind FP64.  The update is therefore
// summed exactly (TwoSum, Knuth) and rounded to one of the two floats around
// the exact value with probability given by the distance (stochastic
// rounding), which has no bias.  The uniform number comes from a hash of the
// site index and the site's previous value, so the result is a deterministic
// function of the state: identical in every kernel variant, batch and replay.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void two_sum_f(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// 32-bit integer hash (C. Wellons' "lowbias32"): a bijection with full avalanche.
__device__ __forceinline__ uint32_t hash32(uint32_t x)
{
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

// s + e (|e| below a few ulps of s) rounded to a neighbouring float: towards
// the exact value's far neighbour with probability |residual| / ulp, u in [0, 1).
// Values outside (0, 1) are returned rounded to nearest (they are clamped next).
__device__ __forceinline__ float round_stochastic_unit(float s, float e, float u)
{
    const float y = __fadd_rn(s, e);
    if (!(y > 0.f && y < 1.f)) return y;
    const float r = __fadd_rn(__fsub_rn(s, y), e);  // s - y is exact (y is within an ulp of s)
    if (r == 0.f) return y;
    const float other = __int_as_float(__float_as_int(y) + (r > 0.f ? 1 : -1));
    const float gap = fabsf(__fsub_rn(other, y));     // one ulp, exact
    return fabsf(r) > __fmul_rn(u, gap) ? other : y;
}

// ---------------------------------------------------------------------------
// Stored reaction variable.  FP64 stores lambda itself.  FP32 stores the
// unburnt fraction y = 1 - lambda: as lambda -> 1 the reaction increments per
// step fall below half the spacing of floats just under 1 (6e-8) and would
// round away, so lambda would stall short of 1 while the heat release
// computed from (1 - lambda) went on; y keeps them with full relative
// precision.  Near lambda = 0 the spacing of y (6e-8) bounds the absolute
// error of a step instead, far below the reaction increments there.
// ---------------------------------------------------------------------------
template <typename real> struct LamStore {
    static constexpr bool complement = false;
    static __host__ __device__ __forceinline__ double to_lambda(double s) { return s; }
    static __host__ __device__ __forceinline__ double from_lambda(double l) { return l; }
};
template <> struct LamStore<float> {
    static constexpr bool complement = true;
    static __host__ __device__ __forceinline__ double to_lambda(double s) { return 1.0 - s; }
    static __host__ __device__ __forceinline__ double from_lambda(double l) { return 1.0 - l; }
};

// ---------------------------------------------------------------------------
// A site's moments from its 33 f (Sec. II.B), ring by ring in Cartesian
// components: rho = sum f, (jx, jy) = sum f v, e2 = sum f |v|^2.  Within a
// ring the 8 directions are summed pairwise and opposite directions are
// differenced first (exact for nearly equal values).  Shared by the step,
// the FP32 moments and the allocation-free totals, so all see the same values.
// ---------------------------------------------------------------------------
template <typename real>
struct RingSpeeds {
    real v[4], v2[4];  // ring speeds v_k and their squares
};

template <typename real>
__device__ __forceinline__ void ring_moments(const real (&f)[NV], const real (&v)[4], const real (&v2)[4],
                                             real &rho, real &jx, real &jy, real &e2)
{
    using O = Op<real>;
    const real H = real(0.70710678118654752440);  // cos(pi/4)
    rho = f[0];
    jx = real(0);
    jy = real(0);
    e2 = real(0);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const real *g = &f[1 + 8 * k];
        const real s0 = O::add(O::add(O::add(g[0], g[4]), O::add(g[2], g[6])),
                               O::add(O::add(g[1], g[5]), O::add(g[3], g[7])));
        const real a = O::sub(g[1], g[5]), b = O::sub(g[3], g[7]);
        const real sx = O::fma(H, O::sub(a, b), O::sub(g[0], g[4]));
        const real sy = O::fma(H, O::add(a, b), O::sub(g[2], g[6]));
        rho = O::add(rho, s0);
        jx = O::fma(v[k], sx, jx);
        jy = O::fma(v[k], sy, jy);
        e2 = O::fma(v2[k], s0, e2);
    }
}

// ---------------------------------------------------------------------------
// One site's FP32 update (Eq. LB_evolution_equation, Eq. Eqlambda), all 33
// velocities unrolled; returns the new stored reaction variable.  f: the site's
// own values; lst: its stored reaction variable y = 1 - lambda.  Velocity (k,
// i) has Cartesian direction i pi / 4, so its moments and equilibrium use the
// fixed direction cosines; its polar Courant numbers use the row's c_i =
// cos(i pi/4 - theta_m), s_i = sin(...), i < 4.  radial(q, i) and theta(q, i)
// give the upwind neighbours of velocity q in direction i, lam_radial(inner)
// and lam_theta(below) those of y; put(q, v) takes the new f of velocity q.
//
// The 8 velocities of a ring go through each operation together: 8 independent
// instructions in a row, which with two warps per SM quarter is what hides
// their latency (velocity by velocity the same update takes 18 % more cycles
// from shared memory to shared memory).
// ---------------------------------------------------------------------------
template <typename Radial, typename Theta, typename Put, typename LamR, typename LamT>
__device__ __forceinline__ float site_update(const StepConsts<float> &C, const float (&f)[NV], float lst, int ld,
                                                int j, int m, float inv_r, const float (&cs)[4],
                                                const float (&sn4)[4], Radial radial, Theta theta, Put put,
                                                LamR lam_radial, LamT lam_theta)
{
    using O = Op<float>;
    const float H = 0.70710678118654752440f;
    const float lam = O::sub(1.f, lst);

    // --- a2: moments, ring by ring (Cartesian components) ------------------
    //     rho = sum f, rho u = sum f v, e2 = sum f v^2, T = (e2/rho - u^2)/2
    float rho, jx, jy, e2;
    ring_moments<float>(f, C.v, C.v2, rho, jx, jy, e2);
    const float inv_rho = O::rcp(rho);
    const float ux = O::mul(jx, inv_rho), uy = O::mul(jy, inv_rho);
    const float u2 = O::fma(ux, ux, O::mul(uy, uy));
    const float T = O::mul(0.5f, O::sub(O::mul(e2, inv_rho), u2));
    const float inv_T = O::rcp(T);

    // --- a3: weights F_k(T), F_0 = 1 - 8 sum F_k ---------------------------
    float F[4];
    float Fsum = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        F[k] = O::mul(T, O::fma(T, O::fma(T, O::fma(T, C.Fc[k][3], C.Fc[k][2]), C.Fc[k][1]), C.Fc[k][0]));
        Fsum = O::add(Fsum, F[k]);
    }
    const float F0 = O::fma(-8.f, Fsum, 1.f);

    // --- a4 coefficients: f^eq = rho F_k [A0 + A1 xi + A2 xi^2 + xi^3/6 + xi^4/24],
    //     xi = v.u / T = v_k w_i; opposite directions have -w ------------------
    const float hh = O::mul(O::mul(0.5f, u2), inv_T);
    const float A1 = O::sub(1.f, hh);
    const float A0 = O::fma(O::mul(0.5f, hh), hh, A1);
    const float A2 = O::mul(0.5f, A1);
    const float wx = O::mul(ux, inv_T), wy = O::mul(uy, inv_T);
    const float w[4] = {wx, O::mul(H, O::add(wx, wy)), wy, O::mul(H, O::sub(wy, wx))};

    // --- a5: Cochran rate with ignition gate; exact lambda step (a9) -------
    const float P = O::mul(rho, T);
    float a = 0.f, b = 0.f;
    if (T > C.T_th) {
        if (C.general_pow) {
            a = O::mul(C.omega1, pow_(P, C.m_exp));
            b = O::mul(C.omega2, pow_(P, C.n_exp));
        } else {
            a = O::mul(C.omega1, P);
            b = O::mul(C.omega2, P);
        }
    }
    const float g = O::fma(b, lam, a);  // a + b lam
    float R = O::mul(lst, g);
    const float sab = O::add(a, b);
    float dlam = 0.f;
    if (sab > 0.f) {
        // lam+ - lam = (1-lam)(a+b lam)(E-1) / [(a+b) + (a+b lam)(E-1)], E = e^{(a+b)dt}
        const float em1 = expm1_(O::mul(sab, C.dt));
        dlam = O::mul(O::mul(O::mul(lst, g), em1), O::rcp(O::fma(g, em1, sab)));
    }
    if (C.reaction_energy) R = O::mul(dlam, C.inv_dt);

    // --- a6+a7 coefficients: f_new = poly(xi) (beta_k - gamma_k xi) + ... ---
    //     M = f^eq ((v-u)^2 - 2T) / (2T^2) Q R with (v-u)^2 = v_k^2 + u^2 - 2 T xi
    const float dtQR = O::mul(C.dt, O::mul(C.Q, R));
    const float half_inv_T2 = O::mul(O::mul(0.5f, inv_T), inv_T);
    const float gam = O::mul(dtQR, inv_T);
    const float u2m2T = O::fma(-2.f, T, u2);
    const float beta0 = O::mul(O::mul(rho, F0), O::fma(O::mul(dtQR, u2m2T), half_inv_T2, C.one_m_decay));
    put(0, O::fma(A0, beta0, O::mul(C.decay, f[0])));

    // --- a8: |C_r| / v_k, |C_theta| / v_k and their sum, once per opposite pair
    //     (the trig table's entry i + 4 is the exact negation of entry i) ------
    float ar[4], at[4], sa[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        ar[i] = O::mul(fabsf(cs[i]), C.cr_scale);
        at[i] = O::mul(O::mul(fabsf(sn4[i]), C.ct_scale), inv_r);
        sa[i] = O::add(ar[i], at[i]);
    }

    // --- a7 + a11: update all velocities -----------------------------------
    //     f_new = f^eq (1 - E + dt M/f^eq) + (E - |C_r| - |C_th|) f
    //             + |C_r| f(upwind r) + |C_th| f(upwind theta)
    //     with f^eq (1 - E + dt M / f^eq) = poly(xi) (beta_k - gamma_k xi) in ring k
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const float vk = C.v[k];
        const float rF = O::mul(rho, F[k]);
        const float beta = O::mul(rF, O::fma(O::mul(dtQR, O::add(C.v2[k], u2m2T)), half_inv_T2, C.one_m_decay));
        const float gamma = O::mul(rF, gam);
        const int q = 1 + 8 * k;
        float xi[8], pl[8], t[8], adv[8], keep[4];
#pragma unroll
        for (int i = 0; i < 8; ++i) adv[i] = O::mul(at[i & 3], theta(q + i, i));
#pragma unroll
        for (int i = 0; i < 8; ++i) adv[i] = O::fma(ar[i & 3], radial(q + i, i), adv[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) xi[i] = O::mul(vk, w[i]);
#pragma unroll
        for (int i = 0; i < 4; ++i) xi[i + 4] = -xi[i];
#pragma unroll
        for (int i = 0; i < 8; ++i) pl[i] = O::fma(xi[i], float(1.0 / 24.0), float(1.0 / 6.0));
#pragma unroll
        for (int i = 0; i < 8; ++i) pl[i] = O::fma(xi[i], pl[i], A2);
#pragma unroll
        for (int i = 0; i < 8; ++i) pl[i] = O::fma(xi[i], pl[i], A1);
#pragma unroll
        for (int i = 0; i < 8; ++i) pl[i] = O::fma(xi[i], pl[i], A0);
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = O::fma(-gamma, xi[i], beta);
#pragma unroll
        for (int i = 0; i < 4; ++i) keep[i] = O::fma(-vk, sa[i], C.decay);
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = O::mul(pl[i], t[i]);
#pragma unroll
        for (int i = 0; i < 8; ++i) t[i] = O::fma(keep[i & 3], f[q + i], t[i]);
#pragma unroll
        for (int i = 0; i < 8; ++i) put(q + i, O::fma(vk, adv[i], t[i]));
    }

    // --- a9 + a10: lambda = exact reaction step + upwind transport ---------
    const float cth = cs[0], sth = -sn4[0];
    const float ur = O::fma(ux, cth, O::mul(uy, sth));
    const float uth = O::fma(uy, cth, -O::mul(ux, sth));
    const float tr = O::mul(O::mul(fabsf(ur), C.cr_scale), O::sub(lst, lam_radial(ur >= 0.f)));
    const float tt = O::mul(O::mul(O::mul(fabsf(uth), C.ct_scale), inv_r), O::sub(lst, lam_theta(uth >= 0.f)));
    // transport acts on the stored variable alike (y - y_nb = lambda_nb - lambda),
    // the reaction step's dlam is taken off y: y - dlam - tr - tt summed exactly,
    // then rounded without bias
    float sum, err, e;
    two_sum_f(lst, -dlam, sum, err);
    two_sum_f(sum, -tr, sum, e);
    err = __fadd_rn(err, e);
    two_sum_f(sum, -tt, sum, e);
    err = __fadd_rn(err, e);
    const uint32_t site = (uint32_t)m * (uint32_t)ld + (uint32_t)j;
    const float u = (float)(hash32(site * 0x9e3779b9u ^ __float_as_uint(lst)) >> 8) * 0x1p-24f;
    return fminf(fmaxf(round_stochastic_unit(sum, err, u), 0.f), 1.f);
}

// Upwind signs of a row: whether direction i's radial (theta) neighbour is the
// inner (lower) one.  The trig table's entry i + 4 is the negation of entry i.
__device__ __forceinline__ bool upwind_below(const float (&c)[4], int i)
{
    return i < 4 ? c[i & 3] >= 0.f : c[i & 3] <= 0.f;  // C >= 0: backward difference
}

// The update from row buffers in shared memory: sp/sc/sn hold rows m-1, m, m+1,
// col is the site's column.  A row's directions share their signs and a site
// its two radial neighbours, so a neighbour is one select; only a sector's disc
// centre and first and last row turn the velocity set.
// WHOLE: called by whole warps that vote in `put`; false where a check failed
// and nothing was put.
template <int WP, int LAMOFF, bool WHOLE, typename Put>
__device__ __forceinline__ bool ring_site_update(const StepArgs<float> &A, const StepConsts<float> &C,
                                                 const float *__restrict__ sp, const float *__restrict__ sc,
                                                 const float *__restrict__ sn, int col, int j, int m, float inv_r,
                                                 const float (&cs)[4], const float (&sn4)[4], bool active, Put put)
{
    // the site's stores stay inside its instance's planes
    bool ok = DBM_DEBUG_CHECK(j >= 0 && (j < A.nr || !active) && A.nr <= A.ld && m >= 0 && m < A.ntheta, A.status);
    if (!(WHOLE ? DBM_DEBUG_CHECK_WARP(ok, A.status) : ok)) return false;
    float f[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) f[q] = sc[q * WP + col];
    // inner ghost: zero-gradient; on a full disc the site across the centre,
    // which fill_centre_ghost put in the halo column before col
    const float *left = sc + col - (j > 0 || C.centre == 2 ? 1 : 0), *right = sc + col + (j < A.nr - 1 ? 1 : 0);
    const float *prev = sp + col, *next = sn + col;
    const float *rn[8], *tn[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        rn[i] = upwind_below(cs, i) ? left : right;
        tn[i] = upwind_below(sn4, i) ? prev : next;
    }
    if (C.sector) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            if (C.centre == 1 && j == 0 && upwind_below(cs, i)) rn[i] += (((i + 4) & 7) - i) * WP;  // same site, i -> i+4
            if (m == 0 && upwind_below(sn4, i)) tn[i] += (((i + 1) & 7) - i) * WP;  // row -1 = last row, i -> i+1
            if (m == A.ntheta - 1 && !upwind_below(sn4, i)) tn[i] += (((i + 7) & 7) - i) * WP;  // row 0, i -> i-1
        }
    }
#ifdef DBM_DEBUG
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        // velocity planes q = 1 + i .. 25 + i of direction i: neighbour reads
        // stay inside the 33 planes of their row buffer
        const int r = (int)(rn[i] - sc), t = (int)(tn[i] - (upwind_below(sn4, i) ? sp : sn));
        ok = ok && (1 + i) * WP + r >= 0 && (25 + i) * WP + r < NV * WP && (1 + i) * WP + t >= 0 &&
             (25 + i) * WP + t < NV * WP;
    }
    if (!(WHOLE ? DBM_DEBUG_CHECK_WARP(ok, A.status) : DBM_DEBUG_CHECK(ok, A.status))) return false;
#endif
    const float ln = site_update(
        C, f, sc[LAMOFF + col], A.ld, j, m, inv_r, cs, sn4, [&](int q, int i) { return rn[i][q * WP]; },
        [&](int q, int i) { return tn[i][q * WP]; }, put, [&](bool inner) { return (inner ? left : right)[LAMOFF]; },
        [&](bool below) { return (below ? prev : next)[LAMOFF]; });
    if (active) A.lam_out[(long long)m * A.ld + j] = ln;
    return true;
}

}  // namespace dbm

#include "dbm_update64.cuh"

namespace dbm {

// ---------------------------------------------------------------------------
// Full disc (centre == 2, Sec. II.D with a full 2 pi grid): the inner ghost of
// radial site 0 in row m is site 0 of row m + ntheta/2, the point across the
// centre, with the same (Cartesian) velocity and the same lambda.  The thread
// of site 0 copies those 33 f and lambda from the step's input into the halo
// column HALO - 1 of its own row buffer, where its backward differences read
// them; no other thread reads that column of the row.  The caller fences the
// generic writes against the TMA copies that later refill the buffer.
// ---------------------------------------------------------------------------
template <typename real, int WP, int LAMOFF, int HALO>
__device__ __forceinline__ void fill_centre_ghost(const StepArgs<real> &A, real *sc, int m)
{
    const int half = A.ntheta / 2;
    const int mm = m + half < A.ntheta ? m + half : m + half - A.ntheta;
    const real *src = A.f_in + (long long)mm * A.ld;
    real g[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) g[q] = src[(long long)q * A.plane];
    const real lg = A.lam_in[(long long)mm * A.ld];
#pragma unroll
    for (int q = 0; q < NV; ++q) sc[q * WP + HALO - 1] = g[q];
    sc[LAMOFF + HALO - 1] = lg;
}

// ---------------------------------------------------------------------------
// Work lists.  A work item is W radial sites x a run of theta rows of one
// instance.  SingleWork decodes items of one instance arithmetically (its
// arguments live in kernel parameter space); BatchWork reads items of many
// uneven instances from a device table and decides on the device, from the
// global step counter T, which instances are active in this step.
// ---------------------------------------------------------------------------
template <typename real, int W>
struct SingleWork {
    static constexpr bool kCopyArgs = false;
    const StepArgs<real> *A;
    __device__ __forceinline__ int count() const { return A->items; }
    __device__ __forceinline__ bool item(int it, const StepArgs<real> *&a, int &j0, int &mb,
                                         int &me, int &cidx) const
    {
        a = A;
        cidx = -1;
        const int strip = it % A->strips;
        const int seg = it / A->strips;
        j0 = strip * W;
        mb = seg * A->rows_per_item;
        me = min(mb + A->rows_per_item, A->ntheta);
        return true;
    }
};

// One batch slot: the instance's step arguments for both ping-pong parities
// and the global steps [start, end) during which it advances.
template <typename real>
struct BatchSlot {
    StepArgs<real> args[2];  // [p]: reads buffer p, writes buffer 1 - p
    long long start, end;
    int par0;                // the instance's buffer index at global step start
    int cidx;                // the instance's entry in the batch constant table
    int first, chunks;       // straight from global memory: units of the slots before, units per band of rows
};

template <typename real>
struct BatchArgs {
    const BatchSlot<real> *slots;
    const int4 *items;        // (slot, j0, mb, me)
    const int *n_items;       // device words: number of valid items, units of all slots
    const long long *T;       // device word: global step at the start of this replay
    int s;                    // step index within the replay
    int max_slots;
};

// What a unit of a batch stepped straight from global memory needs of its slot.
template <typename real>
struct DirectSlot {
    const real *f_in, *lam_in, *rowtab, *inv_r;
    real *f_out, *lam_out;
    int *status;
    long long plane;
    int nr, ntheta, ld;
    int first, chunks;
    int cidx;  // < 0: does not advance in this step
};

// Such a batch's slots, 32 at a time in shared memory, so that a unit's loads
// do not wait for a chain of table look-ups; the lanes hold the first units.
// An empty slot has no units: the last slot whose first is not beyond a unit
// is the unit's.  Called by all threads of a block.
template <typename real>
struct DirectSlots {
    int first;  // this lane's slot's
    int end;    // the group's last unit + 1
    int total;  // of all units
    __device__ __forceinline__ void load(const BatchArgs<real> &B, int base, DirectSlot<real> (&slots)[32])
    {
        const int s = base + (threadIdx.x & 31);
        total = B.n_items[1];
        end = base + 32 < B.max_slots ? B.slots[base + 32].first : total;
        first = s < B.max_slots ? B.slots[s].first : 0x7fffffff;
        __syncthreads();  // the group before is done with
        if (threadIdx.x < 32 && s < B.max_slots) {
            const BatchSlot<real> &sl = B.slots[s];
            const long long T = *B.T + B.s;
            const StepArgs<real> &A = sl.args[(int)((T - sl.start + sl.par0) & 1)];
            slots[threadIdx.x] = {A.f_in, A.lam_in, A.rowtab, A.inv_r, A.f_out, A.lam_out, A.status, A.plane, A.nr,
                                  A.ntheta, A.ld, first, sl.chunks, T < sl.start || T >= sl.end ? -1 : sl.cidx};
        }
        __syncthreads();
    }
    // The slot of a unit of the group, by all lanes of a warp.
    __device__ __forceinline__ int of(int unit) const
    {
        return __popc(__ballot_sync(0xffffffffu, first <= unit)) - 1;
    }
};

// UNIFORM: a slot's constants through uniform registers (see march2).
template <typename real, int W, bool UNIFORM = false>
struct BatchWork {
    static constexpr bool kCopyArgs = true, kUniform = UNIFORM;
    const BatchSlot<real> *slots;
    const int4 *items;
    int n;
    long long T;
    __device__ __forceinline__ int count() const { return n; }
    __device__ __forceinline__ bool item(int it, const StepArgs<real> *&a, int &j0, int &mb,
                                         int &me, int &cidx) const
    {
        const int4 e = items[it];
        if (e.x < 0) return false;  // padding of the load-balanced table
        const BatchSlot<real> &sl = slots[e.x];
        if (T < sl.start || T >= sl.end) return false;
        a = &sl.args[(int)((T - sl.start + sl.par0) & 1)];
        cidx = sl.cidx;
        j0 = e.y;
        mb = e.z;
        me = e.w;
        return true;
    }
};

// ---------------------------------------------------------------------------
// The fused persistent step: march over this CTA's work items (items
// blockIdx.x, blockIdx.x + gridDim.x, ...), keeping the TMA row ring full
// across item boundaries.
// ---------------------------------------------------------------------------
template <typename real, int W, int NSTAGE, typename Work>
__device__ __forceinline__ void march(const Work &work, unsigned char *smem_raw,
                                      StepArgs<real> *sargs)
{
    constexpr int HALO = Halo<real>::value;
    constexpr int WP = W + 2 * HALO;
    constexpr int SLOT = NARR * WP;  // elements per row buffer
    static_assert(NSTAGE >= 3, "rows m-1, m, m+1 must be resident");

    real *sm = reinterpret_cast<real *>(smem_raw);
    uint64_t *bars = reinterpret_cast<uint64_t *>(smem_raw + sizeof(real) * NSTAGE * SLOT);
    __shared__ int abort_flag;

    const int tx = threadIdx.x;
    const int lane = tx & 31;
    const bool producer = tx < 32;  // warp 0 issues the copies
    const int nitems = work.count();

    if (tx == 0) {
        for (int s = 0; s < NSTAGE; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
        abort_flag = 0;
    }
    __syncthreads();

    // Total row loads of this CTA: rows mb-1 .. me of each active item.
    long long total_loads = 0;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const StepArgs<real> *a;
        int j0, mb, me, cidx;
        if (!work.item(it, a, j0, mb, me, cidx)) continue;
        total_loads += (me - mb) + 2;
#ifdef DBM_DEBUG
        if (a->stop_loads > 0) total_loads = min(total_loads, (long long)a->stop_loads);
#endif
    }

    // Producer cursor (replicated in the lanes of warp 0).
    long long issued = 0;
    int p_item = blockIdx.x, p_row = 0;
    const StepArgs<real> *pa = nullptr;
    int pj0 = 0, pmb = 0, pme = 0, pcidx = 0;
    bool p_ok = false;

    auto issue_one = [&]() {
        while (!p_ok) {  // find the next active item
            p_ok = work.item(p_item, pa, pj0, pmb, pme, pcidx);
            if (!p_ok) p_item += gridDim.x;
        }
        int m = pmb - 1 + p_row;
        const int nth = pa->ntheta;
        m = m < 0 ? m + nth : (m >= nth ? m - nth : m);
        const int slot = (int)(issued % NSTAGE);
        const int jlo = max(pj0 - HALO, 0);
        const int jhi = min(pj0 + W + HALO, (pa->nr + HALO - 1) / HALO * HALO);  // row padding not read
        const uint32_t nbytes = (uint32_t)((jhi - jlo) * (int)sizeof(real));
        real *dst = sm + slot * SLOT + (jlo - (pj0 - HALO));
        if (lane == 0) mbar_arrive_expect_tx(&bars[slot], nbytes * NARR);
        __syncwarp();
        const long long roff = (long long)m * pa->ld + jlo;
        for (int a = lane; a < NARR; a += 32) {
            const real *src = (a < NV) ? pa->f_in + (long long)a * pa->plane + roff : pa->lam_in + roff;
            bulk_g2s(dst + a * WP, src, nbytes, &bars[slot]);
        }
        ++issued;
        if (++p_row == (pme - pmb) + 2) {
            p_row = 0;
            p_item += gridDim.x;
            p_ok = false;
        }
    };

    if (producer) {
        while (issued < NSTAGE && issued < total_loads) issue_one();
    }

    long long base = 0;  // sequence position of the current item's first load
    bool ok = true;
    for (int it = blockIdx.x; it < nitems && ok; it += gridDim.x) {
        const StepArgs<real> *ga;
        int j0, mb, me, cidx;
        if (!work.item(it, ga, j0, mb, me, cidx)) continue;
        const StepArgs<real> *ap = ga;
        if constexpr (Work::kCopyArgs) {
            // per-instance constants into shared memory (read by every thread)
            const int nw = (int)(sizeof(StepArgs<real>) / sizeof(int));
            for (int q = tx; q < nw; q += blockDim.x)
                reinterpret_cast<int *>(sargs)[q] = reinterpret_cast<const int *>(ga)[q];
            __syncthreads();
            ap = sargs;
        }
        const StepArgs<real> &A = *ap;
        const StepConsts<real> &C = Work::kCopyArgs ? batch_consts<real>(cidx) : A.c;
        const int L = me - mb;
        const int j = j0 + tx;
        const bool active = j < A.nr;
        const real inv_r = A.inv_r[active ? j : 0];

        for (int c = 1; c <= L; ++c) {
            const long long P = base + c;
            // wait for rows at positions P-1, P, P+1
            bool late = false;
#pragma unroll
            for (int d = -1; d <= 1; ++d) {
                const long long Q = P + d;
                late = late || !mbar_wait_bounded(&bars[Q % NSTAGE], (uint32_t)((Q / NSTAGE) & 1));
            }
            if (late) {
                atomicOr(A.status, ST_WAIT_TIMEOUT);
                abort_flag = 1;
            }
            const int m = mb + c - 1;
            if constexpr (sizeof(real) == 8) {  // every lane takes part (idle ones store nothing)
                if (!warp_any(late)) {
                    const bool ghost = C.centre == 2 && j == 0;
                    if (ghost) fill_centre_ghost<real, WP, NV * WP, HALO>(A, sm + (P % NSTAGE) * SLOT, m);
                    __syncwarp();
                    site_update64_ring<WP, NV * WP, HALO>(A, C, sm + ((P - 1) % NSTAGE) * SLOT,
                                                          sm + (P % NSTAGE) * SLOT, sm + ((P + 1) % NSTAGE) * SLOT,
                                                          j0, tx, m, A.rowtab + (long long)m * 16);
                    if (ghost) fence_proxy_async_smem();
                }
            } else if (active && !late) {
                real cs[4], sn4[4];
                const real *rt = A.rowtab + (long long)m * 16;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    cs[i] = rt[i];
                    sn4[i] = rt[8 + i];
                }
                const bool ghost = C.centre == 2 && j == 0;
                if (ghost) fill_centre_ghost<real, WP, NV * WP, HALO>(A, sm + (P % NSTAGE) * SLOT, m);
                real *out = A.f_out + (long long)m * A.ld + j;
                ring_site_update<WP, NV * WP, false>(A, C, sm + ((P - 1) % NSTAGE) * SLOT, sm + (P % NSTAGE) * SLOT,
                                         sm + ((P + 1) % NSTAGE) * SLOT, HALO + tx, j, m, inv_r, cs, sn4, true,
                                         [&](int q, float v) { out[(long long)q * A.plane] = v; });
                if (ghost) fence_proxy_async_smem();
            }
            if (__syncthreads_or(*(volatile int *)&abort_flag)) {  // the block's answer
                ok = false;
                break;
            }
            // positions before need_from are no longer read
            const long long need_from = (c < L) ? P : base + L + 2;
            if (producer) {
                fence_proxy_async_smem();
                while (issued < need_from + NSTAGE && issued < total_loads) issue_one();
            }
        }
        base += L + 2;
    }

    if (!ok && tx == 0) {
        // Drain: wait (bounded) for every copy still in flight before exiting.
        for (long long Q = base; Q < issued; ++Q)
            mbar_wait_bounded(&bars[Q % NSTAGE], (uint32_t)((Q / NSTAGE) & 1));
    }
}

template <typename real, int W, int NSTAGE>
__global__ void __launch_bounds__(W, 2) step_kernel(const __grid_constant__ StepArgs<real> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SingleWork<real, W> work{&A};
    march<real, W, NSTAGE>(work, smem_raw, nullptr);
}

template <typename real, int W, int NSTAGE>
__global__ void __launch_bounds__(W, 2) batch_step_kernel(const __grid_constant__ BatchArgs<real> B)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(16) StepArgs<real> sargs;
    BatchWork<real, W> work{B.slots, B.items, *B.n_items, *B.T + B.s};
    march<real, W, NSTAGE>(work, smem_raw, &sargs);
}

// Advance the batch's global step counter after a replay of k steps.
static __global__ void batch_advance_kernel(long long *T, int k)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) *T += k;
}

// Row-buffer layout of the v2 pipeline (in elements of real).
template <typename real, int W>
struct V2Layout {
    static constexpr int wp = W + 2 * Halo<real>::value;
    static constexpr int a128 = 128 / (int)sizeof(real);
    static constexpr int lam = (NV * wp + a128 - 1) / a128 * a128;  // 128-byte aligned
    static constexpr int tab = lam + wp;                            // 16 trig values
    static constexpr int slot = (tab + 16 + a128 - 1) / a128 * a128;
};

// ---------------------------------------------------------------------------
// v2 pipeline: warp-specialised.  Warp W/32 is the producer: it issues the
// TMA bulk copies of each row (34 arrays + the row's 16 trig values) into a
// ring of NSTAGE buffers.  The W/32 consumer warps each update 32 sites of the
// row.  Per buffer, a "full" mbarrier (count 1 + transaction bytes) tells the
// consumers a row has landed, and an "empty" mbarrier (count = consumer warps)
// tells the producer every consumer warp is done with it.  There is no
// CTA-wide barrier per row, so warps drift within the ring instead of waiting
// for the slowest.  Positions are released after their last use: after
// centre P the buffer of P-1, and at an item's last centre also P and P+1.
// ---------------------------------------------------------------------------
template <typename real, int W, int NSTAGE, bool STAGE, bool TMAP, typename Work>
__device__ __forceinline__ void march2(const Work &work, unsigned char *smem_raw,
                                       StepArgs<real> *sargs2)
{
    constexpr int HALO = Halo<real>::value;
    constexpr int WP = W + 2 * HALO;
    constexpr int TAB = 16;
    constexpr int NCW = W / 32;            // consumer warps
    // Row buffer layout (elements): 33 f rows of WP, then lambda at the next
    // 128-byte boundary (tensor-TMA destinations must be 128-byte aligned),
    // then the 16 trig values; the buffer size is a multiple of 128 bytes.
    constexpr int LAMOFF = V2Layout<real, W>::lam;
    constexpr int RTOFF = V2Layout<real, W>::tab;
    constexpr int SLOT = V2Layout<real, W>::slot;
    static_assert(NSTAGE >= 3, "rows m-1, m, m+1 must be resident");
    static_assert((SLOT * sizeof(real)) % 128 == 0, "row buffers must be 128-byte aligned");
    static_assert((LAMOFF * sizeof(real)) % 128 == 0, "lambda tile must be 128-byte aligned");
    static_assert((RTOFF * sizeof(real)) % 16 == 0, "trig row must be 16-byte aligned");

    real *sm = reinterpret_cast<real *>(smem_raw);
    static_assert(!STAGE || (TMAP && sizeof(real) == 4), "staged rows are FP32, stored through a tensor map");
    uint64_t *full = reinterpret_cast<uint64_t *>(smem_raw + sizeof(real) * (NSTAGE * SLOT + (STAGE ? NV * W : 0)));
    uint64_t *empty = full + NSTAGE;
    __shared__ int abort_flag;
    __shared__ int issued_total;

    const int tx = threadIdx.x;
    const int warp = tx >> 5, lane = tx & 31;
    const int nitems = work.count();

    if (tx == 0) {
        for (int s = 0; s < NSTAGE; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], NCW);
        }
        fence_mbar_init();
        abort_flag = 0;
        issued_total = 0;
    }
    __syncthreads();
    if ((smem_addr(smem_raw) & 127u) != 0u) {  // layout assumption broken: report, copy nothing
        if (tx == 0 && nitems > 0) {
            const StepArgs<real> *a;
            int j0, mb, me, cidx;
            for (int it = blockIdx.x; it < nitems; it += gridDim.x)
                if (work.item(it, a, j0, mb, me, cidx)) {
                    atomicOr(a->status, ST_SMEM_ALIGN);
                    break;
                }
        }
        return;
    }

    if (warp == NCW) {
        // ------------------------------ producer ------------------------------
        int total_loads = 0;  // ring positions of this CTA (32-bit: cheap slot arithmetic)
        for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
            const StepArgs<real> *a;
            int j0, mb, me, cidx;
            if (!work.item(it, a, j0, mb, me, cidx)) continue;
            total_loads += (me - mb) + 2;
#ifdef DBM_DEBUG
            if (a->stop_loads > 0) total_loads = min(total_loads, a->stop_loads);
#endif
        }
        int issued = 0;
        int p_item = blockIdx.x, p_row = 0;
        const StepArgs<real> *pa = nullptr;
        int pj0 = 0, pmb = 0, pme = 0, pcidx = 0;
        bool p_ok = false;
        while (issued < total_loads) {
            const int slot = issued % NSTAGE;
            while (!p_ok) {
                p_ok = work.item(p_item, pa, pj0, pmb, pme, pcidx);
                if (!p_ok) p_item += gridDim.x;
            }
            if (issued >= NSTAGE) {
                const uint32_t par = (uint32_t)((issued / NSTAGE - 1) & 1);
                if (!mbar_wait_bounded(&empty[slot], par)) {
                    atomicOr(pa->status, ST_WAIT_TIMEOUT);
                    abort_flag = 1;
                }
                // (a consumer that gave up raised the flag before it let go of a buffer)
                if (warp_any(*(volatile int *)&abort_flag)) break;
            }
            int m = pmb - 1 + p_row;
            const int nth = pa->ntheta;
            m = m < 0 ? m + nth : (m >= nth ? m - nth : m);
            real *buf = sm + slot * SLOT;
#ifdef DBM_DEBUG
            {
                // the row is in the grid; the strip starts inside the row; a tensor
                // box's first column is on a 16-byte boundary; bulk extents are
                // inside the padded row and multiples of 16 bytes
                const int jlo = max(pj0 - HALO, 0), jhi = min(pj0 + W + HALO, (pa->nr + HALO - 1) / HALO * HALO);
                bool ok = m >= 0 && m < nth && pj0 >= 0 && pj0 < pa->nr && pa->nr <= pa->ld;
                if (TMAP) ok = ok && ((pj0 - HALO) * (int)sizeof(real)) % 16 == 0;
                else ok = ok && jhi > jlo && ((jhi - jlo) * (int)sizeof(real)) % 16 == 0 &&
                          (((long long)m * pa->ld + jlo) * (long long)sizeof(real)) % 16 == 0;
                if (!ok) {  // uniform over the warp: every input is
                    if (lane == 0) {
                        atomicOr(pa->status, ST_BOUNDS);
                        abort_flag = 1;
                    }
                    break;
                }
            }
#endif
            if constexpr (TMAP) {
                // one 3-D tile (all 33 f planes of the strip's row), one 2-D tile
                // (lambda), one bulk copy (trig row); the box starts at the
                // halo column pj0 - HALO and out-of-range columns are zeros
                if (lane == 0) {
                    if (Work::kCopyArgs && p_row == 0) {  // maps of a batch slot, in global memory
                        fence_tensormap_acquire(&pa->tm_f);
                        fence_tensormap_acquire(&pa->tm_lam);
                    }
                    mbar_arrive_expect_tx(&full[slot], (uint32_t)(WP * NARR + TAB) * (uint32_t)sizeof(real));  // 33 + 1 rows + trig
                    fence_proxy_async_smem();
                    tma_load_3d(buf, &pa->tm_f, pj0 - HALO, m, 0, &full[slot]);
                    tma_load_2d(buf + LAMOFF, &pa->tm_lam, pj0 - HALO, m, &full[slot]);
                    bulk_g2s(buf + RTOFF, pa->rowtab + (long long)m * TAB, TAB * sizeof(real), &full[slot]);
                }
                __syncwarp();
            } else {
                const int jlo = max(pj0 - HALO, 0);
                const int jhi = min(pj0 + W + HALO, (pa->nr + HALO - 1) / HALO * HALO);  // row padding not read
                const uint32_t nbytes = (uint32_t)((jhi - jlo) * (int)sizeof(real));
                real *dst = buf + (jlo - (pj0 - HALO));
                if (lane == 0) mbar_arrive_expect_tx(&full[slot], nbytes * NARR + TAB * (uint32_t)sizeof(real));
                __syncwarp();
                fence_proxy_async_smem();
                const long long roff = (long long)m * pa->ld + jlo;
                for (int a = lane; a < NARR; a += 32) {
                    const real *src = (a < NV) ? pa->f_in + (long long)a * pa->plane + roff : pa->lam_in + roff;
                    bulk_g2s(a < NV ? dst + a * WP : dst + LAMOFF, src, nbytes, &full[slot]);
                }
                if (lane == 31) bulk_g2s(buf + RTOFF, pa->rowtab + (long long)m * TAB, TAB * sizeof(real), &full[slot]);
            }
            ++issued;
            if (++p_row == (pme - pmb) + 2) {
                p_row = 0;
                p_item += gridDim.x;
                p_ok = false;
            }
        }
        if (lane == 0) issued_total = issued;
    } else {
        // ------------------------------ consumers -----------------------------
        int parity = 0;
        // A warp of which a wait has run out, or that finds the flag of one that has,
        // gives up: it reports, waits for no further row and goes through what is left,
        // staged rows left out and others computed from what is in the buffers, so that
        // it does not part, no barrier is missed, and a step ends a few waits after a
        // row failed to come.  The state is undefined then.
        bool gave_up = false;
        real *stage = sm + NSTAGE * SLOT + warp * (NV * 32);  // STAGE: this warp's outgoing row
        // Ring position taken next: slot and phase parity.  A wait, even for a row
        // that has landed, takes some 150 cycles, so each row asks for the next
        // one's barrier in the middle of its own arithmetic (`landed`).
        int slot = 0;
        uint32_t phase = 0;
        bool landed = false;
        auto ask = [&]() { landed = mbar_test_wait(&full[slot], phase); };
        auto take = [&](const StepArgs<real> &A) -> int {
            // lanes were answered one by one: the warp's decision is a vote
            constexpr bool ASKS = STAGE || sizeof(real) == 8;
            if (!ASKS || warp_any(!landed && !gave_up)) {
                // (having given up: two tries, some 10 us)
                if (!mbar_wait_bounded(&full[slot], phase, gave_up ? 0 : kWaitLimitCycles)) {
                    atomicOr(A.status, ST_WAIT_TIMEOUT);
                    abort_flag = 1;
                }
                if (warp_any(*(volatile int *)&abort_flag)) gave_up = true;
            }
            landed = false;
            const int taken = slot;
            if (++slot == NSTAGE) {
                slot = 0;
                phase ^= 1u;
            }
            return taken;
        };
        // One work item: rows [mb, me) of the strip starting at radial site j0.
        auto run_item = [&](const StepArgs<real> &A, const StepConsts<real> &C, const CUtensorMap *out_map, int j0,
                            int mb, int me) {
            const int j = j0 + tx;
            const bool active = j < A.nr;
            const real inv_r = A.inv_r[active ? j : 0];
            if (gave_up) atomicOr(A.status, ST_WAIT_TIMEOUT);
            int s_prev = take(A), s_cur = take(A);
            for (int m = mb; m < me; ++m) {
                const int s_next = take(A);
                // (all lanes agree already: with this vote 600^2 takes 19.2, without 19.5 us per step)
                if (STAGE && warp_any(gave_up)) return;
                real *sc = sm + s_cur * SLOT;
                const real *sp = sm + s_prev * SLOT, *sn = sm + s_next * SLOT, *rt = sc + RTOFF;
                const bool ghost = C.centre == 2 && j == 0;
                if constexpr (sizeof(real) == 8) {  // every lane takes part (idle ones store nothing)
                    ask();
                    if (ghost) fill_centre_ghost<real, WP, LAMOFF, HALO>(A, sc, m);
                    __syncwarp();
                    site_update64_ring<WP, LAMOFF, HALO>(A, C, sp, sc, sn, j0, tx, m, rt);
                    if (ghost) fence_proxy_async_smem();
                    __syncwarp();
                } else if (STAGE ? !Work::kCopyArgs || j - lane < A.nr : active) {
                    // STAGE: whole warps.  A batch, with many narrow last strips, leaves
                    // out warps without a site (1 % of its time; the test costs a single
                    // simulation 2 to 4 %).
                    real cs[4], sn4[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        cs[i] = rt[i];
                        sn4[i] = rt[8 + i];
                    }
                    if (ghost) fill_centre_ghost<real, WP, LAMOFF, HALO>(A, sc, m);
                    if constexpr (STAGE) {
                        const bool put = ring_site_update<WP, LAMOFF, true>(
                            A, C, sp, sc, sn, HALO + tx, j, m, inv_r, cs, sn4, active, [&](int q, float v) {
                                if (q == 0) {
                                    ask();
                                    // the store before has read the staging row
                                    if (lane == 0) bulk_wait_read();
                                    __syncwarp();
                                }
                                stage[q * 32 + lane] = v;
                            });
                        fence_proxy_async_smem();
                        __syncwarp();
                        if (put && lane == 0 && (Work::kCopyArgs || j < A.nr)) {
                            tma_store_3d(out_map, stage, j, m, 0);
                            bulk_commit();
                        }
                    } else {
                        real *out = A.f_out + (long long)m * A.ld + j;
                        ring_site_update<WP, LAMOFF, false>(A, C, sp, sc, sn, HALO + tx, j, m, inv_r, cs, sn4, true,
                                                            [&](int q, float v) { out[(long long)q * A.plane] = v; });
                        if (ghost) fence_proxy_async_smem();
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(&empty[s_prev]);
                    if (m == me - 1) {
                        mbar_arrive(&empty[s_cur]);
                        mbar_arrive(&empty[s_next]);
                    }
                }
                s_prev = s_cur;
                s_cur = s_next;
            }
        };
        for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
            const StepArgs<real> *ga;
            int j0, mb, me, cidx;
            if (!work.item(it, ga, j0, mb, me, cidx)) continue;
            if constexpr (Work::kCopyArgs) {
                // per-instance constants into shared memory, double-buffered:
                // the barrier of the previous item guarantees nobody still
                // reads the copy made two items ago
                StepArgs<real> *dst = sargs2 + parity;
                const int nw = (int)(sizeof(StepArgs<real>) / sizeof(int));
                for (int q = tx; q < nw; q += W)
                    reinterpret_cast<int *>(dst)[q] = reinterpret_cast<const int *>(ga)[q];
                named_bar_sync(1, W);
                parity ^= 1;
                if (STAGE && lane == 0) fence_tensormap_acquire(&ga->tm_out);
                // The item's pointers and sizes from there into registers for
                // the item (a single instance reads its constants from the
                // constant bank as instruction operands).  Its constants stay
                // in the batch constant table, at an index that the reduction
                // makes uniform, so that they come through uniform registers,
                // or are copied into some 30 registers of every thread: which
                // of the two is faster depends on the batch's size (see
                // batch_uniform).
                const StepArgs<real> Areg = *dst;
                if constexpr (Work::kUniform) {
                    run_item(Areg, batch_consts<real>((int)__reduce_or_sync(0xffffffffu, (unsigned)cidx)), &ga->tm_out, j0,
                             mb, me);
                } else {
                    const StepConsts<real> Creg = batch_consts<real>(cidx);
                    run_item(Areg, Creg, &ga->tm_out, j0, mb, me);
                }
            } else {
                run_item(*ga, ga->c, &ga->tm_out, j0, mb, me);
            }
        }
        if (STAGE && lane == 0) bulk_wait_all();  // rows written, and read out of shared memory
    }
    __syncthreads();
    if (abort_flag && tx == 0) {
        // Drain: wait (bounded) for the copies of the last NSTAGE positions.
        const int n = issued_total;
        for (int Q = (n > NSTAGE ? n - NSTAGE : 0); Q < n; ++Q)
            mbar_wait_bounded(&full[Q % NSTAGE], (uint32_t)((Q / NSTAGE) & 1));
    }
}

template <typename real, int W, int NSTAGE, bool STAGE, int MINB, bool TMAP>
__global__ void __launch_bounds__(W + 32, MINB) step_kernel_v2(const __grid_constant__ StepArgs<real> A)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    SingleWork<real, W> work{&A};
    march2<real, W, NSTAGE, STAGE, TMAP>(work, smem_raw, nullptr);
}

template <typename real, int W, int NSTAGE, bool STAGE, int MINB, bool TMAP, bool UNIFORM>
__global__ void __launch_bounds__(W + 32, MINB) batch_step_kernel_v2(const __grid_constant__ BatchArgs<real> B)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ __align__(64) StepArgs<real> sargs2[2];
    BatchWork<real, W, UNIFORM> work{B.slots, B.items, *B.n_items, *B.T + B.s};
    march2<real, W, NSTAGE, STAGE, TMAP>(work, smem_raw, sargs2);
}

template <typename real, int W, int NSTAGE, bool STAGE>
constexpr int smem_bytes_v2()
{
    return (int)(sizeof(real) * (NSTAGE * V2Layout<real, W>::slot + (STAGE ? NV * W : 0)) + 16 * NSTAGE);
}

// Self-test of the bounded wait every pipeline uses: one CTA waits on an
// mbarrier with `limit` cycles.  With arrive = 0 nothing ever arrives, the
// wait runs out and the kernel reports ST_WAIT_TIMEOUT in *status and returns
// (the context stays usable); with arrive = 1 warp 1 arrives and the wait
// succeeds.
static __global__ void wait_selftest_kernel(int *status, int arrive, long long limit)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (arrive && threadIdx.x == 32) mbar_arrive(&bar);
    if (!mbar_wait_bounded(&bar, 0, limit) && (threadIdx.x & 31) == 0) atomicOr(status, ST_WAIT_TIMEOUT);
}

// Self-test of Op<float>::rcp against the correctly rounded division.
static __global__ void rcp_selftest_kernel(const float *x, float *approx, float *ieee, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        approx[i] = Op<float>::rcp(x[i]);
        ieee[i] = __fdiv_rn(1.0f, x[i]);
    }
}

// Self-test of rcp64 against the correctly rounded division.
static __global__ void rcp64_selftest_kernel(const double *x, double *fast, double *ieee, int n)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        fast[i] = rcp64(x[i]);
        ieee[i] = __ddiv_rn(1.0, x[i]);
    }
}

// ---------------------------------------------------------------------------
// Initial state: f = f^eq(rho, u, T) (Eq. feq) of the initial fields, lambda
// stored.  fields: [5][ntheta][nr] doubles (rho, u_r, u_theta, T, lambda).
// f^eq is evaluated in the state's precision with the arithmetic of the
// step's own equilibrium (weights F_k by Horner, expansion coefficients from
// u^2 / T, xi = v_k (e_i . u) / T), from the fields rounded to `real` and the
// row's cos / sin of the geometry table; opposite directions share the even
// and odd parts of the expansion.  Every value is checked (rho > 0, T > 0,
// all finite): a block that finds a bad one sets *bad, which the host reports
// as DBM_EINVAL (the state is then undefined).
// ---------------------------------------------------------------------------
template <typename real>
struct InitArgs : RingPowers<real> {
    const double *fields;
    real *f;
    real *lam;
    const real *rowtab;  // [ntheta][16]: cos, sin of (i pi/4 - theta_m)
    int *bad;
    long long plane;
    int nr, ntheta, ld;
    int m0, m1;          // theta rows [m0, m1) of this launch
    real v[4], v2[4];
    real Fc[4][4];
};

template <typename real>
__global__ void __launch_bounds__(256) init_kernel(const InitArgs<real> A)
{
    using O = Op<real>;
    const real H = real(0.70710678118654752440);
    const real one = real(1), half = real(0.5);
    const long long N = (long long)A.nr * A.ntheta;
    bool bad = false;
    for (long long s = (long long)A.m0 * A.nr + blockIdx.x * (long long)blockDim.x + threadIdx.x;
         s < (long long)A.m1 * A.nr; s += (long long)gridDim.x * blockDim.x) {
        const int m = (int)(s / A.nr), j = (int)(s - (long long)m * A.nr);
        const double rho_d = A.fields[s], ur_d = A.fields[N + s], uth_d = A.fields[2 * N + s];
        const double T_d = A.fields[3 * N + s], lam_d = A.fields[4 * N + s];
        if (!(rho_d > 0.0) || !(T_d > 0.0) || !isfinite(rho_d) || !isfinite(T_d) || !isfinite(ur_d) ||
            !isfinite(uth_d) || !isfinite(lam_d)) {
            bad = true;
            continue;
        }
        const real rho = (real)rho_d, ur = (real)ur_d, uth = (real)uth_d, T = (real)T_d;
        const real cth = A.rowtab[(long long)m * 16], sth = -A.rowtab[(long long)m * 16 + 8];
        const real ux = O::fma(ur, cth, -O::mul(uth, sth));
        const real uy = O::fma(ur, sth, O::mul(uth, cth));
        const real u2 = O::fma(ux, ux, O::mul(uy, uy));
        const real inv_T = O::rcp(T);
        real F[4], Fsum = real(0);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            F[k] = O::mul(T, O::fma(T, O::fma(T, O::fma(T, A.Fc[k][3], A.Fc[k][2]), A.Fc[k][1]), A.Fc[k][0]));
            Fsum = O::add(Fsum, F[k]);
        }
        const real F0 = O::fma(real(-8), Fsum, one);
        const real hh = O::mul(O::mul(half, u2), inv_T);
        const real A1 = O::sub(one, hh);
        const real A0 = O::fma(O::mul(half, hh), hh, A1);
        const real A2 = O::mul(half, A1);
        const real wx = O::mul(ux, inv_T), wy = O::mul(uy, inv_T);
        const real w[4] = {wx, O::mul(H, O::add(wx, wy)), wy, O::mul(H, O::sub(wy, wx))};
        real *out = A.f + (long long)m * A.ld + j;
        out[0] = O::mul(O::mul(rho, F0), A0);
        if constexpr (sizeof(real) == 8) {
            // bound by FP64 instructions: E(w^2) +- w O(w^2) as in site_update64
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double rF = rho * F[k];
                const double e0 = rF * A0, o0 = A.v[k] * (rF * A1), e1 = A.v2[k] * (rF * A2);
                const double o1 = rF * A.v3_6[k], e4 = rF * A.v4_24[k];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const double w2 = w[i] * w[i];
                    const double Ev = fma(w2, fma(w2, e4, e1), e0), Od = fma(w2, o1, o0);
                    out[(long long)(1 + 8 * k + i) * A.plane] = fma(w[i], Od, Ev);
                    out[(long long)(5 + 8 * k + i) * A.plane] = fma(-w[i], Od, Ev);
                }
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const real rF = O::mul(rho, F[k]);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const real xi = O::mul(A.v[k], w[i]);  // direction i + 4 has -xi
                    const real x2 = O::mul(xi, xi);
                    const real Ev = O::fma(x2, O::fma(x2, real(1.0 / 24.0), A2), A0);
                    const real Od = O::mul(xi, O::fma(x2, real(1.0 / 6.0), A1));
                    out[(long long)(1 + 8 * k + i) * A.plane] = O::mul(rF, O::add(Ev, Od));
                    out[(long long)(5 + 8 * k + i) * A.plane] = O::mul(rF, O::sub(Ev, Od));
                }
            }
        }
        A.lam[(long long)m * A.ld + j] = (real)LamStore<real>::from_lambda(lam_d);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) atomicExch(A.bad, 1);
}

// ---------------------------------------------------------------------------
// FP64 diagnostics.  GB300 issues one FP64 warp instruction per 19 cycles and
// SM (one per 64 cycles and SM quarter), conversions to and from FP64
// included, so these kernels cost what they count in FP64 instructions, tens
// of times their memory time.  A ring's eight f are therefore reduced first,
// by additions alone, to the harmonics its moments need (the velocities of a
// ring are v_k (cos i pi/4, sin i pi/4)), and all moments are taken from the
// few ring harmonics.
// ---------------------------------------------------------------------------
// f widened to FP64.  Floats by shifting their bits, a few integer instructions
// in place of a conversion at the FP64 rate (subnormals excepted).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x)
{
    const uint32_t b = __float_as_uint(x), mag = b & 0x7fffffffu;
    if (mag - 1u < 0x007fffffu) return (double)x;  // subnormal
    uint32_t hi = (mag >> 3) + 0x38000000u;
    if (mag >= 0x7f800000u) hi |= 0x38000000u;  // infinity, NaN
    if (mag == 0u) hi = 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(b << 29));
}

// Harmonics of a ring's f: s0 = sum g, (c1, s1) = sum g (cos, sin)(phi),
// (c2, s2) of 2 phi, (c3, s3) of 3 phi, phi = i pi / 4.
struct RingHarmonics {
    double s0, c1, s1, c2, s2, c3, s3;
};
__device__ __forceinline__ RingHarmonics ring_harmonics(const double (&g)[8])
{
    const double H = 0.70710678118654752440;
    const double p0 = g[0] + g[4], p1 = g[1] + g[5], p2 = g[2] + g[6], p3 = g[3] + g[7];
    const double d0 = g[0] - g[4], d1 = g[1] - g[5], d2 = g[2] - g[6], d3 = g[3] - g[7];
    const double a = d1 - d3, b = d1 + d3;
    RingHarmonics r;
    r.s0 = (p0 + p2) + (p1 + p3);
    r.c2 = p0 - p2;
    r.s2 = p1 - p3;
    r.c1 = fma(H, a, d0);
    r.c3 = fma(-H, a, d0);
    r.s1 = fma(H, b, d2);
    r.s3 = fma(H, b, -d2);
    return r;
}

// ---------------------------------------------------------------------------
// Moments (Sec. II.B) from f, plus per-block partial sums of the
// area-weighted totals {mass, momentum x, momentum y, energy}, summed in FP64
// across sites.  Each site's rho, rho u and sum f v^2 are taken in the state's
// precision ring by ring exactly as the step computes them (ring_moments), u
// and T from those; FP32 values are widened to double (the FP32 state itself
// carries ~6e-8 relative rounding per value, so FP64 per-site arithmetic would
// add no accuracy).  The FP64 kernel is bound by its FP64 instructions: about
// 110 per site this way, 369 with per-velocity sums, a second pass for T and
// the row's angle evaluated at every site.  FP64's T = (sum f v^2 / rho - u^2) / 2
// loses digits to the subtraction as u grows; from about u^2 = 1.5 T on a second pass
// is the more exact (rms error, states within 5 % of f^eq at T = 1: 1.5e-16
// against 2.6e-16 at u = 0.5, 2.6 against 2.7 at 1.25, 7.2 against 4.3 at 2; a
// second pass velocity by velocity 3.4, 3.5 and 4.7), so those sites take it
// (2048^2: 0.84 ms without, 1.64 with every site in it).
// out: [5][ntheta][nr] doubles; partials: [gridDim.x][4] (scratch).
// ---------------------------------------------------------------------------
template <typename real>
struct MomArgs {
    const real *f;
    const real *lam;
    double *out;
    double *partials;
    int *status;
    const real *rowtab;  // [ntheta][16] (moments)
    long long plane;
    int nr, ntheta, ld;
    double r_in, dr, dtheta;
    double th_over_pi;  // theta_m / pi per row
    double v[4], v2[4], v3[4], v4[4];  // ring speeds and their powers
    real vr[4], v2r[4];  // ring speeds and squares in real (moments)
    int m0, m1;          // theta rows [m0, m1) of this launch
};

constexpr int MOMENT_THREADS = 256;

// Sums of four values over a warp: component lane / 8 in every lane.  Halving
// the values while halving the lanes takes 6 additions where a tree per value
// takes 20 (and FP64 additions are what the reduction costs).
__device__ __forceinline__ double warp_sum4(const double (&v)[4], int lane)
{
    const unsigned ALL = 0xffffffffu;
    const bool upper = lane & 16, odd = lane & 8;
    double k0 = upper ? v[2] : v[0], k1 = upper ? v[3] : v[1];
    k0 += __shfl_xor_sync(ALL, upper ? v[0] : v[2], 16);
    k1 += __shfl_xor_sync(ALL, upper ? v[1] : v[3], 16);
    double k = (odd ? k1 : k0) + __shfl_xor_sync(ALL, odd ? k0 : k1, 8);
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(ALL, k, o);
    return k;
}

// T = sum f |v - u|^2 / (2 rho) of an FP64 site in which the flow is fast, from
// its f once more: with w_i = e_i . u, |v_k e_i - u|^2 = (v_k - w_i)^2 + w_{i+2}^2.
__device__ __forceinline__ double peculiar_T(const double *fp, long long plane, const double (&v)[4], double ux,
                                             double uy, double inv_rho)
{
    const double H = 0.70710678118654752440;
    const double w[4] = {ux, H * (ux + uy), uy, H * (uy - ux)};
    double e = fp[0] * fma(ux, ux, uy * uy);
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double w2 = w[(i + 2) & 3] * w[(i + 2) & 3], a = v[k] - w[i], b = v[k] + w[i];
            e = fma(fp[(1 + 8 * k + i) * plane], fma(a, a, w2), e);
            e = fma(fp[(5 + 8 * k + i) * plane], fma(b, b, w2), e);
        }
    }
    return 0.5 * (e * inv_rho);
}

template <typename real>
__global__ void __launch_bounds__(MOMENT_THREADS) moments_kernel(const MomArgs<real> A)
{
    const long long N = (long long)A.nr * A.ntheta;
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    bool bad = false;
    if constexpr (sizeof(real) == 4) {
        using O = Op<float>;
        for (long long s = (long long)A.m0 * A.nr + blockIdx.x * (long long)blockDim.x + threadIdx.x;
             s < (long long)A.m1 * A.nr; s += (long long)gridDim.x * blockDim.x) {
            const int m = (int)(s / A.nr), j = (int)(s - (long long)m * A.nr);
            const float *fp = A.f + (long long)m * A.ld + j;
            float fv[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) fv[q] = fp[(long long)q * A.plane];
            float rho, jx, jy, e2;
            ring_moments<float>(fv, A.vr, A.v2r, rho, jx, jy, e2);
            const float inv_rho = O::rcp(rho);
            const float ux = O::mul(jx, inv_rho), uy = O::mul(jy, inv_rho);
            const float u2 = O::fma(ux, ux, O::mul(uy, uy));
            const float T = O::mul(0.5f, O::sub(O::mul(e2, inv_rho), u2));
            const float cth = A.rowtab[(long long)m * 16], sth = -A.rowtab[(long long)m * 16 + 8];
            const float ur = O::fma(ux, cth, O::mul(uy, sth));
            const float uth = O::fma(uy, cth, -O::mul(ux, sth));
            // conversions by integer shifts: each would cost an FP64 instruction, and
            // those, 16 per site with them and 7 without, would take the time
            const float y = A.lam[(long long)m * A.ld + j];
            if (A.out) {
                A.out[s] = widen(rho);
                A.out[N + s] = widen(ur);
                A.out[2 * N + s] = widen(uth);
                A.out[3 * N + s] = widen(T);
                A.out[4 * N + s] = LamStore<float>::to_lambda(widen(y));
            }
            bad |= !isfinite(rho) || !isfinite(ur) || !isfinite(uth) || !isfinite(T) || !isfinite(y);
            // weight r dr dtheta: dr dtheta applied per block; j + 1/2 from the bits of 2^52 + j
            const double r = fma(__hiloint2double(0x43300000, j) - 4503599627370495.5, A.dr, A.r_in);
            acc[0] = fma(widen(rho), r, acc[0]);
            acc[1] = fma(widen(jx), r, acc[1]);
            acc[2] = fma(widen(jy), r, acc[2]);
            acc[3] = fma(widen(e2), r, acc[3]);  // rho T + rho u^2 / 2 = (1/2) sum f v^2 for D = 2
        }
        const double wa = A.dr * A.dtheta;
        acc[0] *= wa;
        acc[1] *= wa;
        acc[2] *= wa;
        acc[3] *= 0.5 * wa;
    } else {
        const double wa = A.dr * A.dtheta;
        for (long long s = (long long)A.m0 * A.nr + blockIdx.x * (long long)blockDim.x + threadIdx.x;
             s < (long long)A.m1 * A.nr; s += (long long)gridDim.x * blockDim.x) {
            const int m = (int)(s / A.nr), j = (int)(s - (long long)m * A.nr);
            const real *fp = A.f + (long long)m * A.ld + j;
            real fv[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) fv[q] = fp[(long long)q * A.plane];
            real rho, jx, jy, e2;
            ring_moments<real>(fv, A.vr, A.v2r, rho, jx, jy, e2);
            const double inv_rho = 1.0 / rho;
            const double ux = jx * inv_rho, uy = jy * inv_rho;
            const double u2 = fma(ux, ux, uy * uy);
            double T = 0.5 * fma(e2, inv_rho, -u2);
            // by the upper words, FP64 instructions being what this kernel costs: u^2 > 1.25 to 1.5 T
            if (__double2hiint(u2) > __double2hiint(T) + 0x80000LL) T = peculiar_T(fp, A.plane, A.vr, ux, uy, inv_rho);
            const double cth = A.rowtab[(long long)m * 16], sth = -A.rowtab[(long long)m * 16 + 8];
            const double ur = fma(ux, cth, uy * sth), uth = fma(uy, cth, -(ux * sth));
            const double lam = LamStore<real>::to_lambda((double)A.lam[(long long)m * A.ld + j]);
            if (A.out) {
                A.out[s] = rho;
                A.out[N + s] = ur;
                A.out[2 * N + s] = uth;
                A.out[3 * N + s] = T;
                A.out[4 * N + s] = lam;
            }
            bad |= !isfinite(rho) || !isfinite(ur) || !isfinite(uth) || !isfinite(T) || !isfinite(lam);
            const double r = A.r_in + (j + 0.5) * A.dr;  // weight r dr dtheta: dr dtheta applied per block
            acc[0] = fma(rho, r, acc[0]);
            acc[1] = fma(jx, r, acc[1]);
            acc[2] = fma(jy, r, acc[2]);
            acc[3] = fma(e2, r, acc[3]);  // rho T + rho u^2 / 2 = (1/2) sum f v^2 for D = 2
        }
        acc[0] *= wa;
        acc[1] *= wa;
        acc[2] *= wa;
        acc[3] *= 0.5 * wa;
    }
    if (bad) atomicOr(A.status, ST_NONFINITE);
    // deterministic block reduction: each warp, then warp 0 over the 8 warps
    static_assert(MOMENT_THREADS == 256, "one value per lane in the second round");
    __shared__ double red[4][8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const double v = warp_sum4(acc, lane);
    if ((lane & 7) == 0) red[lane >> 3][wid] = v;
    __syncthreads();
    if (wid == 0) {
        double t = red[lane >> 3][lane & 7];
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if ((lane & 7) == 0 && A.partials) A.partials[blockIdx.x * 4 + (lane >> 3)] = t;
    }
}

// Non-equilibrium manifestations (Sec. II.E): Delta*_m = M*_m(f) - M*_m(f^eq)
// in FP64 from f.  The central moments of the discrete f^eq equal the
// Maxwellian's (M*_2 = rho T I, M*_3 = M*_{3,1} = 0, M*_{4,2} = 2 rho T^2 I for
// D = 2), so only f's moments are summed.  out: [12][ntheta][nr] doubles in the
// order rr, rth, thth | rrr, rrth, rthth, ththth | r, th | rr, rth, thth.
// Raw moments of order up to four from the ring harmonics, turned into the
// site's polar frame harmonic by harmonic (an n-th harmonic turns by n theta),
// then made central with u.  About 240 FP64 instructions per site where the
// 33 x 12 direct sums took 1180.  The row's angles are evaluated once per
// block and row.
//
// What u contributes to raw moments is taken off again with its rounding: that
// of Delta*_2's r-theta part, the smallest, passes that of sums over v - u first,
// by 1.3 at u^2 = T / 4 (all others at 0.5 to 1 times theirs) and all of them by
// 2 to 3 at u = 2, T = 1.6.  FP64 sites beyond u^2 = T / 4 take those sums
// (2048^2: 1.90 ms without, 6.0 where every site does; 9.2 with the 33 x 12 sums).
// FP32 states carry 1e9 times that rounding in f and don't.

// Delta* by sums over v - u of an FP64 site's f (about 630 FP64 instructions).
// t: cos, sin of theta; U, V: u in the polar frame.
template <typename real>
__device__ __forceinline__ void central_sums(const real *fp, long long plane, const double (&v)[4], double U,
                                             double V, const double *t, double inv_rho, double *out, long long N)
{
    const double H = 0.70710678118654752440, c = t[0], s = t[1];
    const double ex[4] = {c, H * (c + s), s, H * (s - c)}, ey[4] = {-s, H * (c - s), c, H * (c + s)};
    double rr = 0.0, rt = 0.0, tt = 0.0, rrr = 0.0, rrt = 0.0, rtt = 0.0, ttt = 0.0, f_rr = 0.0, f_rt = 0.0, f_tt = 0.0;
    auto add = [&](double g, double a, double b) {
        const double ga = g * a, gb = g * b, gaa = ga * a, gab = ga * b, gbb = gb * b, s2 = fma(a, a, b * b);
        rr = fma(ga, a, rr);
        rt = fma(ga, b, rt);
        tt = fma(gb, b, tt);
        rrr = fma(gaa, a, rrr);
        rrt = fma(gaa, b, rrt);
        rtt = fma(gbb, a, rtt);
        ttt = fma(gbb, b, ttt);
        f_rr = fma(s2, gaa, f_rr);
        f_rt = fma(s2, gab, f_rt);
        f_tt = fma(s2, gbb, f_tt);
    };
    add(widen(fp[0]), -U, -V);
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            add(widen(fp[(1 + 8 * k + i) * plane]), fma(v[k], ex[i], -U), fma(v[k], ey[i], -V));
            add(widen(fp[(5 + 8 * k + i) * plane]), fma(-v[k], ex[i], -U), fma(-v[k], ey[i], -V));
        }
    }
    const double rT = 0.5 * (rr + tt), rTT2 = 2.0 * rT * (rT * inv_rho);
    out[0] = rr - rT;
    out[N] = rt;
    out[2 * N] = tt - rT;
    out[3 * N] = rrr;
    out[4 * N] = rrt;
    out[5 * N] = rtt;
    out[6 * N] = ttt;
    out[7 * N] = 0.5 * (rrr + rtt);
    out[8 * N] = 0.5 * (rrt + ttt);
    out[9 * N] = fma(0.5, f_rr, -rTT2);
    out[10 * N] = 0.5 * f_rt;
    out[11 * N] = fma(0.5, f_tt, -rTT2);
}

template <typename real>
__global__ void __launch_bounds__(256) noneq_kernel(const MomArgs<real> A)
{
    __shared__ double trig[256][6];  // cos, sin of theta, 2 theta, 3 theta of the block's rows
    const long long N = (long long)A.nr * A.ntheta;
    const long long first = (long long)A.m0 * A.nr, end = (long long)A.m1 * A.nr;
    for (long long base = first + blockIdx.x * 256LL; base < end; base += gridDim.x * 256LL) {
        const int row0 = (int)(base / A.nr);
        const int rows = (int)((min(base + 256, end) - 1) / A.nr) - row0 + 1;
        for (int t = threadIdx.x; t < 3 * rows; t += 256) {
            const int r = t / 3, n = t - 3 * r;
            sincospi((n + 1) * (A.th_over_pi * (row0 + r)), &trig[r][2 * n + 1], &trig[r][2 * n]);
        }
        __syncthreads();
        const long long s = base + threadIdx.x;
        if (s < end) {
            const int m = (int)(s / A.nr), j = (int)(s - (long long)m * A.nr);
            const real *fp = A.f + (long long)m * A.ld + j;
            real fv[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) fv[q] = fp[(long long)q * A.plane];
            // sums over the rings: order 0, 1, 2 (trace and second harmonic), 3
            // (first and third harmonic), 4 (trace and second harmonic)
            double rho = widen(fv[0]), jx = 0.0, jy = 0.0, E2 = 0.0, X2 = 0.0, Y2 = 0.0;
            double A1 = 0.0, B1 = 0.0, A3 = 0.0, B3 = 0.0, E4 = 0.0, X4 = 0.0, Y4 = 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                double g[8];
#pragma unroll
                for (int i = 0; i < 8; ++i) g[i] = widen(fv[1 + 8 * k + i]);
                const RingHarmonics h = ring_harmonics(g);
                rho += h.s0;
                jx = fma(A.v[k], h.c1, jx);
                jy = fma(A.v[k], h.s1, jy);
                E2 = fma(A.v2[k], h.s0, E2);
                X2 = fma(A.v2[k], h.c2, X2);
                Y2 = fma(A.v2[k], h.s2, Y2);
                A1 = fma(A.v3[k], h.c1, A1);
                B1 = fma(A.v3[k], h.s1, B1);
                A3 = fma(A.v3[k], h.c3, A3);
                B3 = fma(A.v3[k], h.s3, B3);
                E4 = fma(A.v4[k], h.s0, E4);
                X4 = fma(A.v4[k], h.c2, X4);
                Y4 = fma(A.v4[k], h.s2, Y4);
            }
            // into the polar frame
            const double *t = trig[m - row0];
            auto turn = [](double &x, double &y, double c, double sn) {
                const double a = fma(x, c, y * sn);
                y = fma(y, c, -(x * sn));
                x = a;
            };
            turn(jx, jy, t[0], t[1]);
            turn(A1, B1, t[0], t[1]);
            turn(X2, Y2, t[2], t[3]);
            turn(X4, Y4, t[2], t[3]);
            turn(A3, B3, t[4], t[5]);
            const double inv_rho = 1.0 / rho;
            const double U = jx * inv_rho, V = jy * inv_rho;
            const double UU = U * U, UV = U * V, VV = V * V, u2 = UU + VV;
            // M*_2 (central): rr, r-theta, theta-theta
            const double rr = fma(-rho, UU, 0.5 * (E2 + X2)), rt = fma(-rho, UV, 0.5 * Y2),
                         tt = fma(-rho, VV, 0.5 * (E2 - X2));
            double *out = A.out + s;
            // u^2 > T / 4, rho u^2 against an eighth of 2 rho T by their upper words
            if (sizeof(real) == 8 && __double2hiint(rho * u2) > __double2hiint(rr + tt) - (3LL << 20)) {
                central_sums(fp, A.plane, A.v, U, V, t, inv_rho, out, N);
            } else {
                // M*_3: raw third moment less u's products with M*_2 and rho u u u
                const double c3 = fma(rho, UU, 3.0 * rr), d3 = fma(rho, VV, 3.0 * tt);
                const double rrr = fma(-U, c3, 0.25 * fma(3.0, A1, A3));
                const double ttt = fma(-V, d3, 0.25 * fma(3.0, B1, -B3));
                const double rrt = fma(-V, fma(rho, UU, rr), fma(-2.0 * U, rt, 0.25 * (B1 + B3)));
                const double rtt = fma(-U, fma(rho, VV, tt), fma(-2.0 * V, rt, 0.25 * (A1 - A3)));
                const double q_r = rrr + rtt, q_t = rrt + ttt;  // sum f |v*|^2 v*
                // 2 M*_{4,2}: sum f |v|^2 v v less what u contributes
                const double tr = rr + tt, w_r = fma(U, rr, V * rt), w_t = fma(U, rt, V * tt);
                const double z = fma(rho, u2, tr);
                const double h_r = q_r + 2.0 * w_r, h_t = q_t + 2.0 * w_t;
                const double f_rr = fma(-UU, z, 0.5 * (E4 + X4)) - 2.0 * fma(U, h_r, fma(U, rrr, V * rrt)) - u2 * rr;
                const double f_tt = fma(-VV, z, 0.5 * (E4 - X4)) - 2.0 * fma(V, h_t, fma(U, rtt, V * ttt)) - u2 * tt;
                const double f_rt = fma(-UV, z, 0.5 * Y4) - fma(V, h_r, U * h_t) - 2.0 * fma(U, rrt, V * rtt) - u2 * rt;
                // less the Maxwellian's: rho T = half the trace, 2 rho T^2
                const double rT = 0.5 * tr, rTT2 = 2.0 * rT * (rT * inv_rho);
                out[0] = rr - rT;
                out[N] = rt;
                out[2 * N] = tt - rT;
                out[3 * N] = rrr;
                out[4 * N] = rrt;
                out[5 * N] = rtt;
                out[6 * N] = ttt;
                out[7 * N] = 0.5 * q_r;
                out[8 * N] = 0.5 * q_t;
                out[9 * N] = fma(0.5, f_rr, -rTT2);
                out[10 * N] = 0.5 * f_rt;
                out[11 * N] = fma(0.5, f_tt, -rTT2);
            }
        }
        __syncthreads();
    }
}

// Sum the per-block partials in a fixed order (one block, a warp per total).
static __global__ void __launch_bounds__(128) totals_kernel(const double *partials, int nblocks, double *totals)
{
    const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double v = 0.0;
    for (int b = lane; b < nblocks; b += 32) v += partials[b * 4 + c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) totals[c] = v;
}

}  // namespace dbm
