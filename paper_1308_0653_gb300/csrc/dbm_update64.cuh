// The FP64 site update, included by dbm_device.cuh.
//
// What bounds it.  GB300 has few FP64 lanes: an SM quarter issues one FP64 warp
// instruction per 64 cycles alone, an SM one per 19 cycles with its four
// quarters busy, whatever the number of active lanes; conversions and
// comparisons of doubles run at that rate too, everything else is tens of
// times faster.  The step is therefore written for few FP64 instructions:
//   - per ring, the equilibrium and chemical terms of opposite directions are
//     E(w^2) +- w O(w^2), w = e_i . u / T, with E and O's coefficients folded
//     once per ring from rho F_k, v_k's powers and the reaction (15
//     instructions per ring, 6 per pair of directions);
//   - the weights of the site's own f and of its two upwind neighbours are
//     K = D - S / r, A and B = S / r with A, D and S depending on the row and
//     (ring, direction) alone: the 16 (k, i) are spread over the warp's lanes
//     and handed round by shuffles.  A is taken as E - D and B as D - K, E =
//     e^{-dt/tau}: differences that are exact for Courant numbers up to 1/2,
//     so the three weights sum to E and their rounding moves no mass;
//   - upwind signs are read from sign bits.
// About 390 FP64 instructions per site without heat release, 440 with, where
// the same update velocity by velocity took 558: in the row ring 2048^2 went
// from 4.55 to 3.61 ms per step.
#pragma once

namespace dbm {

// 1/x: hardware estimate and two Newton-Raphson steps (r += r (1 - x r)) for
// 2^-1000 <= |x| < 2^1001, else the IEEE division.  The estimate's relative error
// is below 2^-19 (1.0e-6 at most in 2^31 mantissas), the second step's 2^-76, so
// the result is the rounded reciprocal unless that lies within 2^-23 of an ulp of
// halfway between two doubles.  The mantissa of ones alone, whose reciprocal is
// 2^-53 of an ulp from there, came out an ulp low and takes the division too; in
// 2^31 random mantissas there was no difference (dbm_selftest_rcp64).  CUDA's
// __drcp_rn instead: 2048^2 with heat release 3.681 -> 3.731 ms per step.
__device__ __forceinline__ double rcp64(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x);
    const bool ones = (hi & 0xfffffu) == 0xfffffu && __double2loint(x) == -1;
    if (((hi >> 20) & 0x7ffu) - 23u > 2000u || ones) return __ddiv_rn(1.0, x);
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    r = __fma_rn(r, __fma_rn(-x, r, 1.0), r);
    return __fma_rn(r, __fma_rn(-x, r, 1.0), r);
}

__device__ __forceinline__ bool sign_bit(double x) { return __double2hiint(x) < 0; }

// Not +-0 (NaN counts), without an FP64 comparison.
__device__ __forceinline__ bool nonzero(double x)
{
    return ((__double2hiint(x) & 0x7fffffff) | __double2loint(x)) != 0;
}

// A ring's sums, as in ring_moments: s0 = sum g, (sx, sy) = sum g e_i.
__device__ __forceinline__ void ring_sums64(const double *g, double &s0, double &sx, double &sy)
{
    using O = Op<double>;
    const double H = 0.70710678118654752440;  // cos(pi/4)
    s0 = O::add(O::add(O::add(g[0], g[4]), O::add(g[2], g[6])), O::add(O::add(g[1], g[5]), O::add(g[3], g[7])));
    const double a = O::sub(g[1], g[5]), b = O::sub(g[3], g[7]);
    sx = O::fma(H, O::sub(a, b), O::sub(g[0], g[4]));
    sy = O::fma(H, O::add(a, b), O::sub(g[2], g[6]));
}

template <bool B> struct Flag { static constexpr bool value = B; };

// Where a site's values lie: plane 0 of its own f, of its radial neighbours
// (the site itself, or the site across a disc's centre, at a boundary) and of
// rows m - 1 and m + 1, and the same places of lambda.
struct Places64 {
    const double *own, *left, *right, *prev, *next;
    const double *lown, *lleft, *lright, *lprev, *lnext;
};

// One site (G = 1, every lane its own) or a quarter of one (G = 4: lane 8 k + s
// updates ring k of the warp's site s; the moments and the coefficients common
// to the rings are evaluated by all four lanes alike).  All 32 lanes call it;
// `active` lanes store.  Bits do not depend on G.
// AHEAD: neighbours are loaded one ring before their use (70 registers more;
// for warps that have an SM quarter to themselves).  PLANE: distance between the planes of f at p, or 0 where plane_rt gives it.
template <int G, int PLANE, bool AHEAD>
__device__ __forceinline__ void site_update64(const StepConsts<double> &C, const Places64 &p, long long plane_rt,
                                              const double *rt, double inv_r, int j, int m, int ntheta, bool active,
                                              double *out, long long out_plane, double *lam_out)
{
    // sums that could be contracted with a product are written as intrinsics:
    // the bits must not depend on where the compiler inlines this
    using Op64 = Op<double>;
    const auto plane = [&] { if constexpr (PLANE > 0) return PLANE; else return plane_rt; }();
    const unsigned ALL = 0xffffffffu;
    const double H = 0.70710678118654752440;
    const int lane = threadIdx.x & 31;
    const int mine = G == 4 ? lane >> 3 : 0;  // this lane's ring, or the first

    // this lane's (ring, direction) share of the row's weights
    double A_l, D_l, S_l;
    {
        const int k = (lane >> 2) & 3, i = lane & 3;
        S_l = C.v[k] * (C.ct_scale * fabs(rt[8 + i]));
        D_l = Op64::sub(C.decay, C.v[k] * (C.cr_scale * fabs(rt[i])));
        A_l = Op64::sub(C.decay, D_l);
    }

    // moments, summed over the rings in order
    const double f0 = p.own[0];
    double f[G == 4 ? 8 : 32];
    double rho = f0, jx = 0.0, jy = 0.0, e2 = 0.0;
    if constexpr (G == 4) {
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = p.own[(1 + 8 * mine + i) * plane];
        double s0, sx, sy;
        ring_sums64(f, s0, sx, sy);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int src = (lane & 7) + 8 * k;
            const double t0 = __shfl_sync(ALL, s0, src);
            rho += t0;
            jx = fma(C.v[k], __shfl_sync(ALL, sx, src), jx);
            jy = fma(C.v[k], __shfl_sync(ALL, sy, src), jy);
            e2 = fma(C.v2[k], t0, e2);
        }
    } else {
#pragma unroll
        for (int q = 0; q < 32; ++q) f[q] = p.own[(1 + q) * plane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            double s0, sx, sy;
            ring_sums64(f + 8 * k, s0, sx, sy);
            rho += s0;
            jx = fma(C.v[k], sx, jx);
            jy = fma(C.v[k], sy, jy);
            e2 = fma(C.v2[k], s0, e2);
        }
    }
    const double lam = *p.lown;
    // upwind neighbours of ring k
    const bool centre0 = C.centre == 1 && j == 0;
    const bool wrap_prev = C.sector && m == 0, wrap_next = C.sector && m == ntheta - 1;
    auto neighbours = [&](int k, double (&fr)[8], double (&ft)[8]) {
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            // of direction i < 4 by its sign bits; i + 4 the reverse
            const bool inwards = sign_bit(rt[d & 3]) == (d >= 4), below = sign_bit(rt[8 + (d & 3)]) == (d >= 4);
            const double *r = inwards ? p.left : p.right, *t = below ? p.prev : p.next;
            const int q = 1 + 8 * k + d;
            int qr = q, qt = q;
            if (centre0 && inwards) qr += ((d + 4) & 7) - d;
            if (wrap_prev && below) qt += ((d + 1) & 7) - d;
            if (wrap_next && !below) qt += ((d + 7) & 7) - d;
            fr[d] = r[qr * plane];
            ft[d] = t[qt * plane];
        }
    };
    double nr0[8], nt0[8];
    if (AHEAD || G == 4) neighbours(mine, nr0, nt0);
    const double inv_rho = rcp64(rho);
    const double ux = jx * inv_rho, uy = jy * inv_rho;
    const double u2 = fma(ux, ux, uy * uy);
    const double T = 0.5 * fma(e2, inv_rho, -u2);
    const double inv_T = rcp64(T);
    const double P = rho * T;

    // f^eq = rho F_k [A0 + A1 xi + A2 xi^2 + xi^3/6 + xi^4/24], xi = v_k w
    const double hT = 0.5 * inv_T;
    const double hh = u2 * hT;
    const double A1 = Op64::sub(1.0, hh);
    const double A0 = fma(0.5 * hh, hh, A1);
    const double A2 = 0.5 * A1;
    const double wx = ux * inv_T, wy = uy * inv_T;
    const double w[4] = {wx, H * Op64::add(wx, wy), wy, H * Op64::sub(wy, wx)};

    // Cochran rate with ignition gate, exact lambda step.  Below the gate a =
    // b = 0, so the explicit R is 0, or NaN where lambda is not finite, and the
    // consistent one, dlam / dt, is 0.
    double dlam = 0.0;
    const bool no_rate = (((uint32_t)__double2hiint(lam) >> 20) & 0x7ffu) == 0x7ffu && !C.reaction_energy;
    double R = no_rate ? lam - lam : 0.0;
    const bool burns = T > C.T_th;
    if (__any_sync(ALL, burns)) {
        double a = 0.0, b = 0.0;
        if (burns) {
            if (C.general_pow) {
                a = C.omega1 * pow(P, C.m_exp);
                b = C.omega2 * pow(P, C.n_exp);
            } else {
                a = C.omega1 * P;
                b = C.omega2 * P;
            }
        }
        const double om = 1.0 - lam;
        const double g = fma(b, lam, a);
        R = om * g;
        const double sab = Op64::add(a, b);
        if (sab > 0.0) {
            // lam+ - lam = (1-lam)(a+b lam)(E-1) / [(a+b) + (a+b lam)(E-1)], E = e^{(a+b)dt}
            if (nonzero(R)) {
                const double em1 = expm1(sab * C.dt);
                dlam = (R * em1) * rcp64(fma(g, em1, sab));
            }
        }
        if (C.reaction_energy) R = dlam * C.inv_dt;
    }
    // f^eq (1 - E) + dt M = poly(xi) rho F_k (b_k - gam xi), b_k = b0 + v_k^2 bs
    const double gam = (C.dt * (C.Q * R)) * inv_T;
    const double bs = gam * hT;
    const double b0 = fma(fma(-2.0, T, u2), bs, C.one_m_decay);

    double rF[4];
    if constexpr (G == 4) {
        const double own = P * fma(T, fma(T, fma(T, C.Fc[mine][3], C.Fc[mine][2]), C.Fc[mine][1]), C.Fc[mine][0]);
#pragma unroll
        for (int k = 0; k < 4; ++k) rF[k] = __shfl_sync(ALL, own, (lane & 7) + 8 * k);
    } else {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            rF[k] = P * fma(T, fma(T, fma(T, C.Fc[k][3], C.Fc[k][2]), C.Fc[k][1]), C.Fc[k][0]);
    }
    const double rF0 = fma(-8.0, Op64::add(Op64::add(Op64::add(rF[0], rF[1]), rF[2]), rF[3]), rho);
    if (active && (G == 1 || mine == 0)) out[0] = fma(A0, rF0 * b0, C.decay * f0);

    // Ring k: coefficients of E and O, then pairs of opposite directions.  Without
    // heat release (gam = bs = 0) the terms in them are left out: the same bits.
    auto ring = [&](auto heat, int k, const double *fk, double rFk, const double (&fr)[8], const double (&ft)[8]) {
        constexpr bool HEAT = decltype(heat)::value;
        double be, e0, o0, e1, o1, e4, o2 = 0.0;
        if constexpr (HEAT) {
            be = rFk * fma(C.v2[k], bs, b0);
            const double ga = rFk * gam, gA1 = ga * A1;
            e0 = be * A0;
            o0 = C.v[k] * fma(be, A1, -(ga * A0));
            e1 = C.v2[k] * fma(be, A2, -gA1);
            o1 = fma(be, C.v3_6[k], -(gA1 * C.v3_2[k]));
            e4 = fma(be, C.v4_24[k], -(ga * C.v4_6[k]));
            o2 = -ga * C.v5_24[k];
        } else {
            be = rFk * b0;
            e0 = be * A0;
            o0 = C.v[k] * (be * A1);
            e1 = C.v2[k] * (be * A2);
            o1 = be * C.v3_6[k];
            e4 = be * C.v4_24[k];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const double w2 = w[i] * w[i];
            const double E = fma(w2, fma(w2, e4, e1), e0);
            const double O = fma(w2, HEAT ? fma(w2, o2, o1) : o1, o0);
            const int src = 4 * k + i;
            const double A = __shfl_sync(ALL, A_l, src), D = __shfl_sync(ALL, D_l, src);
            const double K = fma(-__shfl_sync(ALL, S_l, src), inv_r, D), B = Op64::sub(D, K);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int d = i + 4 * h;
                const double eq = fma(h ? -w[i] : w[i], O, E);
                const double v = fma(K, fk[d], fma(A, fr[d], fma(B, ft[d], eq)));
                if (active) out[(1 + 8 * k + d) * out_plane] = v;
            }
        }
    };
    auto rings = [&](auto heat) {
        if constexpr (G == 4) {
            ring(heat, mine, f, mine < 2 ? (mine == 0 ? rF[0] : rF[1]) : (mine == 2 ? rF[2] : rF[3]), nr0, nt0);
        } else if constexpr (AHEAD) {
            double nr1[8], nt1[8];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                if (k < 3) neighbours(k + 1, k & 1 ? nr0 : nr1, k & 1 ? nt0 : nt1);
                ring(heat, k, f + 8 * k, rF[k], k & 1 ? nr1 : nr0, k & 1 ? nt1 : nt0);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                neighbours(k, nr0, nt0);
                ring(heat, k, f + 8 * k, rF[k], nr0, nt0);
            }
        }
    };
    if (__any_sync(ALL, nonzero(R)))
        rings(Flag<true>());
    else
        rings(Flag<false>());

    // lambda: exact reaction step + upwind transport
    const double cth = rt[0], sth = -rt[8];
    const double ur = fma(ux, cth, uy * sth), uth = fma(uy, cth, -(ux * sth));
    const double lr = *(sign_bit(ur) ? p.lright : p.lleft), lt = *(sign_bit(uth) ? p.lnext : p.lprev);
    double ln = Op64::add(lam, dlam);
    ln = fma(-(fabs(ur) * C.cr_scale), lam - lr, ln);
    ln = fma(-((fabs(uth) * C.ct_scale) * inv_r), lam - lt, ln);
    if (active && (G == 1 || mine == 0)) *lam_out = fmin(fmax(ln, 0.0), 1.0);
}

// One site of a row ring: lane tx of the strip that starts at j0.
template <int WP, int LAMOFF, int HALO>
__device__ __forceinline__ void site_update64_ring(const StepArgs<double> &A, const StepConsts<double> &C,
                                                   const double *sp, const double *sc, const double *sn, int j0,
                                                   int tx, int m, const double *rt)
{
    const int j = min(j0 + tx, A.nr - 1), col = HALO + j - j0;
    if (!DBM_DEBUG_CHECK_WARP(j >= 0 && A.nr <= A.ld && m >= 0 && m < A.ntheta && col >= 1 && col + 1 < WP, A.status))
        return;
    const int left = col - (j > 0 || C.centre == 2 ? 1 : 0), right = col + (j < A.nr - 1 ? 1 : 0);
    const Places64 p{sc + col,          sc + left,          sc + right,          sp + col,          sn + col,
                     sc + LAMOFF + col, sc + LAMOFF + left, sc + LAMOFF + right, sp + LAMOFF + col, sn + LAMOFF + col};
    const long long at = (long long)m * A.ld + j;
    site_update64<1, WP, false>(C, p, 0, rt, A.inv_r[j], j, m, A.ntheta, j0 + tx < A.nr,
                     A.f_out + at, A.plane, A.lam_out + at);
}

}  // namespace dbm
