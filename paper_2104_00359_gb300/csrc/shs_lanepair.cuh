// SH products and the projected exponential for 6 to 8 bands, one shading
// point per pair of lanes.
//
// Lane 2q (even) and 2q + 1 (odd) of a warp share a point: the even lane owns
// the SH coefficients with l + |m| even, the odd lane those with l + |m| odd
// (36 and 28 of 64 at 8 bands), so a point's coefficient vectors live in
// registers.  Products run through a quadrature that is exact for their degree
// (truncated Eq. 7): Gauss-Legendre nodes in z come in pairs +-z, and a
// coefficient's Legendre factor is even or odd in z with l + |m|.  Per pair of
// nodes the even lane forms the azimuthal coefficients of the even part E, the
// odd lane those of the odd part O; one exchange gives the even lane E + O
// (the function on the circle z) and the odd lane E - O (the circle -z); each
// lane evaluates its circle, multiplies, and accumulates the products against
// the harmonics; one exchange turns the two circles' sums back into the even
// and the odd part.  On a circle the azimuths phi, -phi, pi - phi, pi + phi
// share cos(m phi), sin(m phi): four sub-sums (cos / sin, even / odd m) give
// all four values, so a circle of 24 azimuths takes 6 x 15 multiply-adds where
// evaluating each azimuth takes 24 x 15.  An 8-band square is about 5.2 k
// FP32 instructions against 13.7 k for the plain separable rule, and no
// operand of the forward pass lives in local memory (the adjoint keeps f and
// the operands of the squarings there: 2.8 KB a thread at 8 bands).  Measured against one thread per point with
// the plain rule (8 bands, 300 spheres, 1M points): forward 5.62 -> 3.1 ms
// (with the pair terms of shs_hi.cuh), adjoint 17.1 -> 8.6 ms; projected
// exponential, forward 4.18 -> 2.61 ms; 6 bands (unrolled Gaunt products
// before), exponential and shading of 200k points 152 -> 75 us.
#pragma once

#include <type_traits>
#include <cuda_runtime.h>

#include "shs_exp.cuh"
#include "shs_point.cuh"

namespace shs {
namespace {

// Slots of a lane's coefficients: for each order m, cos terms then (m > 0) sin
// terms, r = 0, 1, ..: l = m + b + 2 r with b = 0 on the even, 1 on the odd
// lane.  Slots with l >= NB (odd lane, NB - m odd) are empty and hold zero.
__host__ __device__ constexpr int lp_legs(int m) { return (NB - m + 1) / 2; }
__host__ __device__ constexpr int lp_leg(int m, int r) {
    int b = 0;
    for (int k = 0; k < m; ++k) b += lp_legs(k);
    return b + r;
}
__host__ __device__ constexpr int lp_slot(int m, int sn, int r) {
    return m == 0 ? r : lp_legs(0) + 2 * (lp_leg(m, 0) - lp_legs(0)) + sn * lp_legs(m) + r;
}
constexpr int NF = 2 * NB - 1;                   // harmonics 1, cos m phi, sin m phi
constexpr int NL = lp_leg(NB, 0);                // Legendre factors per lane and node
constexpr int NS = 2 * NL - lp_legs(0);          // coefficient slots per lane
constexpr int NSP = (NS + 3) / 4 * 4;
static_assert(NL % 4 == 0, "Legendre tables are read as float4");

// Order and place of slot s (compile-time).
__host__ __device__ constexpr int lp_m(int s) {
    int m = 0;
    while (m + 1 < NB && s >= lp_slot(m + 1, 0, 0)) ++m;
    return m;
}
__host__ __device__ constexpr int lp_sin(int s) {
    return lp_m(s) > 0 && s - lp_slot(lp_m(s), 0, 0) >= lp_legs(lp_m(s)) ? 1 : 0;
}
__host__ __device__ constexpr int lp_l(int s, int b) {
    return lp_m(s) + b + 2 * (s - lp_slot(lp_m(s), lp_sin(s), 0));
}
// Linear SH index of slot s on the lane of parity b; -1 for an empty slot.
__host__ __device__ constexpr int lp_index(int s, int b) {
    return lp_l(s, b) >= NB ? -1 : lp_l(s, b) * (lp_l(s, b) + 1) + (lp_sin(s) ? -lp_m(s) : lp_m(s));
}

// Calls fn(integral_constant<int, I>) for I = 0 .. N - 1: slot arithmetic
// stays in constant expressions.
template <int N, int I = 0, class F>
__device__ __forceinline__ void static_for(F&& fn) {
    if constexpr (I < N) {
        fn(std::integral_constant<int, I>{});
        static_for<N, I + 1>(fn);
    }
}

struct LanePair {
    bool odd;
    float sgn;   // +1 on the even lane, -1 on the odd lane
};

__device__ __forceinline__ LanePair lane_pair() {
    const bool odd = threadIdx.x & 1;
    return LanePair{odd, odd ? -1.f : 1.f};
}

// E + O on the even lane, E - O on the odd lane, from E (even lane) and O (odd
// lane); its own inverse up to the factor the weights carry.
__device__ __forceinline__ float lp_exchange(float v, const LanePair& lp) {
    return fmaf(lp.sgn, v, __shfl_xor_sync(0xffffffffu, v, 1));
}

__device__ __forceinline__ float lp_sum(float v) { return v + __shfl_xor_sync(0xffffffffu, v, 1); }
__device__ __forceinline__ float lp_even(float v) {
    return __shfl_sync(0xffffffffu, v, threadIdx.x & 30);
}

__device__ __forceinline__ void lp_load_legs(const float* tab, float* L) {
    const float4* t4 = reinterpret_cast<const float4*>(tab);
#pragma unroll
    for (int i = 0; i < NL / 4; ++i) {
        const float4 v = t4[i];
        L[4 * i] = v.x;
        L[4 * i + 1] = v.y;
        L[4 * i + 2] = v.z;
        L[4 * i + 3] = v.w;
    }
}

// Azimuthal coefficients of the lane's circle: a holds the lane's slots, ST
// floats apart, but for slot 0, which is a0.
template <int ST = 1>
__device__ __forceinline__ void lp_circle(const float* a, float a0, const float* L, const LanePair& lp, float* c) {
    static_for<NF>([&](auto h) {
        constexpr int m = (h + 1) / 2, sn = m && h % 2 == 0, s = lp_slot(m, sn, 0), g = lp_leg(m, 0);
        float t = (h ? a[s * ST] : a0) * L[g];
#pragma unroll
        for (int r = 1; r < lp_legs(m); ++r) t = fmaf(a[(s + r) * ST], L[g + r], t);
        c[h] = lp_exchange(t, lp);
    });
}

// o += the projection of the circle's sums d.
__device__ __forceinline__ void lp_project(const float* d, const float* L, const LanePair& lp, float* o) {
    static_for<NF>([&](auto h) {
        constexpr int m = (h + 1) / 2, sn = m && h % 2 == 0, s = lp_slot(m, sn, 0), g = lp_leg(m, 0);
        const float t = lp_exchange(d[h], lp);
#pragma unroll
        for (int r = 0; r < lp_legs(m); ++r) o[s + r] = fmaf(t, L[g + r], o[s + r]);
    });
}

// Rows 1, cos phi, sin phi, cos 2 phi, .. of the quads.  ProductRule and
// ExpRule are read in fully unrolled loops, where their entries become
// immediate operands; RolledRule in a rolled loop (constant memory).  Unrolled
// is faster where a kernel has one or two products (forward 0.78 against 0.82
// ms at 262k points, 300 spheres, 8 bands); the adjoint, whose loop bodies
// then outgrow the instruction cache, is faster rolled (step of 1M points 12.4
// against 12.9 ms).
struct ProductRule {
    __device__ __forceinline__ static float trig(int b, int h) { return SH::lp_trig(b, h); }
};
struct ExpRule {
    __device__ __forceinline__ static float trig(int b, int h) { return SH::le_trig(b, h); }
};
struct RolledRule {
    __device__ __forceinline__ static float trig(int b, int h) { return SH::lp_trig_row(b)[h]; }
};

// Values at phi_b, -phi_b, pi - phi_b, pi + phi_b.
template <class R>
__device__ __forceinline__ void lp_values(const float* c, int b, float* v) {
    float ec = c[0], oc = c[1] * R::trig(b, 1), es = 0.f, os = c[2] * R::trig(b, 2);
#pragma unroll
    for (int m = 2; m < NB; ++m) {
        if (m & 1) {
            oc = fmaf(c[2 * m - 1], R::trig(b, 2 * m - 1), oc);
            os = fmaf(c[2 * m], R::trig(b, 2 * m), os);
        } else {
            ec = fmaf(c[2 * m - 1], R::trig(b, 2 * m - 1), ec);
            es = m == 2 ? c[4] * R::trig(b, 4) : fmaf(c[2 * m], R::trig(b, 2 * m), es);
        }
    }
    const float p = ec + oc, q = es + os, r = ec - oc, t = os - es;
    v[0] = p + q;
    v[1] = p - q;
    v[2] = r + t;
    v[3] = r - t;
}

// d += the four values against the harmonics (first: d is set).
template <class R>
__device__ __forceinline__ void lp_accumulate(const float* v, int b, bool first, float* d) {
    const float p = v[0] + v[1], q = v[0] - v[1], r = v[2] + v[3], t = v[2] - v[3];
    const float ec = p + r, oc = p - r, es = q - t, os = q + t;
    d[0] = first ? ec : d[0] + ec;
#pragma unroll
    for (int m = 1; m < NB; ++m) {
        const float xc = (m & 1) ? oc : ec, xs = (m & 1) ? os : es;
        const float tc = R::trig(b, 2 * m - 1), ts = R::trig(b, 2 * m);
        d[2 * m - 1] = first ? xc * tc : fmaf(xc, tc, d[2 * m - 1]);
        d[2 * m] = first ? xs * ts : fmaf(xs, ts, d[2 * m]);
    }
}

// Truncated SH product o = a * b (SQR: a * a).  legs: the lane's first row of
// the product table in shared memory.  The constant parts go separately: with
// a = a_0 y_0 + a~, a * b = a~ * b~ + y_0 (a_0 b~ + b_0 a~) + y_0 a_0 b_0 e_0
// exactly; the exponential's operands are dominated by their constant part,
// and this keeps the rounding of the quadrature sums relative to the small
// remainder.
// The operands' slots are ST floats apart (32: a lane's column of shared
// memory, for kernels that have no registers for them).  ROLLED: see RolledRule.
template <class R, bool SQR>
__device__ __forceinline__ void lp_quad(const float* ca, const float* cb, int q, bool first, float* d) {
    float va[4], vb[4];
    lp_values<R>(ca, q, va);
    if constexpr (!SQR) lp_values<R>(cb, q, vb);
#pragma unroll
    for (int k = 0; k < 4; ++k) va[k] *= SQR ? va[k] : vb[k];
    lp_accumulate<R>(va, q, first, d);
}

template <bool SQR, bool ROLLED = false, int ST = 1>
__device__ __forceinline__ void lp_product(const float* a, const float* b, const float* legs, const LanePair& lp,
                                           float* o) {
    const float a0 = lp_even(a[0]), b0 = SQR ? a0 : lp_even(b[0]);
    const float az = lp.odd ? a[0] : 0.f, bz = SQR ? az : (lp.odd ? b[0] : 0.f);
#pragma unroll
    for (int s = 0; s < NS; ++s) o[s] = 0.f;
#pragma unroll 1
    for (int t = 0; t < SH::LPS; ++t) {
        float L[NL], ca[NF], cb[SQR ? 1 : NF], d[NF];
        lp_load_legs(legs + t * 2 * NL, L);
        lp_circle<ST>(a, az, L, lp, ca);
        if constexpr (!SQR) lp_circle<ST>(b, bz, L, lp, cb);
        if constexpr (ROLLED) {
#pragma unroll
            for (int h = 0; h < NF; ++h) d[h] = 0.f;
#pragma unroll 2
            for (int q = 0; q < SH::LPQ; ++q) lp_quad<RolledRule, SQR>(ca, cb, q, false, d);
        } else {
#pragma unroll
            for (int q = 0; q < SH::LPQ; ++q) lp_quad<ProductRule, SQR>(ca, cb, q, q == 0, d);
        }
        lp_project(d, L, lp, o);
    }
    const float ya = kInvSqrt4Pi * a0, yb = kInvSqrt4Pi * b0;
    o[0] = SQR ? fmaf(2.f * ya, az, o[0]) : fmaf(ya, bz, fmaf(yb, az, o[0]));
    o[0] = fmaf(lp.odd ? 0.f : ya, b0, o[0]);
#pragma unroll
    for (int s = 1; s < NS; ++s)
        o[s] = SQR ? fmaf(2.f * ya, a[s * ST], o[s]) : fmaf(ya, b[s * ST], fmaf(yb, a[s * ST], o[s]));
}

// Projected exponential U = P_n[exp(f^)] (f^ = f without its constant term) by
// the variant's 2n x 4n rule; legs: the lane's first row of the plain table,
// the weighted one follows at LES * 2 * NL.
__device__ __forceinline__ void lp_proj_exp(const float* f, const float* legs, const LanePair& lp, float* U) {
    const float fz = lp.odd ? f[0] : 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s) U[s] = 0.f;
#pragma unroll 1
    for (int t = 0; t < SH::LES; ++t) {
        float L[NL], c[NF], d[NF];
        lp_load_legs(legs + t * 2 * NL, L);
        lp_circle(f, fz, L, lp, c);
#pragma unroll
        for (int q = 0; q < SH::LEQ; ++q) {
            float v[4];
            lp_values<ExpRule>(c, q, v);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = expf(v[k]);
            lp_accumulate<ExpRule>(v, q, q == 0, d);
        }
        lp_load_legs(legs + (SH::LES + t) * 2 * NL, L);
        lp_project(d, L, lp, U);
    }
}

// Adjoint of V = e0 U but for the constant term: for j >= 1,
// df_j = e0 sum_q w_q exp(f^_q) (sum_i dV_i y_i(q)) y_j(q); df_0 is the caller's.
__device__ __forceinline__ void lp_proj_exp_adjoint(const float* f, const float* dV, float e0, const float* legs,
                                                    const LanePair& lp, float* df) {
    const float fz = lp.odd ? f[0] : 0.f;
#pragma unroll
    for (int s = 0; s < NS; ++s) df[s] = 0.f;
#pragma unroll 1
    for (int t = 0; t < SH::LES; ++t) {
        float L[NL], c[NF], g[NF], d[NF];
        lp_load_legs(legs + t * 2 * NL, L);
        lp_circle(f, fz, L, lp, c);
        lp_circle(dV, dV[0], L, lp, g);
#pragma unroll
        for (int q = 0; q < SH::LEQ; ++q) {
            float v[4], u[4];
            lp_values<ExpRule>(c, q, v);
            lp_values<ExpRule>(g, q, u);
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = expf(v[k]) * u[k];
            lp_accumulate<ExpRule>(v, q, q == 0, d);
        }
        lp_load_legs(legs + (SH::LES + t) * 2 * NL, L);
        lp_project(d, L, lp, df);
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) df[s] *= e0;
}

// Columns of the un-normalised SH in z: with R_lm(z) = d^m P_l / dz^m /
// (2l - 1)!!, l = m .. NB - 1, Ybar_l,+-m = (2l - 1)!! R_lm (C_m, S_m) with
// C_m + i S_m = (x + i y)^m, and d R_lm / dz = R_l,m+1.  Each column comes from
// its own three-term recurrence (stable at every z; stepping from column m to
// m + 1 loses several bits near the equator),
//   R_{l+1,m} = z / (l + 1 - m) R_lm - (l + m) / ((4 l^2 - 1)(l + 1 - m)) R_{l-1,m},
// whose first factor z / (i + 1) depends on i = l - m only: zi[i], shared by
// the columns.  col[i] holds l = m + i.
__device__ __forceinline__ void sh_column_factors(float z, float* zi) {
#pragma unroll
    for (int i = 0; i + 1 < NB; ++i) zi[i] = z * (1.f / float(i + 1));
}
template <int M>
__device__ __forceinline__ void sh_column(const float* zi, float* col) {
    if constexpr (M < NB) {
        col[0] = 1.f;
        if constexpr (M + 1 < NB) col[1] = zi[0];
#pragma unroll
        for (int i = 1; i + 1 < NB - M; ++i) {
            const int l = M + i;
            col[i + 1] = fmaf(zi[i], col[i], -(float(l + M) / float((4 * l * l - 1) * (i + 1))) * col[i - 1]);
        }
    }
}
__host__ __device__ constexpr float dfact(int l) {   // (2l - 1)!!
    float v = 1.f;
    for (int k = 1; k < 2 * l; k += 2) v *= float(k);
    return v;
}
// A_hat_l NORM_lm (2l - 1)!!
__device__ __forceinline__ float lobe_factor(int l, int m) {
    return l < NB ? SH::ahat(l) * SH::norm(l * (l + 1) + m) * dfact(l) : 0.f;
}

// The lane's slots of the clamped-cosine lobe H_lm = A_hat_l y_lm(u).
__device__ __forceinline__ void lp_cosine_lobe(float ux, float uy, float uz, const LanePair& lp, float* H) {
    float zi[NB], C = 1.f, S = 0.f;
    sh_column_factors(uz, zi);
    static_for<NB>([&](auto mm) {
        constexpr int m = mm, s = lp_slot(m, 0, 0);
        float col[NB + 1];
        col[NB - m] = 0.f;
        sh_column<m>(zi, col);
        if (m) {
            const float c1 = fmaf(ux, C, -(uy * S)), s1 = fmaf(ux, S, uy * C);
            C = c1;
            S = s1;
        }
#pragma unroll
        for (int r = 0; r < lp_legs(m); ++r) {
            const int l = m + 2 * r;
            const float h = lp.odd ? lobe_factor(l + 1, m) * col[2 * r + 1] : lobe_factor(l, m) * col[2 * r];
            H[s + r] = h * C;
            if (m) H[s + lp_legs(m) + r] = h * S;
        }
    });
}

// Gradient (of some extension off the sphere; the caller projects it) of
// sum_i dH_i A_hat_l y_i(u) with respect to u, from the lane pair's slots.
__device__ __forceinline__ void lp_lobe_adjoint(float ux, float uy, float uz, const float* dH, const LanePair& lp,
                                                float& gx, float& gy, float& gz) {
    float zi[NB], C = 1.f, S = 0.f;
    gx = gy = gz = 0.f;
    sh_column_factors(uz, zi);
    static_for<NB>([&](auto mm) {
        constexpr int m = mm, s = lp_slot(m, 0, 0);
        float col[NB + 1], nxt[NB + 1];   // R_lm from l = m, R_l,m+1 from l = m + 1
        col[NB - m] = nxt[NB - m - 1] = 0.f;
        sh_column<m>(zi, col);
        sh_column<m + 1>(zi, nxt);
        float ac = 0.f, as = 0.f, bc = 0.f, bs = 0.f;
#pragma unroll
        for (int r = 0; r < lp_legs(m); ++r) {
            const int l = m + 2 * r;
            const float q = lp.odd ? lobe_factor(l + 1, m) * col[2 * r + 1] : lobe_factor(l, m) * col[2 * r];
            const float dq = lp.odd ? lobe_factor(l + 1, m) * nxt[2 * r]
                                    : (r ? lobe_factor(l, m) * nxt[r ? 2 * r - 1 : 0] : 0.f);
            const float wc = dH[s + r];
            ac = fmaf(q, wc, ac);
            bc = fmaf(dq, wc, bc);
            if (m) {
                const float ws = dH[s + lp_legs(m) + r];
                as = fmaf(q, ws, as);
                bs = fmaf(dq, ws, bs);
            }
        }
        if (m) {
            const float fm = static_cast<float>(m);   // C, S still hold order m - 1
            gx = fmaf(fm, fmaf(ac, C, as * S), gx);
            gy = fmaf(fm, fmaf(as, C, -(ac * S)), gy);
            const float c1 = fmaf(ux, C, -(uy * S)), s1 = fmaf(ux, S, uy * C);
            C = c1;
            S = s1;
        }
        gz = fmaf(bc, C, fmaf(bs, S, gz));
    });
    gx = lp_sum(gx);
    gy = lp_sum(gy);
    gz = lp_sum(gz);
}

// One exchange of a halving sum over the 16 lanes of one parity: CNT values
// left, lane distance O.  Every index is a compile-time constant.
template <int CNT, int O>
__device__ __forceinline__ void lp_halve(float* v, int lane) {
    if constexpr (O >= 2) {
        constexpr int half = CNT / 2;
        const bool up = lane & O;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const float send = up ? v[i] : v[i + half];
            const float keep = up ? v[i + half] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
        }
        lp_halve<half, O / 2>(v, lane);
    }
}

}  // namespace
}  // namespace shs
