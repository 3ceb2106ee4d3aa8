// Shared by the forward and adjoint kernels of 6, 7 and 8 bands (the method as
// in shs_kern.cu, which holds 1 to 5 bands).
//
// A pair of lanes shares a shading point (shs_lanepair.cuh): 64 points per
// 128-thread block.  In the pair loop each lane sums every second sphere and
// the two halves are exchanged; in the exponential, the shading and their
// adjoints each lane holds half the SH coefficients in registers.
#pragma once

#include "shs_point.cuh"
#include "shs_exp.cuh"
#include "shs_lanepair.cuh"

namespace shs {
namespace {

constexpr int kTile = tile_points(NB);        // points per block tile
constexpr int kWarpPoints = kTile / NWARP;    // points per warp
static_assert(kTile * 2 == kBlock && kWarpPoints == 16, "a lane pair per point");

// One pair's log-visibility terms in the lanes' column form, added to acc:
// acc[m, i] += s2 P_l'(c) R_lm(s_hat) (C_m, S_m), l = m + i (l = 0: 1 - c); the
// factors 1 / (l (l + 1)), (2l - 1)!!, NORM and -2 pi eps follow once per
// point (f_factor).  About 195 FP32 instructions a pair at 8 bands.
__host__ __device__ constexpr int acc_col(int m) { return m ? NB + (m - 1) * (2 * NB - m) : 0; }   // (cos, sin) pairs

template <bool CULL>
__device__ __forceinline__ void pair_forward(float px, float py, float pz, float4 sp, float* acc, Normal u) {
    const PairGeom g = pair_geometry<CULL>(px, py, pz, sp, u);
    float G[NB], zi[NB], C = 1.f, S = 0.f;
    // P_l' by its own recurrence, (l - 1) P_l' = (2l - 1) c P_{l-1}' - l P_{l-2}'
    G[1] = g.s2;
    G[2] = 3.f * (g.c * G[1]);
#pragma unroll
    for (int l = 3; l < NB; ++l)
        G[l] = fmaf((2.f * l - 1.f) / (l - 1.f) * g.c, G[l - 1], -(float(l) / (l - 1.f)) * G[l - 2]);
    G[0] = 1.f - g.c;
    const float sx = g.dx * g.invD, sy = g.dy * g.invD;
    sh_column_factors(g.dz * g.invD, zi);
    static_for<NB>([&](auto mm) {
        constexpr int m = mm, a0 = acc_col(m);
        float col[NB];
        sh_column<m>(zi, col);
        if constexpr (m > 0) {
            const float c1 = fmaf(sx, C, -(sy * S)), s1 = fmaf(sx, S, sy * C);
            C = m == 1 ? sx : c1;
            S = m == 1 ? sy : s1;
        }
#pragma unroll
        for (int i = 0; i < NB - m; ++i) {
            if constexpr (m == 0) {
                acc[i] = i ? fmaf(G[i], col[i], acc[i]) : acc[0] + G[0];
            } else {
                const float h = i ? G[m + i] * col[i] : G[m];
                acc[a0 + 2 * i] = fmaf(h, C, acc[a0 + 2 * i]);
                acc[a0 + 2 * i + 1] = fmaf(h, S, acc[a0 + 2 * i + 1]);
            }
        }
    });
}
// Place of slot s's coefficient in acc on the lane of parity b, and its factor.
__host__ __device__ constexpr int acc_slot(int s, int b) {
    return acc_col(lp_m(s)) + (lp_m(s) ? 2 * (lp_l(s, b) - lp_m(s)) + lp_sin(s) : lp_l(s, b));
}
__device__ __forceinline__ float f_factor(int l, int m) {
    return SH::norm(l * (l + 1) + m) * (dfact(l) / float(l ? l * (l + 1) : 1));
}

// ---------------------------------------------------------------------------
// block state in shared memory
// ---------------------------------------------------------------------------

// Rows of Legendre tables a block keeps: the product rule, and for the
// projected exponential also its own plain and weighted rule.
constexpr int kLegProduct = SH::LPS * 2 * NL, kLegExp = 2 * SH::LES * 2 * NL;

// The lighting in the lanes' slot order, s_lt[b][c][slot], from the staged rows.
__device__ __forceinline__ void slot_lighting(const float* s_light, float (*s_lt)[3][NSP]) {
    for (int e = threadIdx.x; e < 2 * 3 * NSP; e += kBlock) (&s_lt[0][0][0])[e] = 0.f;
    __syncthreads();
    for (int e = threadIdx.x; e < 3 * K; e += kBlock) {
        const int c = e / K, i = e % K;
        int l = 0;
        while ((l + 1) * (l + 1) <= i) ++l;
        const int m = i - l * (l + 1), am = m < 0 ? -m : m, b = (l + am) & 1;
        s_lt[b][c][lp_slot(am, m < 0, (l - am - b) >> 1)] = s_light[c * KPAD + i];
    }
    __syncthreads();
}

__device__ __forceinline__ void load_rules(float* s_leg, bool with_exp) {
    for (int e = threadIdx.x; e < kLegProduct; e += kBlock) s_leg[e] = SH::lp_leg()[e];
    if (with_exp)
        for (int e = threadIdx.x; e < kLegExp; e += kBlock) s_leg[kLegProduct + e] = SH::le_leg()[e];
}

// ---------------------------------------------------------------------------
// log-visibility and exponential
// ---------------------------------------------------------------------------

// The lane's slots of point q of a [K][P] array; zeros for a dead point.
__device__ __forceinline__ void lp_load(const float* src, int64_t P, int64_t q, bool live, const LanePair& lp,
                                        float* v) {
    static_for<NS>([&](auto s) {
        constexpr int i0 = lp_index(s, 0), i1 = lp_index(s, 1);
        v[s] = load_or(src, (lp.odd ? i1 : i0) * P + q, live && (i1 >= 0 || !lp.odd));
    });
}

// ... and the lane's slots stored to point p.
__device__ __forceinline__ void lp_store(const float* v, int64_t P, int64_t p, const LanePair& lp, float* dst) {
    static_for<NS>([&](auto s) {
        constexpr int i0 = lp_index(s, 0), i1 = lp_index(s, 1);
        if (i1 >= 0 || !lp.odd) dst[(lp.odd ? i1 : i0) * P + p] = v[s];
    });
}

// The exponential a kernel is compiled for; kExpAny: asked of each scene.
constexpr int kExpSquarings = 0, kExpProjected = 1, kExpAny = 2;
template <int EXPM>
__device__ __forceinline__ bool projected_exp(const SceneView& sc) {
    return EXPM == kExpAny ? sc.exp_mode == 1 : EXPM == kExpProjected;
}

// Unit normal for a kernel compiled with culling: a scene that does not cull
// gets NaN, which no sphere's test is below.
__device__ __forceinline__ Normal cull_normal(const SceneView& sc, float nx, float ny, float nz) {
    const float off = __int_as_float(0x7fffffff);
    return sc.horizon_cull ? unit_normal(nx, ny, nz) : Normal{off, off, off};
}

// Log-visibility f of the lane pair's point: each lane sums every second
// sphere, then the lanes exchange halves and keep their own slots.
template <bool CULL>
__device__ __forceinline__ void lp_log_visibility(const SceneView& sc, const float4* s_sph, float px, float py,
                                                  float pz, Normal u, const LanePair& lp, float* f) {
    float acc[K];
#pragma unroll
    for (int i = 0; i < K; ++i) acc[i] = 0.f;
#pragma unroll 1
    for (int j = lp.odd ? 1 : 0; j < sc.n_spheres; j += 2) pair_forward<CULL>(px, py, pz, s_sph[j], acc, u);
    __syncwarp();
    static_for<NS>([&](auto s) {
        constexpr int m = lp_m(s), l0 = lp_l(s, 0), l1 = lp_l(s, 1), j0 = acc_slot(s, 0),
                      j1 = l1 < NB ? acc_slot(s, 1) : 0;
        const float v0 = acc[j0], v1 = l1 < NB ? acc[j1] : 0.f;
        const float own = (lp.odd ? v1 : v0) + __shfl_xor_sync(0xffffffffu, lp.odd ? v0 : v1, 1);
        f[s] = sc.neg_2pi_eps * (lp.odd ? (l1 < NB ? f_factor(l1, m) : 0.f) : f_factor(l0, m)) * own;
    });
}

// Scaling and optimal linear step, then the squarings: S with V = e0 S.
// hist (if not null): operand of every squaring.  The loop runs to the warp's
// largest k (the exchanges need every lane); a pair past its own k keeps S.
template <class H>
__device__ __forceinline__ void lp_squarings(float* S, int k, const float* legs, const LanePair& lp, H&& keep) {
    const int kmax = __reduce_max_sync(0xffffffffu, k);
#pragma unroll 1
    for (int t = 0; t < kmax; ++t) {
        float T[NS];
        keep(t, S);
        lp_product<true>(S, nullptr, legs, lp, T);
        const bool on = t < k;
#pragma unroll
        for (int s = 0; s < NS; ++s) S[s] = on ? T[s] : S[s];
    }
}

__device__ __forceinline__ float lp_norm2(const float* f, const LanePair& lp) {
    float n2 = lp.odd ? f[0] * f[0] : 0.f;
#pragma unroll
    for (int s = 1; s < NS; ++s) n2 = fmaf(f[s], f[s], n2);
    return lp_sum(n2);
}

// Three resident blocks per SM (168 registers) for every kernel here: two and
// four measured slower (8-band step of 1M points and 300 spheres: 12.4 ms with
// three, 12.9 with four in the tail adjoint; two cost the forward 12 %).
#ifndef SHS_LP_MINB
#define SHS_LP_MINB 3
#endif

}  // namespace
}  // namespace shs
