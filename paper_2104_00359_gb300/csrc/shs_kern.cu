// Forward and adjoint shading kernels for one band count, compiled once per
// n_bands with -DSHS_NB=n.
//
// Forward (Sec. 3.2-3.3, Eq. 8-13), one thread per shading point:
//   f(x)  = sum_j rotate( ZH of log V'_j , (c_j - x)/|c_j - x| )     pair loop
//   V(x)  = exp*(f)   (DC isolation, 2^-k scaling, optimal linear step,
//                      k squarings with the triple product)
//   H(x)  = rotate( ZH of max(z, 0), n(x) )
//   B_c   = a_c * L_c . (V * H)
// Adjoint: the same steps in reverse, recomputing each sphere's terms instead
// of storing them; scene gradients are reduced warp -> block -> scene scratch.
//
// Per-sphere log-visibility (Sec. 3.3.2, Eq. 13): with s = sin(alpha) =
// min(r / D, 1) and c = cos(alpha), the ZH of -eps * 1[w_z >= c] has
// coefficients -2 pi eps N_l0 int_c^1 P_l(t) dt, and rotating to direction s_hat
// gives F_lm = -2 pi eps (int_c^1 P_l) y_lm(s_hat).  The integral is
//   int_c^1 P_0 = 1 - c,   int_c^1 P_l = (1 - c^2) P_l'(c) / (l (l + 1))  (l >= 1),
// both from Legendre's equation; d/dc int_c^1 P_l = -P_l(c).

#include <type_traits>
#include <cstdint>
#include <cuda_runtime.h>

#include "shs_point.cuh"
#include "shs_exp.cuh"
#include "shs_warp.cuh"

namespace shs {
namespace {

// Up to 5 bands, G_l and P_l in closed form in s2 = sin^2 alpha and
// c = cos alpha, with c^2 = 1 - s2 substituted (fewer operations than the
// recurrences, and s2 = r^2 / D^2 is the accurately known quantity):
//   G_0 = 1 - c, G_1 = s2/2, G_2 = c s2/2, G_3 = s2 (1/2 - 5 s2/8),
//   G_4 = c s2 (1/2 - 7 s2/8);
//   P_1 = c, P_2 = 1 - 3 s2/2, P_3 = c (1 - 5 s2/2), P_4 = 1 - 5 s2 + 35 s2^2/8.
__device__ __forceinline__ void cap_closed(float c, float s2, float* G, float* P) {   // NB <= 5 only
    G[0] = 1.f - c;
    P[0] = 1.f;
    if constexpr (NB > 1) {
        G[1] = 0.5f * s2;
        P[1] = c;
    }
    if constexpr (NB > 2) {
        G[2] = G[1] * c;
        P[2] = fmaf(-1.5f, s2, 1.f);
    }
    if constexpr (NB > 3) {
        G[3] = s2 * fmaf(-0.625f, s2, 0.5f);
        P[3] = c * fmaf(-2.5f, s2, 1.f);
    }
    if constexpr (NB > 4) {
        G[4] = G[2] * fmaf(-1.75f, s2, 1.f);
        P[4] = fmaf(s2, fmaf(4.375f, s2, -5.f), 1.f);
    }
}

// The pair terms are accumulated in the monomial basis: for each band l the
// pair adds G_l(c) x^a y^b z^c (a+b+c = l) at s_hat, and the harmonic
// combination is taken once per point (mono_to_f).
static_assert(NB <= 5, "from 6 bands: shs_hi_forward.cu, shs_hi_backward.cu");
constexpr int NACC = SH::NA;

// One pair's un-normalised log-visibility terms, added to acc.
template <bool CULL = false>
__device__ __forceinline__ void pair_forward(float px, float py, float pz, float4 sp, float* acc, Normal u = {}) {
    const PairGeom g = pair_geometry<CULL>(px, py, pz, sp, u);
    float P[NB], G[NB];
    cap_closed(g.c, g.s2, G, P);
    const float sx = g.dx * g.invD, sy = g.dy * g.invD, sz = g.dz * g.invD;
    SH::accumulate(G, sx, sy, sz, acc);
}

// Two pairs at once in the packed float32x2 instructions of sm_100+, one
// sphere per half of every float2 (same arithmetic as pair_forward).  The
// spheres come interleaved: qa = (x0, x1, y0, y1), qb = (z0, z1, r0, r1).
template <bool CULL = false>
__device__ __forceinline__ void pair_forward2(float2 npx, float2 npy, float2 npz, float4 qa, float4 qb,
                                              float2* acc, Normal u = {}) {
    const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f);
    const float2 dx = __fadd2_rn(make_float2(qa.x, qa.y), npx);
    const float2 dy = __fadd2_rn(make_float2(qa.z, qa.w), npy);
    const float2 dz = __fadd2_rn(make_float2(qb.x, qb.y), npz);
    const float2 D2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
    const float2 invD = make_float2(D2.x > 0.f ? rsqrtf(D2.x) : 0.f, D2.y > 0.f ? rsqrtf(D2.y) : 0.f);
    const float2 r = make_float2(qb.z, qb.w);
    const float2 r2i = __fmul2_rn(__fmul2_rn(r, r), __fmul2_rn(invD, invD));
    float2 s2 = make_float2(fminf(r2i.x, 1.f), fminf(r2i.y, 1.f));
    const float2 om = __ffma2_rn(s2, mone, one);
    float2 c = __fmul2_rn(om, make_float2(rsqrtf(fmaxf(om.x, 1e-30f)), rsqrtf(fmaxf(om.y, 1e-30f))));
    if constexpr (CULL) {   // as in pair_geometry
        const float2 h = __ffma2_rn(dx, make_float2(u.x, u.x),
                                    __ffma2_rn(dy, make_float2(u.y, u.y), __fmul2_rn(dz, make_float2(u.z, u.z))));
        if (h.x < -qb.z) {
            s2.x = 0.f;
            c.x = 1.f;
        }
        if (h.y < -qb.w) {
            s2.y = 0.f;
            c.y = 1.f;
        }
    }
    float2 G[NB];
    G[0] = __ffma2_rn(c, mone, one);
    if constexpr (NB > 1) G[1] = __fmul2_rn(make_float2(0.5f, 0.5f), s2);
    if constexpr (NB > 2) G[2] = __fmul2_rn(G[1], c);
    if constexpr (NB > 3) G[3] = __fmul2_rn(s2, __ffma2_rn(make_float2(-0.625f, -0.625f), s2, make_float2(0.5f, 0.5f)));
    if constexpr (NB > 4) G[4] = __fmul2_rn(G[2], __ffma2_rn(make_float2(-1.75f, -1.75f), s2, one));
    SH::accumulate2(G, __fmul2_rn(dx, invD), __fmul2_rn(dy, invD), __fmul2_rn(dz, invD), acc);
}

// Interleave the staged spheres in place for pair_forward2: entries 2q and
// 2q+1 become (x, x', y, y') and (z, z', r, r'); an odd last sphere stays as
// it is.  The caller synchronises the block before and after.
__device__ __forceinline__ void interleave_sphere_pairs(float4* s_sph, int N) {
    for (int q = threadIdx.x; q < (N >> 1); q += blockDim.x) {
        const float4 a = s_sph[2 * q], b = s_sph[2 * q + 1];
        s_sph[2 * q] = make_float4(a.x, b.x, a.y, b.y);
        s_sph[2 * q + 1] = make_float4(a.z, b.z, a.w, b.w);
    }
}

// Adjoint of two pairs, one sphere with two points (one per half of every
// float2), in the packed float32x2 instructions.  The pair's loss term is
// Psi = sum_l G_l(c) Phi_l(s_hat) with the per-band homogeneous polynomials
// Phi_l(s) = sum_m dfp_lm Hbar_lm(s) (degree l), dfp_i = dLoss/df_i (-2 pi eps)
// NORM_i.  Euler's identity s . grad Phi_l = l Phi_l makes every needed
// quantity a dot product with the per-band gradients:
//   a = sum_l G_l grad Phi_l,    b = sum_l (P_l / l) grad Phi_l   (l >= 1)
//   dPsi/dc = -sum_l P_l Phi_l = -(s_hat . b) - Phi_0
//   dPsi/dd = (a - (s_hat . a) s_hat) / D + 2 (dPsi/dD^2) d
// so only the gradient polynomials (degree l-1) are evaluated per pair.  q:
// the two points' x, y, z, Phi_0 and tensor entries.  The results
// are the gradients with respect to the sphere's centre (the points get the
// negatives) and radius.
template <bool CULL>
__device__ __forceinline__ void pair_backward2(float4 sp, const float2* q, float2* d, const float2* u) {
    const float2 one = make_float2(1.f, 1.f);
    const PairGeom2 g = pair_geometry2<CULL>(q[0], q[1], q[2], sp, u);
    const float2 s2 = g.s2, c = g.c, sx = __fmul2_rn(g.dx, g.invD), sy = __fmul2_rn(g.dy, g.invD),
                 sz = __fmul2_rn(g.dz, g.invD);
    float2 dc = q[3], ax{}, ay{}, az{};   // dc: -dPsi/dc
    if constexpr (NB > 1) {
        float2 gx[NB - 1], gy[NB - 1], gz[NB - 1], G[NB], Pl[NB];   // Pl: P_l / l
        SH::grad_eval2(sx, sy, sz, [&](int o) { return q[4 + o]; }, gx, gy, gz);
        auto k2 = [](float v) { return make_float2(v, v); };
        G[1] = __fmul2_rn(k2(0.5f), s2);
        Pl[1] = c;
        if constexpr (NB > 2) {
            G[2] = __fmul2_rn(G[1], c);
            Pl[2] = __ffma2_rn(k2(-0.75f), s2, k2(0.5f));
        }
        if constexpr (NB > 3) {
            G[3] = __fmul2_rn(s2, __ffma2_rn(k2(-0.625f), s2, k2(0.5f)));
            Pl[3] = __fmul2_rn(c, __ffma2_rn(k2(-2.5f / 3.f), s2, k2(1.f / 3.f)));
        }
        if constexpr (NB > 4) {
            G[4] = __fmul2_rn(G[2], __ffma2_rn(k2(-1.75f), s2, one));
            Pl[4] = __ffma2_rn(s2, __ffma2_rn(k2(4.375f / 4.f), s2, k2(-1.25f)), k2(0.25f));
        }
        ax = __fmul2_rn(G[1], gx[0]);
        ay = __fmul2_rn(G[1], gy[0]);
        az = __fmul2_rn(G[1], gz[0]);
        float2 bx = __fmul2_rn(Pl[1], gx[0]), by = __fmul2_rn(Pl[1], gy[0]), bz = __fmul2_rn(Pl[1], gz[0]);
#pragma unroll
        for (int l = 2; l < NB; ++l) {
            ax = __ffma2_rn(G[l], gx[l - 1], ax);
            ay = __ffma2_rn(G[l], gy[l - 1], ay);
            az = __ffma2_rn(G[l], gz[l - 1], az);
            bx = __ffma2_rn(Pl[l], gx[l - 1], bx);
            by = __ffma2_rn(Pl[l], gy[l - 1], by);
            bz = __ffma2_rn(Pl[l], gz[l - 1], bz);
        }
        dc = __ffma2_rn(sx, bx, __ffma2_rn(sy, by, __ffma2_rn(sz, bz, dc)));
    }
    pair_finish2(g, sp.w, sx, sy, sz, ax, ay, az, dc, d);
}

// A warp's 32 points for the pair adjoint: 16 rows of two points each, per row
// x, y, z, Phi_0 and the NG tensor entries as float2; the row length (in
// float2, 2 mod 4) spreads the lanes' writes over the banks.
constexpr int kRowUsed = 4 + SH::NG;
constexpr int kRow = kRowUsed + (6 - kRowUsed % 4) % 4;
constexpr int kWarpRows = 16;
static_assert(kRow % 4 == 2 && kRow >= kRowUsed, "row length");

__device__ __forceinline__ void load_row(const float4* row, float2* q) {
#pragma unroll
    for (int i = 0; i < (kRowUsed + 1) / 2; ++i) {
        const float4 v = row[i];
        q[2 * i] = make_float2(v.x, v.y);
        q[2 * i + 1] = make_float2(v.z, v.w);
    }
}

__host__ __device__ constexpr int harm_of(int i) {   // 0: 1, 2m-1: cos m phi, 2m: sin m phi
    return (i - band_of(i) * band_of(i) - band_of(i)) == 0
               ? 0
               : ((i - band_of(i) * band_of(i) - band_of(i)) > 0
                      ? 2 * (i - band_of(i) * band_of(i) - band_of(i)) - 1
                      : -2 * (i - band_of(i) * band_of(i) - band_of(i)));
}

// Projected-exponential variant of the SH exponential: V = e0 P_n[exp(f^)],
// e0 = exp(f_0 y_0), f^ = f without its constant term, by the variant's rule
// (2n Gauss-Legendre nodes in cos(theta) x 4n azimuths, separable as above):
// per latitude the azimuthal coefficients of f^, its value and exp at each
// azimuth, accumulated against the harmonics, projected with the weight.
// U = P_n[exp(f^)] is returned too (the adjoint needs it).
__device__ __forceinline__ void proj_exp(const float* __restrict__ f, float* __restrict__ V,
                                            float* __restrict__ U) {
    constexpr int EZ = SH::EZ, EP = SH::EP, QF = 2 * NB - 1;
    const float* leg = SH::eleg();
    const float* trig = SH::etrig();
    const float* qw = SH::ew();
    float F[K], O[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        F[i] = f[i];
        O[i] = 0.f;
    }
#pragma unroll 1
    for (int za = 0; za < EZ; ++za) {
        float c[QF], d[QF];
#pragma unroll
        for (int q = 0; q < QF; ++q) {
            c[q] = 0.f;
            d[q] = 0.f;
        }
#pragma unroll
        for (int i = 1; i < K; ++i) c[harm_of(i)] = fmaf(F[i], leg[za * K + i], c[harm_of(i)]);
#pragma unroll 1
        for (int pb = 0; pb < EP; ++pb) {
            const float* T = trig + pb * QF;
            float v = 0.f;
#pragma unroll
            for (int q = 0; q < QF; ++q) v = fmaf(c[q], T[q], v);
            const float E = expf(v);
#pragma unroll
            for (int q = 0; q < QF; ++q) d[q] = fmaf(E, T[q], d[q]);
        }
        const float w = qw[za];
#pragma unroll
        for (int i = 0; i < K; ++i) O[i] = fmaf(w * leg[za * K + i], d[harm_of(i)], O[i]);
    }
    const float e0 = expf(F[0] * kInvSqrt4Pi);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        U[i] = O[i];
        V[i] = e0 * O[i];
    }
}

// Adjoint of proj_exp: df from dV.  df_0 = y_0 e0 (dV . U); for j >= 1,
// df_j = e0 sum_q w_q exp(f^_q) (sum_i dV_i y_i(q)) y_j(q).
__device__ __forceinline__ void proj_exp_adjoint(const float* __restrict__ f, const float* __restrict__ U,
                                                    const float* __restrict__ dV, float* __restrict__ df) {
    constexpr int EZ = SH::EZ, EP = SH::EP, QF = 2 * NB - 1;
    const float* leg = SH::eleg();
    const float* trig = SH::etrig();
    const float* qw = SH::ew();
    float F[K], G[K], O[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        F[i] = f[i];
        G[i] = dV[i];
        O[i] = 0.f;
    }
#pragma unroll 1
    for (int za = 0; za < EZ; ++za) {
        float c[QF], g[QF], d[QF];
#pragma unroll
        for (int q = 0; q < QF; ++q) {
            c[q] = 0.f;
            g[q] = 0.f;
            d[q] = 0.f;
        }
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const float L = leg[za * K + i];
            if (i > 0) c[harm_of(i)] = fmaf(F[i], L, c[harm_of(i)]);
            g[harm_of(i)] = fmaf(G[i], L, g[harm_of(i)]);
        }
#pragma unroll 1
        for (int pb = 0; pb < EP; ++pb) {
            const float* T = trig + pb * QF;
            float v = 0.f, dv = 0.f;
#pragma unroll
            for (int q = 0; q < QF; ++q) {
                v = fmaf(c[q], T[q], v);
                dv = fmaf(g[q], T[q], dv);
            }
            const float p = expf(v) * dv;
#pragma unroll
            for (int q = 0; q < QF; ++q) d[q] = fmaf(p, T[q], d[q]);
        }
        const float w = qw[za];
#pragma unroll
        for (int i = 1; i < K; ++i) O[i] = fmaf(w * leg[za * K + i], d[harm_of(i)], O[i]);
    }
    const float e0 = expf(F[0] * kInvSqrt4Pi);
    float de0 = 0.f;
#pragma unroll
    for (int i = 0; i < K; ++i) de0 = fmaf(G[i], U[i], de0);
    df[0] = de0 * e0 * kInvSqrt4Pi;
#pragma unroll
    for (int i = 1; i < K; ++i) df[i] = e0 * O[i];
}

// Clamped-cosine SH for a (not necessarily unit) normal; also returns the unit
// normal and 1/|n| for the adjoint.
__device__ __forceinline__ void cosine_lobe(float nx, float ny, float nz, float* H, float& ux,
                                            float& uy, float& uz, float& inv_len) {
    const float n2 = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
    inv_len = n2 > 0.f ? rsqrtf(n2) : 0.f;
    ux = nx * inv_len;
    uy = ny * inv_len;
    uz = nz * inv_len;
    float Y[K];
    SH::ybar(ux, uy, uz, Y);
#pragma unroll
    for (int i = 0; i < K; ++i) H[i] = SH::ahat(band_of(i)) * SH::norm(i) * Y[i];
}

// Scale the raw pair sums to the log-visibility f.
__device__ __forceinline__ void finish_f(const SceneView& sc, const float* acc, float* f) {
    float fr[K];
    SH::mono_to_f(acc, fr);
#pragma unroll
    for (int i = 0; i < K; ++i) f[i] = sc.neg_2pi_eps * SH::norm(i) * fr[i];
}

// ---------------------------------------------------------------------------
// forward kernel
// ---------------------------------------------------------------------------

// Forward shading of point p of one request (Eq. 8), scene staged in shared
// memory.  MODE kFwdFull: pair terms, exponential and shading; kFwdTail: f
// read from the saved state, then the exponential and shading (lighting or
// albedo changed, geometry not).
template <int MODE = kFwdFull>
__device__ __forceinline__ void forward_point(const FwdArgs& a, const float4* s_sph, const float* s_light,
                                              int64_t p) {
    float f[K];
    if constexpr (MODE == kFwdTail) {
#pragma unroll
        for (int i = 0; i < K; ++i) f[i] = __ldg(a.saved_f + i * a.n_points + p);
    } else {
    const float px = __ldg(a.points + 3 * p), py = __ldg(a.points + 3 * p + 1),
                pz = __ldg(a.points + 3 * p + 2);

    float acc[NACC];
    const int N = a.sc.n_spheres;
    // spheres interleaved in pairs (interleave_sphere_pairs)
    float2 acc2[NACC];
#pragma unroll
    for (int i = 0; i < NACC; ++i) acc2[i] = make_float2(0.f, 0.f);
    const float2 npx = make_float2(-px, -px), npy = make_float2(-py, -py), npz = make_float2(-pz, -pz);
    if (a.sc.horizon_cull) {
        const Normal u = unit_normal(__ldg(a.normals + 3 * p), __ldg(a.normals + 3 * p + 1),
                                     __ldg(a.normals + 3 * p + 2));
#pragma unroll 1
        for (int q = 0; q < (N >> 1); ++q)
            pair_forward2<true>(npx, npy, npz, s_sph[2 * q], s_sph[2 * q + 1], acc2, u);
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = acc2[i].x + acc2[i].y;
        if (N & 1) pair_forward<true>(px, py, pz, s_sph[N - 1], acc, u);
    } else {
#pragma unroll 1
        for (int q = 0; q < (N >> 1); ++q) pair_forward2(npx, npy, npz, s_sph[2 * q], s_sph[2 * q + 1], acc2);
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = acc2[i].x + acc2[i].y;
        if (N & 1) pair_forward(px, py, pz, s_sph[N - 1], acc);
    }

    finish_f(a.sc, acc, f);
    }
    float V[K];
    int k = 0;
    if (a.sc.exp_mode == 1) {
        float U[K];
        proj_exp(f, V, U);
    } else {
        float nrm2 = 0.f;
#pragma unroll
        for (int i = 1; i < K; ++i) nrm2 = fmaf(f[i], f[i], nrm2);
        k = scaling_k(a.sc, nrm2);
        const float scale = ldexpf(1.f, -k);
        const OLCoef ol = ol_coef(a.sc, nrm2 * scale * scale);
        float S[K];
        S[0] = ol.a * kSqrt4Pi;
#pragma unroll
        for (int i = 1; i < K; ++i) S[i] = ol.b * (f[i] * scale);
        for (int t = 0; t < k; ++t) {
            float T[K];
            SH::sqr(S, T);
#pragma unroll
            for (int i = 0; i < K; ++i) S[i] = T[i];
        }
        const float e0 = expf(f[0] * kInvSqrt4Pi);
#pragma unroll
        for (int i = 0; i < K; ++i) V[i] = e0 * S[i];
    }

    float H[K], ux, uy, uz, il;
    cosine_lobe(__ldg(a.normals + 3 * p), __ldg(a.normals + 3 * p + 1), __ldg(a.normals + 3 * p + 2),
                H, ux, uy, uz, il);
    float W[K];
    SH::mul_lobe(V, H, W);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < K; ++i) d = fmaf(s_light[c * KPAD + i], W[i], d);
        a.radiance[3 * p + c] = __ldg(a.albedo + 3 * p + c) * d;
    }
    if (MODE == kFwdFull && a.saved_f) {
#pragma unroll
        for (int i = 0; i < K; ++i) a.saved_f[i * a.n_points + p] = f[i];
        a.saved_k[p] = k;
    }
}

#ifndef SHS_FWD_MINB
#define SHS_FWD_MINB 4
#endif
#ifndef SHS_BWD_MINB
#define SHS_BWD_MINB 3
#endif
template <int MODE>
__global__ void __launch_bounds__(kBlock, NB <= 4 ? SHS_FWD_MINB : 1) forward_kernel_t(FwdArgs a) {
    __shared__ __align__(16) float4 s_sph[kMaxSpheres];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(8) uint64_t s_bar;
    if (!stage_scene(a.sc, s_sph, s_light, &s_bar)) return;
    interleave_sphere_pairs(s_sph, a.sc.n_spheres);
    __syncthreads();
    const int64_t p = static_cast<int64_t>(blockIdx.x) * kBlock + threadIdx.x;
    if (p >= a.n_points) return;
    forward_point<MODE>(a, s_sph, s_light, p);
}


// ---------------------------------------------------------------------------
// backward kernel
// ---------------------------------------------------------------------------

// The point gradients of lane pairs that each hold a row: sums over the pair's
// spheres, written by the row's point h on lane 2 r + h.
__device__ __forceinline__ void store_row_points(const BwdArgs& a, float2* gp, int64_t p0, int lane) {
    const int64_t p = p0 + lane;
#pragma unroll
    for (int e = 0; e < 3; ++e) {
        gp[e].x += __shfl_xor_sync(0xffffffffu, gp[e].x, 1);
        gp[e].y += __shfl_xor_sync(0xffffffffu, gp[e].y, 1);
        if (p < a.n_points) a.d_points[3 * p + e] = -((lane & 1) ? gp[e].y : gp[e].x);
    }
}

// Pair adjoints of the warp's 32 points from 31 spheres on.  A pair of lanes
// holds a row's coefficients in registers and takes every second sphere; the
// rows walk the spheres at different offsets, so the 32 lanes update 32
// distinct slots of the warp's sphere sums with plain shared-memory
// read-modify-writes, and the point gradients stay in registers.  (Spheres on
// the lanes and the rows' coefficients read as broadcasts measured the same
// without point gradients and 35 % slower with them: those need a sum over the
// lanes per row, and the last step idles lanes.)
template <bool CULL>
__device__ __forceinline__ void warp_pairs(const BwdArgs& a, const float4* s_sph, const float4* rows,
                                           const float2 (*nrm)[3], float4* acc_row, int64_t p0, int lane) {
    const int N = a.sc.n_spheres, M = (N + 1) >> 1, r = lane >> 1, h = lane & 1;
    float2 q[kRowUsed + 1], u[3] = {}, gp[3] = {};
    load_row(rows + r * (kRow / 2), q);
    if constexpr (CULL) {
#pragma unroll
        for (int e = 0; e < 3; ++e) u[e] = nrm[r][e];
    }
    int m = r;   // M >= 16 rows
#pragma unroll 1
    for (int t = 0; t < M; ++t) {
        const int j = 2 * m + h;
        const bool has = j < N;
        const float4 sp = has ? s_sph[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        float2 d[4];
        pair_backward2<CULL>(sp, q, d, u);
        if (has) {
#pragma unroll
            for (int e = 0; e < 3; ++e) gp[e] = __fadd2_rn(gp[e], d[e]);
            float4 v = acc_row[j];
            v.x += d[0].x + d[0].y;
            v.y += d[1].x + d[1].y;
            v.z += d[2].x + d[2].y;
            v.w += d[3].x + d[3].y;
            acc_row[j] = v;
        }
        __syncwarp();
        m = m + 1 == M ? 0 : m + 1;
    }
    if (a.d_points) store_row_points(a, gp, p0, lane);
}

// Fewer spheres: rows on the lane pairs as above, every row at the same two
// spheres, whose sums over the rows take five shuffles.  (Spheres on the lanes,
// below, need 24 or 30 shuffles a row for the points, and as many steps for 17
// spheres as for 32: 262k points, 4 bands, 20 spheres, adjoint with point
// gradients 118 against 71 us, without 80 against 70 us.)
template <bool CULL>
__device__ __forceinline__ void warp_pairs_rows(const BwdArgs& a, const float4* s_sph, const float4* rows,
                                                const float2 (*nrm)[3], float4* acc_row, int64_t p0, int lane) {
    const int N = a.sc.n_spheres, r = lane >> 1, h = lane & 1;
    float2 q[kRowUsed + 1], u[3] = {}, gp[3] = {};
    load_row(rows + r * (kRow / 2), q);
    if constexpr (CULL) {
#pragma unroll
        for (int e = 0; e < 3; ++e) u[e] = nrm[r][e];
    }
    float* acc = reinterpret_cast<float*>(acc_row);
#pragma unroll 1
    for (int j = h; j - h < N; j += 2) {
        const bool has = j < N;
        const float4 sp = has ? s_sph[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        float2 d[4];
        pair_backward2<CULL>(sp, q, d, u);
        if (!has) d[0] = d[1] = d[2] = d[3] = make_float2(0.f, 0.f);
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = d[e].x + d[e].y;
#pragma unroll
        for (int e = 0; e < 3; ++e) gp[e] = __fadd2_rn(gp[e], d[e]);
        // halving exchanges: lane bits 4 and 3 end up with component 0 .. 3
        const bool up = lane & 16, up2 = lane & 8;
        const float s0 = up ? v[0] : v[2], s1 = up ? v[1] : v[3];
        v[0] = (up ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, s0, 16);
        v[1] = (up ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, s1, 16);
        const float s2 = up2 ? v[0] : v[1];
        v[0] = (up2 ? v[1] : v[0]) + __shfl_xor_sync(0xffffffffu, s2, 8);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 4);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        if (has && (lane & 6) == 0) acc[4 * j + (lane >> 3)] += v[0];
    }
    __syncwarp();
    if (a.d_points) store_row_points(a, gp, p0, lane);
}

// ... or, without point gradients and with the lanes at least 7/8 full: the lanes
// hold `width` spheres (32, 16 or 8, then one, two or four rows at once), whose
// sums stay in registers over the rows (3 bands, 16 spheres, 37 against 40 us).
__device__ __forceinline__ int few_width(int N) { return N > 16 ? 32 : N > 8 ? 16 : 8; }

template <bool CULL>
__device__ __forceinline__ void warp_pairs_few(const BwdArgs& a, const float4* s_sph, const float4* rows,
                                               const float2 (*nrm)[3], float4* acc_row, int lane) {
    const int N = a.sc.n_spheres, width = few_width(N), sub = lane / width, stride = 32 / width;
    const int j = lane % width;
    const bool has = j < N;
    const float4 sp = has ? s_sph[j] : make_float4(0.f, 0.f, 0.f, 0.f);
    float2 acc[4] = {};
#pragma unroll 1
    for (int t = 0; t < kWarpRows; t += stride) {
        const int r = t + sub;
        float2 q[kRowUsed + 1], d[4];
        load_row(rows + r * (kRow / 2), q);
        pair_backward2<CULL>(sp, q, d, nrm[CULL ? r : 0]);
        if (!has) d[0] = d[1] = d[2] = d[3] = make_float2(0.f, 0.f);
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[e] = __fadd2_rn(acc[e], d[e]);
    }
    float s[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        s[e] = acc[e].x + acc[e].y;
        for (int o = width; o < 32; o <<= 1) s[e] += __shfl_xor_sync(0xffffffffu, s[e], o);
    }
    if (has && sub == 0) {
        float4 v = acc_row[j];
        v.x += s[0];
        v.y += s[1];
        v.z += s[2];
        v.w += s[3];
        acc_row[j] = v;
    }
    __syncwarp();
}

// From 4 bands a block's warps start each tile, and go on from the squarings
// (whose number differs by point), together: the unrolled code is larger than
// the instruction cache, and warps that drift apart fetch it again and again
// (1M points, 12 spheres, adjoint: 5 bands 2,113 -> 625 us, 4 bands 242 -> 222).
__device__ __forceinline__ void keep_together() {
    if constexpr (NB >= 4) __syncthreads();
}

// Adjoint of one 128-point tile of one request: per-point outputs are written,
// the scene-level sums are added to the block's shared accumulators
// (s_dl: d_light and loss per warp, s_acc: per warp and sphere).
// CULLM: horizon culling off (0), on (1), or read from the scene per call (2);
// EXPM: the exponential's form: the Gaussian optimal linear step (0), the
// projected exponential (1), the tabulated optimal linear step (3), or the
// scene's exp_mode read per call (2).
template <int CULLM = 2, int EXPM = 2>
__device__ __forceinline__ void backward_tile(const BwdArgs& a, const float4* s_sph, const float* s_light,
                                              float* s_acc, float (*s_dl)[3 * K + 1], float4* s_rows,
                                              float2 (*s_nrm)[3], int64_t tile, int lane, int warp) {
    const int N = a.sc.n_spheres;
    const int64_t P = a.n_points;
    const int64_t p = tile * kBlock + threadIdx.x;
    const bool live = p < P;
    const int64_t q = live ? p : 0;
    const float px = load_or(a.points, 3 * q, live), py = load_or(a.points, 3 * q + 1, live),
                pz = load_or(a.points, 3 * q + 2, live);

    // ---- log-visibility f: saved by the forward pass or recomputed
    float f[K];
    int k;
    if (a.saved_f) {
#pragma unroll
        for (int i = 0; i < K; ++i) f[i] = load_or(a.saved_f, i * P + q, live);
        k = live ? min(max(a.saved_k[q], 0), kMaxK) : 0;   // a foreign buffer cannot overrun hist
    } else {
        float acc[NACC];
#pragma unroll
        for (int i = 0; i < NACC; ++i) acc[i] = 0.f;
        if (CULLM == 1 || (CULLM == 2 && a.sc.horizon_cull)) {
            const Normal u = unit_normal(load_or(a.normals, 3 * q, live), load_or(a.normals, 3 * q + 1, live),
                                         load_or(a.normals, 3 * q + 2, live));
#pragma unroll 2
            for (int j = 0; j < N; ++j) pair_forward<true>(px, py, pz, s_sph[j], acc, u);
        } else {
#pragma unroll 2
            for (int j = 0; j < N; ++j) pair_forward(px, py, pz, s_sph[j], acc);
        }
        finish_f(a.sc, acc, f);
        k = -1;
    }
    float nrm2 = 0.f;
#pragma unroll
    for (int i = 1; i < K; ++i) nrm2 = fmaf(f[i], f[i], nrm2);
    if (k < 0) k = scaling_k(a.sc, nrm2);

    // ---- recompute the exponential, keeping the operand of every squaring
    // (or, for the projected-exponential variant, U = P_n[exp(f^)])
    const bool projexp = EXPM == 2 ? a.sc.exp_mode == 1 : EXPM == 1;
    float scale = 1.f, e0 = 1.f;
    OLCoef ol{1.f, 1.f, 0.f, 0.f};
    float g[K], S[K], V[K], U[K];
    float hist[kMaxK][K];
    if (projexp) {
        proj_exp(f, V, U);
    } else {
        scale = ldexpf(1.f, -k);
        ol = ol_coef<EXPM == 0 ? 0 : EXPM == 3 ? 1 : 2>(a.sc, nrm2 * scale * scale);
        g[0] = 0.f;
#pragma unroll
        for (int i = 1; i < K; ++i) g[i] = f[i] * scale;
        S[0] = ol.a * kSqrt4Pi;
#pragma unroll
        for (int i = 1; i < K; ++i) S[i] = ol.b * g[i];
        for (int t = 0; t < k; ++t) {
            float T[K];
            SH::sqr(S, T);
#pragma unroll
            for (int i = 0; i < K; ++i) {
                hist[t][i] = S[i];
                S[i] = T[i];
            }
        }
        e0 = expf(f[0] * kInvSqrt4Pi);
#pragma unroll
        for (int i = 0; i < K; ++i) V[i] = e0 * S[i];
    }
    keep_together();
    float H[K], ux, uy, uz, il;
    cosine_lobe(load_or(a.normals, 3 * q, live), load_or(a.normals, 3 * q + 1, live),
                load_or(a.normals, 3 * q + 2, live), H, ux, uy, uz, il);
    float W[K];
    SH::mul_lobe(V, H, W);

    // ---- shading adjoint: B_c = a_c L_c . W
    float dB[3], alb[3], loss = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        alb[c] = load_or(a.albedo, 3 * q + c, live);
        if (a.target) {
            const float r = load_or(a.radiance, 3 * q + c, live) - load_or(a.target, 3 * q + c, live);
            dB[c] = r;
            loss = fmaf(0.5f * r, r, loss);
        } else {
            dB[c] = load_or(a.d_radiance, 3 * q + c, live);
        }
    }
    float dW[K];
#pragma unroll
    for (int i = 0; i < K; ++i) dW[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float u = alb[c] * dB[c];
        float lw = 0.f;
#pragma unroll
        for (int i = 0; i < K; ++i) {
            const float L = s_light[c * KPAD + i];
            lw = fmaf(L, W[i], lw);
            dW[i] = fmaf(u, L, dW[i]);
        }
        if (live && a.d_albedo) a.d_albedo[3 * q + c] = dB[c] * lw;
    }
    if (a.d_light) {
        float dl[3 * K];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float u = alb[c] * dB[c];
#pragma unroll
            for (int i = 0; i < K; ++i) dl[c * K + i] = u * W[i];
        }
        warp_sum_into<3 * K>(dl, &s_dl[warp][0], lane);
    }
    if (a.target) {
        const float v = warp_sum(loss);
        if (lane == 0) s_dl[warp][3 * K] += v;
    }
    float dV[K], dH[K];
    SH::mul_lobe(dW, H, dV);                // C is symmetric: adjoint of a*b is d*b
    SH::mul_onto_lobe(dW, V, dH);           // the normal adjoint scales the other bands by zero

    // ---- normal adjoint through H = A_hat_l NORM_i Ybar_i(n / |n|)
    if (live && a.d_normals) {
        float wn[K];
#pragma unroll
        for (int i = 0; i < K; ++i) wn[i] = dH[i] * SH::ahat(band_of(i)) * SH::norm(i);
        float gx, gy, gz;
        SH::ybar_vjp(ux, uy, uz, wn, gx, gy, gz);
        const float ug = ux * gx + uy * gy + uz * gz;
        a.d_normals[3 * q] = (gx - ux * ug) * il;
        a.d_normals[3 * q + 1] = (gy - uy * ug) * il;
        a.d_normals[3 * q + 2] = (gz - uz * ug) * il;
    }

    // ---- exponential adjoint
    float dfp[K];
    if (projexp) {
        proj_exp_adjoint(f, U, dV, dfp);
    } else {
        float de0 = 0.f, dS[K];
#pragma unroll
        for (int i = 0; i < K; ++i) {
            de0 = fmaf(dV[i], S[i], de0);
            dS[i] = e0 * dV[i];
        }
        for (int t = k - 1; t >= 0; --t) {
            float Ht[K], T[K];
#pragma unroll
            for (int i = 0; i < K; ++i) Ht[i] = hist[t][i];
            SH::mul(dS, Ht, T);
#pragma unroll
            for (int i = 0; i < K; ++i) dS[i] = 2.f * T[i];
        }
        // S_0 = a(s) sqrt(4 pi), S_i = b(s) g_i: dg_i = b dS_i + (dA a'/s + dB b'/s) g_i
        const float dA = dS[0] * kSqrt4Pi;
        float dB = 0.f;
#pragma unroll
        for (int i = 1; i < K; ++i) dB = fmaf(dS[i], g[i], dB);
        const float cg = fmaf(dA, ol.ca, dB * ol.cb);
        dfp[0] = de0 * e0 * kInvSqrt4Pi;
#pragma unroll
        for (int i = 1; i < K; ++i) dfp[i] = fmaf(ol.b, dS[i], cg * g[i]) * scale;
    }
#pragma unroll
    for (int i = 0; i < K; ++i) dfp[i] *= a.sc.neg_2pi_eps * SH::norm(i);

    // ---- pair adjoints: the warp's points go through shared memory, two per
    // row; the warp reads only its own rows
    if (!(a.d_centers || a.d_radii || a.d_points) || N == 0) {
        if (live && a.d_points)
            for (int c = 0; c < 3; ++c) a.d_points[3 * q + c] = 0.f;
        return;
    }
    __syncwarp();   // the previous tile's rows have been read
    float* row = reinterpret_cast<float*>(s_rows + warp * (kWarpRows * kRow / 2)) + (lane >> 1) * (2 * kRow) + (lane & 1);
    row[0] = px;
    row[2] = py;
    row[4] = pz;
    row[6] = dfp[0];
    {
        float gq[SH::NG > 0 ? SH::NG : 1];
        SH::grad_coeffs(dfp, gq);
#pragma unroll
        for (int o = 0; o < SH::NG; ++o) row[8 + 2 * o] = gq[o];
    }
    float* nr = reinterpret_cast<float*>(&s_nrm[warp * kWarpRows + (lane >> 1)][0]) + (lane & 1);
    nr[0] = ux;
    nr[2] = uy;
    nr[4] = uz;
    __syncwarp();
    const float4* rows = s_rows + warp * (kWarpRows * kRow / 2);
    const float2(*nrm)[3] = s_nrm + warp * kWarpRows;
    float4* acc_row = reinterpret_cast<float4*>(s_acc) + warp * N;
    auto loops = [&](auto cull_tag) {
        constexpr bool CULL = decltype(cull_tag)::value;
        const int64_t p0 = tile * kBlock + warp * 32;
        if (N >= 2 * kWarpRows - 1) warp_pairs<CULL>(a, s_sph, rows, nrm, acc_row, p0, lane);
        else if (a.d_points || 8 * N < 7 * few_width(N)) warp_pairs_rows<CULL>(a, s_sph, rows, nrm, acc_row, p0, lane);
        else warp_pairs_few<CULL>(a, s_sph, rows, nrm, acc_row, lane);
    };
    if constexpr (CULLM == 2) {
        if (a.sc.horizon_cull) loops(std::true_type{});
        else loops(std::false_type{});
    } else {
        loops(std::integral_constant<bool, CULLM == 1>{});
    }
}

// Layout of one block's reduced scene gradient (E floats):
//   [0, 3K)          d_light, channel-major
//   [3K]             loss
//   [3K+1, 3K+1+4N)  per sphere (d cx, d cy, d cz, d r)
// Up to 4 bands: three resident blocks per SM (167 or 168 registers per thread)
// for the pair loop; above that the tail state needs the registers.
template <int CULLM, int EXPM>
__global__ void __launch_bounds__(kBlock, NB <= 4 ? SHS_BWD_MINB : 1) backward_kernel_t(BwdArgs a) {
    extern __shared__ __align__(16) float4 dyn[];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ float s_dl[NWARP][3 * K + 1];
    __shared__ __align__(16) float4 s_rows[NWARP * kWarpRows * kRow / 2];
    __shared__ __align__(8) float2 s_nrm[NWARP * kWarpRows][3];
    __shared__ bool s_last;
    const int N = a.sc.n_spheres;
    float4* s_sph = dyn;                  // [N]
    float* s_acc = reinterpret_cast<float*>(dyn + N);   // [NWARP][4N]
    if (!stage_scene(a.sc, s_sph, s_light, &s_bar)) return;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < NWARP * 4 * N; e += kBlock) s_acc[e] = 0.f;
    for (int e = threadIdx.x; e < NWARP * (3 * K + 1); e += kBlock) (&s_dl[0][0])[e] = 0.f;
    __syncthreads();

    const int64_t ntiles = (a.n_points + kBlock - 1) / kBlock;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        keep_together();
        backward_tile<CULLM, EXPM>(a, s_sph, s_light, s_acc, s_dl, s_rows, s_nrm, tile, lane, warp);
    }

    // ---- block reduction, then one scene-level reduction
    __syncthreads();
    const int E = 3 * K + 1 + 4 * N;
    float* out = a.partials + static_cast<size_t>(blockIdx.x) * a.partial_stride;
    const bool det = a.counter == nullptr;
    for (int e = threadIdx.x; e < E; e += kBlock) {
        float v = 0.f;
        if (e <= 3 * K) {
#pragma unroll
            for (int w = 0; w < NWARP; ++w) v += s_dl[w][e];
        } else {
            const int s = e - (3 * K + 1);
#pragma unroll
            for (int w = 0; w < NWARP; ++w) v += s_acc[w * 4 * N + s];
        }
        if (det) out[e] = v;
        else atomicAdd(a.partials + e, v);
    }
    if (det) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    finish_scene_sums(a, E);
}

// ---------------------------------------------------------------------------
// batched persistent kernels (serving): many requests, one launch
// ---------------------------------------------------------------------------

// Forward for every tile of every request in the batch.  Blocks take tiles
// from a device counter (consecutive tiles mostly share a request, so a
// request's scene is staged once per run of its tiles).
__global__ void __launch_bounds__(kBlock) forward_batch_kernel(const __grid_constant__ FwdBatch b) {
    __shared__ __align__(16) float4 s_sph[kMaxSpheres];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ long long s_tile;
    mbar_init(&s_bar);
    int staged = -1;
    uint32_t parity = 0;
    for (;;) {
        __syncthreads();                 // previous tile done before restaging
        if (threadIdx.x == 0) s_tile = static_cast<long long>(atomicAdd(b.queue, 1u));
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= b.total_tiles) break;
        const int r = find_request(b.tile_begin, b.n, tile);
        if (r != staged) {
            if (!stage_copy(b.r[r].sc, s_sph, s_light, &s_bar, parity)) return;
            parity ^= 1u;
            staged = r;
            interleave_sphere_pairs(s_sph, b.r[r].sc.n_spheres);
            __syncthreads();
        }
        const int64_t p = (tile - b.tile_begin[r]) * kBlock + threadIdx.x;
        if (p < b.r[r].n_points) forward_point(b.r[r], s_sph, s_light, p);
    }
}

// L2 adjoint for every tile of every request in the batch.  Each tile's scene
// sums go to its request's accumulator with atomics; the tile that completes a
// request writes that request's outputs.
__global__ void __launch_bounds__(kBlock, NB <= 4 ? 4 : 1)
    backward_batch_kernel(const __grid_constant__ BwdBatch b) {
    extern __shared__ __align__(16) float4 dyn[];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ float s_dl[NWARP][3 * K + 1];
    __shared__ __align__(16) float4 s_rows[NWARP * kWarpRows * kRow / 2];
    __shared__ __align__(8) float2 s_nrm[NWARP * kWarpRows][3];
    __shared__ bool s_last;
    __shared__ long long s_tile;
    float4* s_sph = dyn;                                        // [max N]
    float* s_acc = reinterpret_cast<float*>(dyn + b.max_spheres);   // [NWARP][4 max N]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    mbar_init(&s_bar);
    int staged = -1;
    uint32_t parity = 0;
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_tile = static_cast<long long>(atomicAdd(b.queue, 1u));
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= b.total_tiles) break;
        const int r = find_request(b.tile_begin, b.n, tile);
        const BwdArgs& a = b.r[r];
        const int N = a.sc.n_spheres;
        if (r != staged) {
            if (!stage_copy(a.sc, s_sph, s_light, &s_bar, parity)) return;
            parity ^= 1u;
            staged = r;
        }
        for (int e = threadIdx.x; e < NWARP * 4 * N; e += kBlock) s_acc[e] = 0.f;
        for (int e = threadIdx.x; e < NWARP * (3 * K + 1); e += kBlock) (&s_dl[0][0])[e] = 0.f;
        __syncthreads();
        backward_tile(a, s_sph, s_light, s_acc, s_dl, s_rows, s_nrm, tile - b.tile_begin[r], lane, warp);
        __syncthreads();
        const int E = 3 * K + 1 + 4 * N;
        for (int e = threadIdx.x; e < E; e += kBlock) {
            float v = 0.f;
            if (e <= 3 * K) {
#pragma unroll
                for (int w = 0; w < NWARP; ++w) v += s_dl[w][e];
            } else {
                const int q = e - (3 * K + 1);
#pragma unroll
                for (int w = 0; w < NWARP; ++w) v += s_acc[w * 4 * N + q];
            }
            add_tile_sum(a, e, v);
        }
        __threadfence();
        __syncthreads();
        const int64_t ntiles_r = b.tile_begin[r + 1] - b.tile_begin[r];
        if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == static_cast<unsigned>(ntiles_r - 1);
        __syncthreads();
        if (s_last) finish_scene_sums(a, E);
    }
}

size_t backward_dyn_smem(int n_spheres) {
    return static_cast<size_t>(n_spheres) * 16u * (1 + NWARP);
}

template <int CULLM, int EXPM>
cudaError_t run_backward(const BwdArgs& a, size_t smem, cudaStream_t s) {
    static DeviceOnce once;
    const cudaError_t e = allow_dyn_smem(backward_kernel_t<CULLM, EXPM>, backward_dyn_smem(kMaxSpheres), once);
    if (e != cudaSuccess) return e;
    backward_kernel_t<CULLM, EXPM><<<static_cast<unsigned>(a.grid), kBlock, smem, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

template <>
BwdBlocks backward_blocks_per_sm<NB>(int n_spheres, bool) {
    cudaFuncSetAttribute(backward_kernel_t<0, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         static_cast<int>(backward_dyn_smem(kMaxSpheres)));
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, backward_kernel_t<0, 0>, kBlock,
                                                      backward_dyn_smem(n_spheres)) != cudaSuccess || nb < 1)
        nb = 1;
    return BwdBlocks{nb, 0, 0};
}

template <>
cudaError_t launch_forward_batch<NB>(const FwdBatch& b, cudaStream_t s) {
    if (b.total_tiles <= 0) return cudaSuccess;
    static WaveCache wave;
    int grid = 0;
    const cudaError_t e = one_wave(forward_batch_kernel, 0, b.total_tiles, wave, &grid);
    if (e != cudaSuccess) return e;
    forward_batch_kernel<<<grid, kBlock, 0, s>>>(b);
    count_launch();
    return cudaGetLastError();
}

template <>
cudaError_t launch_backward_batch<NB>(const BwdBatch& b, cudaStream_t s) {
    if (b.total_tiles <= 0) return cudaSuccess;
    const size_t smem = backward_dyn_smem(b.max_spheres);
    static DeviceOnce once;
    static WaveCache wave;
    int grid = 0;
    cudaError_t e = allow_dyn_smem(backward_batch_kernel, backward_dyn_smem(kMaxSpheres), once);
    if (e == cudaSuccess) e = one_wave(backward_batch_kernel, smem, b.total_tiles, wave, &grid);
    if (e != cudaSuccess) return e;
    backward_batch_kernel<<<grid, kBlock, smem, s>>>(b);
    count_launch();
    return cudaGetLastError();
}

template <>
cudaError_t launch_forward<NB>(const FwdArgs& a, cudaStream_t s) {
    if (a.n_points <= 0) return cudaSuccess;
    const int64_t blocks = (a.n_points + kBlock - 1) / kBlock;
    if (a.tail_only)
        forward_kernel_t<kFwdTail><<<static_cast<unsigned>(blocks), kBlock, 0, s>>>(a);
    else
        forward_kernel_t<kFwdFull><<<static_cast<unsigned>(blocks), kBlock, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <>
cudaError_t launch_backward<NB>(const BwdArgs& a, cudaStream_t s) {
    if (a.n_points <= 0) return cudaSuccess;
    const size_t smem = backward_dyn_smem(a.sc.n_spheres);
    const bool cull = a.sc.horizon_cull != 0;
    cudaError_t err;
    if (a.sc.exp_mode == 1) err = cull ? run_backward<1, 1>(a, smem, s) : run_backward<0, 1>(a, smem, s);
    else if (a.sc.exp_mode == 2) err = cull ? run_backward<1, 3>(a, smem, s) : run_backward<0, 3>(a, smem, s);
    else err = cull ? run_backward<1, 0>(a, smem, s) : run_backward<0, 0>(a, smem, s);
    if (err != cudaSuccess || a.counter != nullptr) return err;
    const int E = 3 * K + 1 + 4 * a.sc.n_spheres;
    reduce_partials_kernel<<<reduce_blocks(E), kReduceThreads, 0, s>>>(a, a.grid, a.grid);
    count_launch();
    return cudaGetLastError();
}

}  // namespace shs
