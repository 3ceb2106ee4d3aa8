// Adjoint shading kernels for 6, 7 and 8 bands, compiled once per n_bands with
// -DSHS_NB=n (shs_hi.cuh).
//
// Adjoint of the pair terms: one sphere per lane.  A warp owns the 16 points
// whose tail adjoint it has just run; their coefficients go through shared
// memory (read back as broadcasts), each lane keeps its sphere's geometry and
// sums over the 16 points in registers, and the warp walks the spheres in
// groups of 32, so every warp of a block has the same share of the work.

#include <cstdint>
#include <cuda_runtime.h>

#include "shs_hi.cuh"
#include "shs_warp.cuh"

namespace shs {
namespace {

// ---------------------------------------------------------------------------
// pair adjoint
// ---------------------------------------------------------------------------

// Two points' adjoint coefficients in shared memory, one row per pair of
// points and one point per half of every float2: x, y, z, then (horizon culling)
// the unit normals, then for column m
// w_lm = dLoss/df_lm (-2 pi eps) NORM_lm (2l - 1)!! / (l (l + 1)) for l = m ..
// NB - 1 (l = 0: without the division), for m > 0 as (cos, sin) pairs; columns
// start at multiples of two entries (16 bytes).
__host__ __device__ constexpr int wcol(int m) {
    int b = 6;
    for (int k = 0; k < m; ++k) b += ((k ? 2 : 1) * (NB - k) + 1) / 2 * 2;
    return b;
}
constexpr int kWarpRows = kWarpPoints / 2;
constexpr int WST = wcol(NB) + 2;   // entries per row
constexpr int kRowFloats = kWarpRows * 2 * WST;
constexpr int kWarpRegion = kRowFloats > 64 * NS ? kRowFloats : 64 * NS;   // floats

// Adjoint of two pairs (one sphere, two points) Psi = sum_l G_l(c)
// Phi_l(s_hat), Phi_l = sum_m w_lm Ybar_lm: the gradients with respect to the
// sphere's centre (the points get the negatives) and radius.  Per order m, with
// R_lm and d/dz R_lm = R_l,m+1:
//   alpha = sum_l P_l' R_lm w_lm           -> d/dx, d/dy of C_m + i S_m
//   beta  = sum_l P_l' R_l,m+1 w_lm        -> d/dz
//   gamma = sum_l l (l + 1) P_l R_lm w_lm  -> -dPsi/dc
// (the factor s2 of G_l is applied at the end).  The products P_l' R_l,m+1 of
// one order are the next order's P_l' R_lm.  At 8 bands about 440 FP32
// operations a pair, where the evaluation and reverse sweep of all 64
// harmonics took about 800.  Packed, because a scalar multiply-add with three
// different registers issues at 70 - 110 of 128 lanes a clock on this chip
// (register ports), a packed one at 120.
__device__ __forceinline__ float2 k2(float v) { return make_float2(v, v); }

template <int M>
__device__ __forceinline__ void sh_column2(const float2* zi, float2* col) {
    if constexpr (M < NB) {
        col[0] = k2(1.f);
        if constexpr (M + 1 < NB) col[1] = zi[0];
#pragma unroll
        for (int i = 1; i + 1 < NB - M; ++i) {
            const int l = M + i;
            col[i + 1] = __ffma2_rn(zi[i], col[i],
                                    __fmul2_rn(k2(-(float(l + M) / float((4 * l * l - 1) * (i + 1)))), col[i - 1]));
        }
    }
}

template <bool CULL>
__device__ __forceinline__ void pair_backward2(float4 sp, const float2* row, float2* d) {
    const PairGeom2 g = pair_geometry2<CULL>(row[0], row[1], row[2], sp, row + 3);
    float2 P[NB], dP[NB];   // P_l (times l (l + 1) below) and P_l'
    P[0] = k2(1.f);
    P[1] = g.c;
    dP[1] = k2(1.f);
#pragma unroll
    for (int l = 1; l + 1 < NB; ++l) {
        P[l + 1] = __ffma2_rn(__fmul2_rn(k2((2.f * l + 1.f) / (l + 1.f)), g.c), P[l],
                              __fmul2_rn(k2(-(float(l) / (l + 1.f))), P[l - 1]));
        dP[l + 1] = l == 1 ? __fmul2_rn(k2(3.f), P[1]) : __ffma2_rn(k2(2.f * l + 1.f), P[l], dP[l - 1]);
    }
#pragma unroll
    for (int l = 1; l < NB; ++l) P[l] = __fmul2_rn(P[l], k2(float(l * (l + 1))));
    const float2 sx = __fmul2_rn(g.dx, g.invD), sy = __fmul2_rn(g.dy, g.invD), sz = __fmul2_rn(g.dz, g.invD);
    const float2 nsy = __fmul2_rn(sy, k2(-1.f));
    float2 zi[NB], col[NB], nxt[NB], e[NB], C = k2(1.f), S = k2(0.f);
    float2 gx = k2(0.f), gy = k2(0.f), gz = k2(0.f), ga = k2(0.f);
#pragma unroll
    for (int i = 0; i + 1 < NB; ++i) zi[i] = __fmul2_rn(sz, k2(1.f / float(i + 1)));
    sh_column2<0>(zi, col);
    static_for<NB>([&](auto mm) {
        constexpr int m = mm, n = (m ? 2 : 1) * (NB - m);
        float2 wm[(n + 1) / 2 * 2];
        const float4* w4 = reinterpret_cast<const float4*>(row + wcol(m));
#pragma unroll
        for (int i = 0; i < (n + 1) / 2; ++i) {
            const float4 v = w4[i];
            wm[2 * i] = make_float2(v.x, v.y);
            wm[2 * i + 1] = make_float2(v.z, v.w);
        }
        sh_column2<m + 1>(zi, nxt);
        float2 ac{}, as{}, bc{}, bs{}, cc{}, cs{};
#pragma unroll
        for (int i = 0; i < NB - m; ++i) {   // l = m + i
            const float2 h = i ? __fmul2_rn(P[m + i], col[i]) : P[m];
            const float2 wc = wm[m ? 2 * i : i], ws = wm[m ? 2 * i + 1 : 0];
            cc = i ? __ffma2_rn(h, wc, cc) : __fmul2_rn(h, wc);
            if (m) {
                ac = i ? __ffma2_rn(e[i], wc, ac) : __fmul2_rn(e[i], wc);
                as = i ? __ffma2_rn(e[i], ws, as) : __fmul2_rn(e[i], ws);
                cs = i ? __ffma2_rn(h, ws, cs) : __fmul2_rn(h, ws);
            }
            if (i) {
                e[i - 1] = i == 1 ? dP[m + i] : __fmul2_rn(dP[m + i], nxt[i - 1]);
                bc = i > 1 ? __ffma2_rn(e[i - 1], wc, bc) : __fmul2_rn(e[i - 1], wc);
                if (m) bs = i > 1 ? __ffma2_rn(e[i - 1], ws, bs) : __fmul2_rn(e[i - 1], ws);
            }
        }
        if constexpr (m == 0) {
            gz = bc;
            ga = cc;
        } else {
            // C, S still hold order m - 1
            if constexpr (m == 1) {
                gx = ac;
                gy = as;
                C = sx;
                S = sy;
            } else {
                const float2 fc = __fmul2_rn(k2(float(m)), C), fs = __fmul2_rn(k2(float(m)), S);
                gx = __ffma2_rn(ac, fc, __ffma2_rn(as, fs, gx));
                gy = __ffma2_rn(as, fc, __ffma2_rn(__fmul2_rn(ac, k2(-1.f)), fs, gy));
                const float2 c1 = __ffma2_rn(sx, C, __fmul2_rn(nsy, S)), s1 = __ffma2_rn(sx, S, __fmul2_rn(sy, C));
                C = c1;
                S = s1;
            }
            if constexpr (m + 1 < NB) gz = __ffma2_rn(bc, C, __ffma2_rn(bs, S, gz));
            ga = __ffma2_rn(cc, C, __ffma2_rn(cs, S, ga));
        }
#pragma unroll
        for (int i = 0; i + 1 < NB - m; ++i) col[i] = nxt[i];
    });
    pair_finish2(g, sp.w, sx, sy, sz, __fmul2_rn(gx, g.s2), __fmul2_rn(gy, g.s2), __fmul2_rn(gz, g.s2), ga, d);
}

// ---------------------------------------------------------------------------
// adjoint
// ---------------------------------------------------------------------------

constexpr int kDl = (3 * NS + 15) / 16 * 16;   // a lane parity's lighting sums, 16 at a time

struct BwdShared {
    float4* sph;                 // [N]
    float4* acc;                 // [NWARP][N] (d cx, d cy, d cz, d r)
    const float (*lt)[3][NSP];
    const float* leg;
    float (*dl)[2][kDl];         // [NWARP]
    float* loss;                 // [NWARP]
    float* w;                    // per warp: the operands of its products, then its points' rows
    int region;                  // floats of w per warp
};

// Adjoint of the exponential and the shading at the lane pair's point: the
// per-point outputs, the lighting and loss sums, and dLoss/df_i (-2 pi eps)
// NORM_i of the lane's slots in dfp.
template <int EXPM, bool CULL>
__device__ __forceinline__ void lp_tail_adjoint(const BwdArgs& a, const BwdShared& sh, int64_t p, float* dfp) {
    const LanePair lp = lane_pair();
    const bool projected = projected_exp<EXPM>(a.sc);   // (one request per tile: uniform)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = lp.odd ? 1 : 0;
    const int64_t P = a.n_points;
    const bool live = p < P;
    const int64_t q = live ? p : 0;
    const Normal nn{load_or(a.normals, 3 * q, live), load_or(a.normals, 3 * q + 1, live),
                    load_or(a.normals, 3 * q + 2, live)};
    const float* legs = sh.leg + (lp.odd ? NL : 0);
    float f[NS];
    int k;
    if (a.saved_f) {
        lp_load(a.saved_f, P, q, live, lp, f);
        k = live ? min(max(a.saved_k[q], 0), kMaxK) : 0;   // a foreign buffer cannot overrun hist
    } else {
        lp_log_visibility<CULL>(a.sc, sh.sph, load_or(a.points, 3 * q, live), load_or(a.points, 3 * q + 1, live),
                                load_or(a.points, 3 * q + 2, live),
                                CULL ? cull_normal(a.sc, nn.x, nn.y, nn.z) : Normal{}, lp, f);
        k = -1;
    }
    const float n2 = lp_norm2(f, lp);
    if (k < 0) k = scaling_k(a.sc, n2);

    // ---- the exponential again, keeping in local memory f, the operand of
    // every squaring and S with V = e0 S (projected: U).  The operands of the
    // products sit in the warp's columns of shared memory, X and Y (a product's
    // result and work arrays fill the registers).  kmax: the warp's largest k;
    // a pair past its own k keeps S.
    float* X = sh.w + warp * sh.region + lane;
    float* Y = X + 32 * NS;
    float fh[NS], hist[EXPM == kExpProjected ? 1 : kMaxK + 1][NS];
    float scale = 1.f;
    OLCoef ol{1.f, 1.f, 0.f, 0.f};
    const float e0 = expf(lp_even(f[0]) * kInvSqrt4Pi);
    const int kmax = projected ? 0 : __reduce_max_sync(0xffffffffu, k);
#pragma unroll
    for (int s = 0; s < NS; ++s) fh[s] = f[s];
    {
        float S[NS];
        if (projected) {
            if constexpr (EXPM != kExpSquarings) lp_proj_exp(f, legs + kLegProduct, lp, S);
        } else if constexpr (EXPM != kExpProjected) {
            scale = ldexpf(1.f, -k);
            ol = ol_coef(a.sc, n2 * scale * scale);
#pragma unroll
            for (int s = 0; s < NS; ++s) S[s] = ol.b * (f[s] * scale);
            S[0] = lp.odd ? S[0] : ol.a * kSqrt4Pi;
        }
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            X[32 * s] = S[s];
            hist[0][s] = S[s];
        }
    }
#pragma unroll 1
    for (int t = 0; t < kmax; ++t) {
        float T[NS];
        lp_product<true, false, 32>(X, nullptr, legs, lp, T);
        const bool on = t < k;
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            T[s] = on ? T[s] : X[32 * s];
            X[32 * s] = T[s];
            hist[t + 1][s] = T[s];
        }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) X[32 * s] *= e0;

    // ---- loss, dLoss/dB, and u_c = a_c dLoss/dB_c
    float dB[3], uc[3], loss = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        if (a.target) {
            const float r = load_or(a.radiance, 3 * q + c, live) - load_or(a.target, 3 * q + c, live);
            dB[c] = r;
            loss = fmaf(0.5f * r, r, loss);
        } else {
            dB[c] = load_or(a.d_radiance, 3 * q + c, live);
        }
        uc[c] = load_or(a.albedo, 3 * q + c, live) * dB[c];
    }
    if (a.target) {
        const float v = warp_sum(lp.odd ? 0.f : loss);
        if (lane == 0) sh.loss[warp] += v;
    }

    // ---- every two-operand product of the adjoint through one loop body (six
    // inlined products would not fit the instruction cache):
    //   step 0: W = V * H            -> d_albedo, d_light
    //   step 1: dH = dW * V          -> d_normals (C is symmetric: the adjoint of a * b is d * b)
    //   step 2: dV = dW * H
    //   step 3 + i: dS = 2 dS * (operand of squaring kmax - 1 - i)
    const Normal u = unit_normal(nn.x, nn.y, nn.z);
    float de0 = 0.f;   // X: V, then dW, then dV and dS
#pragma unroll 1
    for (int step = 0; step < 3 + kmax; ++step) {
        if (step == 1 && !a.d_normals) continue;
        const int t = kmax + 2 - step;   // squaring, from step 3
        float T[NS];
        if (step == 0 || step == 2) {
            float H[NS];
            lp_cosine_lobe(u.x, u.y, u.z, lp, H);
#pragma unroll
            for (int s = 0; s < NS; ++s) Y[32 * s] = H[s];
        } else {
            const float* h = &hist[step == 1 ? kmax : t][0];
            const float v = step == 1 ? e0 : 1.f;
#pragma unroll
            for (int s = 0; s < NS; ++s) Y[32 * s] = v * h[s];
        }
        lp_product<false, true, 32>(X, Y, legs, lp, T);
        if (step == 0) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                float lw = 0.f;
#pragma unroll
                for (int s = 0; s < NS; ++s) lw = fmaf(sh.lt[b][c][s], T[s], lw);
                lw = lp_sum(lw);
                if (live && !lp.odd && a.d_albedo) a.d_albedo[3 * q + c] = dB[c] * lw;
            }
            if (a.d_light) {
#pragma unroll
                for (int base = 0; base < 3 * NS; base += 16) {
                    float v[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        v[i] = base + i < 3 * NS ? uc[(base + i) / NS] * T[(base + i) % NS] : 0.f;
                    lp_halve<16, 16>(v, lane);
                    sh.dl[warp][b][base + (lane >> 1)] += v[0];
                }
            }
#pragma unroll
            for (int s = 0; s < NS; ++s)
                X[32 * s] = fmaf(uc[0], sh.lt[b][0][s], fmaf(uc[1], sh.lt[b][1][s], uc[2] * sh.lt[b][2][s]));
        } else if (step == 1) {
            float gx, gy, gz;
            lp_lobe_adjoint(u.x, u.y, u.z, T, lp, gx, gy, gz);
            const float n2v = fmaf(nn.x, nn.x, fmaf(nn.y, nn.y, nn.z * nn.z)), il = n2v > 0.f ? rsqrtf(n2v) : 0.f;
            const float ug = u.x * gx + u.y * gy + u.z * gz;
            if (live && !lp.odd) {
                a.d_normals[3 * q] = (gx - u.x * ug) * il;
                a.d_normals[3 * q + 1] = (gy - u.y * ug) * il;
                a.d_normals[3 * q + 2] = (gz - u.z * ug) * il;
            }
        } else if (step == 2) {
#pragma unroll
            for (int s = 0; s < NS; ++s) {
                de0 = fmaf(T[s], hist[kmax][s], de0);
                X[32 * s] = projected ? T[s] : e0 * T[s];
            }
        } else {
            if (t < k) {
#pragma unroll
                for (int s = 0; s < NS; ++s) X[32 * s] = 2.f * T[s];
            }
        }
    }

    // ---- exponent
    if (projected) {
        if constexpr (EXPM != kExpSquarings) {
            float dV[NS];
#pragma unroll
            for (int s = 0; s < NS; ++s) dV[s] = X[32 * s];
            lp_proj_exp_adjoint(fh, dV, e0, legs + kLegProduct, lp, dfp);
        }
    } else if constexpr (EXPM != kExpProjected) {
        // S_0 = a(s) sqrt(4 pi), S_i = b(s) g_i: dg_i = b dS_i + (dA a'/s + dB b'/s) g_i
        const float dA = lp_even(X[0]) * kSqrt4Pi;
        float dBs = lp.odd ? X[0] * (fh[0] * scale) : 0.f;
#pragma unroll
        for (int s = 1; s < NS; ++s) dBs = fmaf(X[32 * s], fh[s] * scale, dBs);
        dBs = lp_sum(dBs);
        const float cg = fmaf(dA, ol.ca, dBs * ol.cb);
#pragma unroll
        for (int s = 0; s < NS; ++s) dfp[s] = fmaf(ol.b, X[32 * s], cg * (fh[s] * scale)) * scale;
    }
    de0 = lp_sum(de0);
    dfp[0] = lp.odd ? dfp[0] : de0 * e0 * kInvSqrt4Pi;
    static_for<NS>([&](auto s) {
        constexpr int i0 = lp_index(s, 0), i1 = lp_index(s, 1);
        dfp[s] *= a.sc.neg_2pi_eps * (lp.odd ? SH::norm(i1 < 0 ? 0 : i1) : SH::norm(i0));
    });
}

// The lane's coefficients into its half of its points' row of shared memory
// (half: a float pointer to the row's entry 0, first or second point).
__device__ __forceinline__ void lp_store_row(const float* dfp, float* half, const LanePair& lp) {
    static_for<NS>([&](auto s) {
        constexpr int m = lp_m(s), l0 = lp_l(s, 0), l1 = lp_l(s, 1), sn = lp_sin(s);
        constexpr int o0 = wcol(m) + (m ? 2 * (l0 - m) + sn : l0), o1 = wcol(m) + (m ? 2 * (l1 - m) + sn : l1);
        constexpr float c0 = dfact(l0) / float(l0 ? l0 * (l0 + 1) : 1), c1 = dfact(l1) / float(l1 * (l1 + 1));
        if (l1 < NB || !lp.odd) half[2 * (lp.odd ? o1 : o0)] = dfp[s] * (lp.odd ? c1 : c0);
    });
}

// Pair adjoints of the warp's 16 points (eight rows of two), one sphere per
// lane; with fewer than 17 (9) spheres the lanes take two (four) rows at once.
template <bool CULL>
__device__ __forceinline__ void lp_pairs(const BwdArgs& a, const BwdShared& sh, int64_t tile) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, N = a.sc.n_spheres;
    const int width = N > 16 ? 32 : N > 8 ? 16 : 8, sub = lane / width, stride = 32 / width;
    float4* acc_row = sh.acc + warp * N;
    const float2* rows = reinterpret_cast<const float2*>(sh.w + warp * sh.region);
    const bool want_pts = a.d_points != nullptr;
    float gp[3] = {0.f, 0.f, 0.f};   // lane t < 16: gradient of the warp's point t
    for (int j0 = 0; j0 < N; j0 += width) {
        const int j = j0 + lane % width;
        const bool has = j < N;
        const float4 sp = has ? sh.sph[j] : make_float4(0.f, 0.f, 0.f, 0.f);
        float2 acc[4] = {};
#pragma unroll 1
        for (int t = 0; t < kWarpRows; t += stride) {
            float2 d[4];
            pair_backward2<CULL>(sp, rows + (t + sub) * WST, d);
            if (!has) d[0] = d[1] = d[2] = d[3] = k2(0.f);
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[e] = __fadd2_rn(acc[e], d[e]);
            if (want_pts) {
#pragma unroll
                for (int e = 0; e < 3; ++e) {
                    for (int o = 1; o < width; o <<= 1) {
                        d[e].x += __shfl_xor_sync(0xffffffffu, d[e].x, o);
                        d[e].y += __shfl_xor_sync(0xffffffffu, d[e].y, o);
                    }
                    // lane 2 (t + i) + h takes half h of the sum its sub-group i holds
                    const int src = (((lane >> 1) - t) & (stride - 1)) * width;
                    const float x = __shfl_sync(0xffffffffu, d[e].x, src), y = __shfl_sync(0xffffffffu, d[e].y, src);
                    if ((lane >> 1) >= t && (lane >> 1) < t + stride) gp[e] -= lane & 1 ? y : x;
                }
            }
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
    }
    const int64_t p = tile * kTile + warp * kWarpPoints + lane;
    if (want_pts && lane < kWarpPoints && p < a.n_points) {
        a.d_points[3 * p] = gp[0];
        a.d_points[3 * p + 1] = gp[1];
        a.d_points[3 * p + 2] = gp[2];
    }
}

// One tile: tail adjoint, then the pair adjoints.  A warp reads only the rows
// it wrote, so warps need no block barrier between the two.  With a workspace
// the two run as launches of their own (kPhaseTail stores the coefficients in
// dfp_ws, kPhasePairs reads them), each of which keeps to one region of code:
// as one launch (kPhaseBoth, for callers without a workspace) the kernel waits
// on instruction fetch (1.1 stalled warps per issue; 1M points, 300 spheres, 8
// bands: 9.2 ms against 8.6 ms).
constexpr int kPhaseBoth = 0, kPhaseTail = 1, kPhasePairs = 2;

template <int EXPM, bool CULL, int PHASE>
__device__ __forceinline__ void lp_backward_tile(const BwdArgs& a, const BwdShared& sh, int64_t tile) {
    const LanePair lp = lane_pair();
    const int row = threadIdx.x >> 1;
    const int64_t p = tile * kTile + row;
    const bool live = p < a.n_points;
    const bool pairs = a.d_centers || a.d_radii || a.d_points;
    float dfp[NS];
    if constexpr (PHASE == kPhasePairs) {
        lp_load(a.dfp_ws, a.n_points, live ? p : 0, live, lp, dfp);
    } else {
        lp_tail_adjoint<EXPM, CULL>(a, sh, p, dfp);
    }
    if constexpr (PHASE == kPhaseTail) {
        if (pairs && live) lp_store(dfp, a.n_points, p, lp, a.dfp_ws);
        return;
    }
    if (!pairs) return;
    __syncwarp();   // the region held the tail's operands
    float* half = sh.w + (row >> 4) * sh.region + ((row & 15) >> 1) * (2 * WST) + (row & 1);
    lp_store_row(dfp, half, lp);
    const int64_t q = live ? p : 0;
    if (!lp.odd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) half[2 * c] = load_or(a.points, 3 * q + c, live);
    } else if (CULL) {
        const Normal u = cull_normal(a.sc, load_or(a.normals, 3 * q, live), load_or(a.normals, 3 * q + 1, live),
                                     load_or(a.normals, 3 * q + 2, live));
        half[6] = u.x;
        half[8] = u.y;
        half[10] = u.z;
    }
    __syncwarp();
    lp_pairs<CULL>(a, sh, tile);
    __syncwarp();
}

// Block total of entry e of the scene-level sums (d_light, loss, spheres).
__device__ __forceinline__ float lp_block_sum(const BwdShared& sh, int N, int e) {
    float v = 0.f;
    if (e < 3 * K) {
        const int c = e / K, i = e % K;
        int l = 0;
        while ((l + 1) * (l + 1) <= i) ++l;
        const int m = i - l * (l + 1), am = m < 0 ? -m : m, b = (l + am) & 1;
        const int s = c * NS + lp_slot(am, m < 0, (l - am - b) >> 1);
#pragma unroll
        for (int w = 0; w < NWARP; ++w) v += sh.dl[w][b][s];
    } else if (e == 3 * K) {
#pragma unroll
        for (int w = 0; w < NWARP; ++w) v += sh.loss[w];
    } else {
        const int q = e - (3 * K + 1);
        const float* acc = reinterpret_cast<const float*>(sh.acc);
#pragma unroll
        for (int w = 0; w < NWARP; ++w) v += acc[w * 4 * N + q];
    }
    return v;
}

#define SHS_LP_BWD_SHARED(EXPM, PHASE)                                                       \
    extern __shared__ __align__(16) float4 dyn[];                                            \
    __shared__ __align__(16) float s_light[3 * KPAD];                                        \
    __shared__ __align__(16) float s_lt[2][3][NSP];                                          \
    __shared__ __align__(16) float s_leg[kLegProduct + ((EXPM) ? kLegExp : 0)];              \
    __shared__ __align__(16) float s_w[NWARP * ((PHASE) == kPhasePairs ? kRowFloats : kWarpRegion)];                       \
    __shared__ float s_dl[NWARP][2][kDl], s_loss[NWARP];                                     \
    __shared__ __align__(8) uint64_t s_bar;                                                  \
    __shared__ bool s_last

__device__ __forceinline__ void clear_sums(const BwdShared& sh, int N) {
    float* acc = reinterpret_cast<float*>(sh.acc);
    for (int e = threadIdx.x; e < NWARP * 4 * N; e += kBlock) acc[e] = 0.f;
    for (int e = threadIdx.x; e < NWARP * 2 * kDl; e += kBlock) (&sh.dl[0][0][0])[e] = 0.f;
    if (threadIdx.x < NWARP) sh.loss[threadIdx.x] = 0.f;
}

// Layout of one block's reduced scene gradient (E floats):
//   [0, 3K)          d_light, channel-major
//   [3K]             loss
//   [3K+1, 3K+1+4N)  per sphere (d cx, d cy, d cz, d r)
template <int EXPM, bool CULL, int PHASE>
__global__ void __launch_bounds__(kBlock, SHS_LP_MINB) backward_lp_kernel(BwdArgs a) {
    SHS_LP_BWD_SHARED(EXPM, PHASE);
    const int N = a.sc.n_spheres;
    const BwdShared sh{dyn, dyn + N, s_lt, s_leg, s_dl, s_loss, s_w, PHASE == kPhasePairs ? kRowFloats : kWarpRegion};
    if (PHASE != kPhasePairs) load_rules(s_leg, EXPM != kExpSquarings);
    if (!stage_scene(a.sc, sh.sph, s_light, &s_bar)) return;
    clear_sums(sh, PHASE == kPhaseTail ? 0 : N);
    slot_lighting(s_light, s_lt);

    const int64_t ntiles = (a.n_points + kTile - 1) / kTile;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x)
        lp_backward_tile<EXPM, CULL, PHASE>(a, sh, tile);

    // ---- block reduction of the phase's entries, then one scene-level
    // reduction (by the last launch)
    __syncthreads();
    const int E = 3 * K + 1 + 4 * N, begin = PHASE == kPhasePairs ? 3 * K + 1 : 0,
              end = PHASE == kPhaseTail ? 3 * K + 1 : E;
    float* out = a.partials + static_cast<size_t>(blockIdx.x) * a.partial_stride;
    const bool det = a.counter == nullptr;
    for (int e = begin + threadIdx.x; e < end; e += kBlock) {
        const float v = lp_block_sum(sh, N, e);
        if (det) out[e] = v;
        else atomicAdd(a.partials + e, v);
    }
    if (det || PHASE == kPhaseTail) return;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    finish_scene_sums(a, E);
}

// ---------------------------------------------------------------------------
// batched persistent kernel (serving): many requests, one launch
// ---------------------------------------------------------------------------

// Adjoint for every tile of every request in the batch.  Each tile's scene
// sums go to its request's accumulator with atomics; the tile that completes a
// request writes that request's outputs.
template <int EXPM, bool CULL>
__global__ void __launch_bounds__(kBlock, SHS_LP_MINB) backward_batch_kernel(const __grid_constant__ BwdBatch b) {
    SHS_LP_BWD_SHARED(EXPM, kPhaseBoth);
    __shared__ long long s_tile;
    const BwdShared sh{dyn, dyn + b.max_spheres, s_lt, s_leg, s_dl, s_loss, s_w, kWarpRegion};
    load_rules(s_leg, EXPM != kExpSquarings);
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
            if (!stage_copy(a.sc, sh.sph, s_light, &s_bar, parity)) return;
            parity ^= 1u;
            staged = r;
            slot_lighting(s_light, s_lt);
        }
        clear_sums(sh, N);
        __syncthreads();
        lp_backward_tile<EXPM, CULL, kPhaseBoth>(a, sh, tile - b.tile_begin[r]);
        __syncthreads();
        const int E = 3 * K + 1 + 4 * N;
        for (int e = threadIdx.x; e < E; e += kBlock) add_tile_sum(a, e, lp_block_sum(sh, N, e));
        __threadfence();
        __syncthreads();
        const int64_t ntiles_r = b.tile_begin[r + 1] - b.tile_begin[r];
        if (threadIdx.x == 0) s_last = atomicAdd(a.counter, 1u) == static_cast<unsigned>(ntiles_r - 1);
        __syncthreads();
        if (s_last) finish_scene_sums(a, E);
    }
}

size_t backward_dyn_smem(int n_spheres) { return static_cast<size_t>(n_spheres) * 16u * (1 + NWARP); }

// The tail launch stages the spheres only to recompute f; it has no sphere sums.
size_t phase_dyn_smem(int phase, int n_spheres) {
    return phase == kPhaseTail ? static_cast<size_t>(n_spheres) * 16u : backward_dyn_smem(n_spheres);
}

template <int EXPM, bool CULL, int PHASE>
cudaError_t launch_backward_lp(const BwdArgs& a, int grid, cudaStream_t s) {
    static DeviceOnce once;
    const cudaError_t e = allow_dyn_smem(backward_lp_kernel<EXPM, CULL, PHASE>, phase_dyn_smem(PHASE, kMaxSpheres), once);
    if (e != cudaSuccess) return e;
    backward_lp_kernel<EXPM, CULL, PHASE>
        <<<static_cast<unsigned>(grid), kBlock, phase_dyn_smem(PHASE, a.sc.n_spheres), s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int PHASE>
cudaError_t launch_phase(const BwdArgs& a, int grid, cudaStream_t s) {
    const bool cull = a.sc.horizon_cull != 0, exp1 = PHASE != kPhasePairs && a.sc.exp_mode == 1;
    constexpr int kExp1 = PHASE != kPhasePairs ? kExpProjected : kExpSquarings;
    if (exp1) return cull ? launch_backward_lp<kExp1, true, PHASE>(a, grid, s) : launch_backward_lp<kExp1, false, PHASE>(a, grid, s);
    return cull ? launch_backward_lp<kExpSquarings, true, PHASE>(a, grid, s)
                : launch_backward_lp<kExpSquarings, false, PHASE>(a, grid, s);
}

template <int PHASE>
int phase_blocks(int n_spheres) {
    cudaFuncSetAttribute(backward_lp_kernel<kExpSquarings, false, PHASE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         static_cast<int>(phase_dyn_smem(PHASE, kMaxSpheres)));
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, backward_lp_kernel<kExpSquarings, false, PHASE>, kBlock,
                                                      phase_dyn_smem(PHASE, n_spheres)) != cudaSuccess || nb < 1)
        nb = 1;
    return nb;
}

template <int EXPM, bool CULL>
cudaError_t launch_backward_batch_lp(const BwdBatch& b, cudaStream_t s) {
    const size_t smem = backward_dyn_smem(b.max_spheres);
    static DeviceOnce once;
    static WaveCache wave;
    int grid = 0;
    cudaError_t e = allow_dyn_smem(backward_batch_kernel<EXPM, CULL>, backward_dyn_smem(kMaxSpheres), once);
    if (e == cudaSuccess) e = one_wave(backward_batch_kernel<EXPM, CULL>, smem, b.total_tiles, wave, &grid);
    if (e != cudaSuccess) return e;
    backward_batch_kernel<EXPM, CULL><<<grid, kBlock, smem, s>>>(b);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

template <>
BwdBlocks backward_blocks_per_sm<NB>(int n_spheres, bool split) {
    if (!split) return BwdBlocks{phase_blocks<kPhaseBoth>(n_spheres), 0, 0};
    return BwdBlocks{0, phase_blocks<kPhaseTail>(n_spheres), phase_blocks<kPhasePairs>(n_spheres)};
}

template <>
cudaError_t launch_backward_batch<NB>(const BwdBatch& b, cudaStream_t s) {
    if (b.total_tiles <= 0) return cudaSuccess;
    if (b.variant.squarings && b.variant.projected) return launch_backward_batch_lp<kExpAny, true>(b, s);
    if (b.variant.projected) {
        return b.variant.cull ? launch_backward_batch_lp<kExpProjected, true>(b, s)
                              : launch_backward_batch_lp<kExpProjected, false>(b, s);
    }
    return b.variant.cull ? launch_backward_batch_lp<kExpSquarings, true>(b, s)
                          : launch_backward_batch_lp<kExpSquarings, false>(b, s);
}

template <>
cudaError_t launch_backward<NB>(const BwdArgs& a, cudaStream_t s) {
    if (a.n_points <= 0) return cudaSuccess;
    cudaError_t err = cudaSuccess;
    if (a.dfp_ws) {
        if (a.tail_grid) err = launch_phase<kPhaseTail>(a, a.tail_grid, s);   // else: ran on the tensor cores
        const bool need_pairs = a.d_centers || a.d_radii || a.d_points;
        if (err == cudaSuccess && (need_pairs || a.counter != nullptr)) err = launch_phase<kPhasePairs>(a, a.grid, s);
    } else {
        err = launch_phase<kPhaseBoth>(a, a.grid, s);
    }
    if (err != cudaSuccess || a.counter != nullptr) return err;
    const int E = 3 * K + 1 + 4 * a.sc.n_spheres;
    reduce_partials_kernel<<<reduce_blocks(E), kReduceThreads, 0, s>>>(a, a.dfp_ws && a.tail_grid ? a.tail_grid : a.grid,
                                                                       a.grid);
    count_launch();
    return cudaGetLastError();
}

}  // namespace shs
