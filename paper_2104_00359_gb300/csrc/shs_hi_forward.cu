// Forward shading kernels for 6, 7 and 8 bands, compiled once per n_bands with
// -DSHS_NB=n: one lane pair per point, 64 points per block (shs_hi.cuh).

#include <cstdint>
#include <cuda_runtime.h>

#include "shs_hi.cuh"

namespace shs {
namespace {

template <int MODE, int EXPM, bool CULL>
__device__ __forceinline__ void lp_forward_tile(const FwdArgs& a, const float4* s_sph, const float (*s_lt)[3][NSP],
                                                const float* s_leg, int64_t tile) {
    const LanePair lp = lane_pair();
    const int64_t p = tile * kTile + (threadIdx.x >> 1);
    const bool live = p < a.n_points;
    const int64_t q = live ? p : 0;
    float f[NS];
    float nx = 0.f, ny = 0.f, nz = 1.f;
    if (MODE != kFwdPairs || CULL) {
        nx = load_or(a.normals, 3 * q, live);
        ny = load_or(a.normals, 3 * q + 1, live);
        nz = load_or(a.normals, 3 * q + 2, live);
    }
    if constexpr (MODE == kFwdTail) {
        lp_load(a.saved_f, a.n_points, q, live, lp, f);
    } else {
        lp_log_visibility<CULL>(a.sc, s_sph, load_or(a.points, 3 * q, live), load_or(a.points, 3 * q + 1, live),
                                load_or(a.points, 3 * q + 2, live), CULL ? cull_normal(a.sc, nx, ny, nz) : Normal{}, lp, f);
        if (a.saved_f && live) lp_store(f, a.n_points, p, lp, a.saved_f);
        if constexpr (MODE == kFwdPairs) return;
    }
    const float* legs = s_leg + (lp.odd ? NL : 0);
    const float e0 = expf(lp_even(f[0]) * kInvSqrt4Pi);
    float V[NS];
    int k = 0;
    // (a tile belongs to one request: the branch is uniform)
    if (projected_exp<EXPM>(a.sc)) {
        if constexpr (EXPM != kExpSquarings) lp_proj_exp(f, legs + kLegProduct, lp, V);
    } else if constexpr (EXPM != kExpProjected) {
        const float n2 = lp_norm2(f, lp);
        k = scaling_k(a.sc, n2);
        const float scale = ldexpf(1.f, -k);
        const OLCoef ol = ol_coef(a.sc, n2 * scale * scale);
#pragma unroll
        for (int s = 0; s < NS; ++s) V[s] = ol.b * (f[s] * scale);
        V[0] = lp.odd ? V[0] : ol.a * kSqrt4Pi;
        lp_squarings(V, k, legs, lp, [](int, const float*) {});
    }
#pragma unroll
    for (int s = 0; s < NS; ++s) V[s] *= e0;
    float H[NS], W[NS];
    const Normal u = unit_normal(nx, ny, nz);
    lp_cosine_lobe(u.x, u.y, u.z, lp, H);
    lp_product<false>(V, H, legs, lp, W);
    float d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d[c] = 0.f;
#pragma unroll
        for (int s = 0; s < NS; ++s) d[c] = fmaf(s_lt[lp.odd ? 1 : 0][c][s], W[s], d[c]);
        d[c] = lp_sum(d[c]);
    }
    if (live && !lp.odd) {
#pragma unroll
        for (int c = 0; c < 3; ++c) a.radiance[3 * p + c] = __ldg(a.albedo + 3 * p + c) * d[c];
        if (MODE == kFwdFull && a.saved_k) a.saved_k[p] = k;
    }
}

template <int MODE, int EXPM, bool CULL>
__global__ void __launch_bounds__(kBlock, SHS_LP_MINB) forward_lp_kernel(FwdArgs a) {
    __shared__ __align__(16) float4 s_sph[MODE == kFwdTail ? 1 : kMaxSpheres];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(16) float s_lt[2][3][NSP];
    __shared__ __align__(16) float s_leg[kLegProduct + (EXPM ? kLegExp : 0)];
    __shared__ __align__(8) uint64_t s_bar;
    if (MODE == kFwdTail) a.sc.n_spheres = 0;
    if (MODE != kFwdPairs) load_rules(s_leg, EXPM != kExpSquarings);
    if (!stage_scene(a.sc, s_sph, s_light, &s_bar)) return;
    if (MODE != kFwdPairs) slot_lighting(s_light, s_lt);
    lp_forward_tile<MODE, EXPM, CULL>(a, s_sph, s_lt, s_leg, blockIdx.x);
}

// ---------------------------------------------------------------------------
// batched persistent kernel (serving): many requests, one launch
// ---------------------------------------------------------------------------

// Forward for every tile of every request in the batch.  Blocks take tiles
// from a device counter (consecutive tiles mostly share a request, so a
// request's scene is staged once per run of its tiles).
template <int EXPM, bool CULL>
__global__ void __launch_bounds__(kBlock, SHS_LP_MINB) forward_batch_kernel(const __grid_constant__ FwdBatch b) {
    __shared__ __align__(16) float4 s_sph[kMaxSpheres];
    __shared__ __align__(16) float s_light[3 * KPAD];
    __shared__ __align__(16) float s_lt[2][3][NSP];
    __shared__ __align__(16) float s_leg[kLegProduct + (EXPM ? kLegExp : 0)];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ long long s_tile;
    load_rules(s_leg, EXPM != kExpSquarings);
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
        const FwdArgs& a = b.r[r];
        if (r != staged) {
            if (!stage_copy(a.sc, s_sph, s_light, &s_bar, parity)) return;
            parity ^= 1u;
            staged = r;
            slot_lighting(s_light, s_lt);
        }
        lp_forward_tile<kFwdFull, EXPM, CULL>(a, s_sph, s_lt, s_leg, tile - b.tile_begin[r]);
    }
}

template <int MODE>
cudaError_t launch_forward_lp(const FwdArgs& a, cudaStream_t s) {
    const unsigned blocks = static_cast<unsigned>((a.n_points + kTile - 1) / kTile);
    const bool exp1 = MODE != kFwdPairs && a.sc.exp_mode == 1;      // the pair pass has no exponential
    const bool cull = MODE != kFwdTail && a.sc.horizon_cull != 0;   // the tail has no spheres
    constexpr int kExp1 = MODE != kFwdPairs ? kExpProjected : kExpSquarings;
    if (exp1 && cull) forward_lp_kernel<MODE, kExp1, MODE != kFwdTail><<<blocks, kBlock, 0, s>>>(a);
    else if (exp1) forward_lp_kernel<MODE, kExp1, false><<<blocks, kBlock, 0, s>>>(a);
    else if (cull) forward_lp_kernel<MODE, kExpSquarings, MODE != kFwdTail><<<blocks, kBlock, 0, s>>>(a);
    else forward_lp_kernel<MODE, kExpSquarings, false><<<blocks, kBlock, 0, s>>>(a);
    count_launch();
    return cudaGetLastError();
}

template <int EXPM, bool CULL>
cudaError_t launch_forward_batch_lp(const FwdBatch& b, cudaStream_t s) {
    static WaveCache wave;
    int grid = 0;
    const cudaError_t e = one_wave(forward_batch_kernel<EXPM, CULL>, 0, b.total_tiles, wave, &grid);
    if (e != cudaSuccess) return e;
    forward_batch_kernel<EXPM, CULL><<<grid, kBlock, 0, s>>>(b);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

template <>
cudaError_t launch_forward_batch<NB>(const FwdBatch& b, cudaStream_t s) {
    if (b.total_tiles <= 0) return cudaSuccess;
    if (b.variant.squarings && b.variant.projected) return launch_forward_batch_lp<kExpAny, true>(b, s);
    if (b.variant.projected) {
        return b.variant.cull ? launch_forward_batch_lp<kExpProjected, true>(b, s)
                              : launch_forward_batch_lp<kExpProjected, false>(b, s);
    }
    return b.variant.cull ? launch_forward_batch_lp<kExpSquarings, true>(b, s)
                          : launch_forward_batch_lp<kExpSquarings, false>(b, s);
}

template <>
cudaError_t launch_forward_pairs<NB>(const FwdArgs& a, cudaStream_t s) {
    return a.n_points <= 0 ? cudaSuccess : launch_forward_lp<kFwdPairs>(a, s);
}

template <>
cudaError_t launch_forward<NB>(const FwdArgs& a, cudaStream_t s) {
    if (a.n_points <= 0) return cudaSuccess;
    return a.tail_only ? launch_forward_lp<kFwdTail>(a, s) : launch_forward_lp<kFwdFull>(a, s);
}

}  // namespace shs
