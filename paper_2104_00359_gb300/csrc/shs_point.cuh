// Shared by the kernels of every band count: staging of a scene into shared
// memory, the geometry of a point-sphere pair, and the scene-level sums'
// finish.  Included by translation units compiled with -DSHS_NB=n.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "generated/shs_sh_gen.cuh"
#include "shs_internal.h"

#ifndef SHS_NB
#error "compile with -DSHS_NB=<n_bands>"
#endif

namespace shs {
namespace {

constexpr int NB = SHS_NB;
constexpr int K = NB * NB;
constexpr int KPAD = (K + 3) / 4 * 4;
constexpr int NWARP = kBlock / 32;
using SH = shsgen::SH<NB>;


__host__ __device__ constexpr int band_of(int i) {
    int l = 0;
    while ((l + 1) * (l + 1) <= i) ++l;
    return l;
}

__device__ __forceinline__ float fast_sqrt(float x) {   // sqrt(x) = x / sqrt(x), x >= 0
    return x * rsqrtf(fmaxf(x, 1e-30f));
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// One mbarrier per block tracks the bulk copies that stage a scene (sphere
// array + lighting) into shared memory.  Initialise it once per block.
__device__ void mbar_init(uint64_t* bar) {
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
}

// Stage a scene with bulk asynchronous copies completing on `bar` (phase
// `parity`, alternating between stagings).  Every thread waits with a bound of
// about one second; the result is block-uniform: false means the copy did not
// complete, the status word is set and the block must not use the data.  The
// caller must have synchronised the block if shared memory held a previous
// scene that threads may still read.
__device__ bool stage_copy(const SceneView& sc, float4* s_sph, float* s_light, uint64_t* bar,
                           uint32_t parity) {
    const uint32_t sph_bytes = static_cast<uint32_t>(sc.n_spheres) * 16u;
    const uint32_t light_bytes = 3u * KPAD * 4u;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;"
                     ::"r"(smem_addr(bar)), "r"(sph_bytes + light_bytes) : "memory");
        if (sph_bytes)
            asm volatile(
                "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                ::"r"(smem_addr(s_sph)), "l"(sc.spheres), "r"(sph_bytes), "r"(smem_addr(bar))
                : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
            ::"r"(smem_addr(s_light)), "l"(sc.light), "r"(light_bytes), "r"(smem_addr(bar))
            : "memory");
    }
    bool done = false;
    const uint64_t t0 = global_ns();
    for (uint32_t it = 0; it < (1u << 26) && !done; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
            " selp.b32 %0, 1, 0, p;\n}\n"
            : "=r"(ok) : "r"(smem_addr(bar)), "r"(parity) : "memory");
        done = ok != 0;
        if (!done && global_ns() - t0 > 1000000000ull) break;
    }
    const bool any_failed = __syncthreads_or(!done);
    if (any_failed && threadIdx.x == 0) atomicExch(sc.status, kDevTimeout);
    return !any_failed;
}

__device__ bool stage_scene(const SceneView& sc, float4* s_sph, float* s_light, uint64_t* bar) {
    mbar_init(bar);
    return stage_copy(sc, s_sph, s_light, bar, 0u);
}

struct PairGeom {
    float dx, dy, dz, invD, invD2, s2, c;
    bool open;
};

// Unit normal of the shading point, used by horizon culling.
struct Normal {
    float x = 0.f, y = 0.f, z = 0.f;
};

__device__ __forceinline__ Normal unit_normal(float nx, float ny, float nz) {
    const float n2 = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
    const float il = n2 > 0.f ? rsqrtf(n2) : 0.f;
    return Normal{nx * il, ny * il, nz * il};
}

// With CULL (the optional horizon-culling reading), a sphere entirely below
// the tangent plane at x, (c - x) . n_hat < -r, becomes an empty cap: s2 = 0
// and c = 1 make every G_l zero, and a closed cap carries no gradient.
template <bool CULL = false>
__device__ __forceinline__ PairGeom pair_geometry(float px, float py, float pz, float4 sp, Normal u = {}) {
    PairGeom g;
    g.dx = sp.x - px;
    g.dy = sp.y - py;
    g.dz = sp.z - pz;
    const float D2 = fmaf(g.dx, g.dx, fmaf(g.dy, g.dy, g.dz * g.dz));
    g.invD = D2 > 0.f ? rsqrtf(D2) : 0.f;     // D = 0: every term below vanishes
    g.invD2 = g.invD * g.invD;
    const float r2i = sp.w * sp.w * g.invD2;
    g.open = r2i < 1.f;
    g.s2 = fminf(r2i, 1.f);                   // point inside the sphere: hemisphere cap
    g.c = fast_sqrt(1.f - g.s2);
    if constexpr (CULL) {
        if (fmaf(g.dx, u.x, fmaf(g.dy, u.y, g.dz * u.z)) < -sp.w) {
            g.s2 = 0.f;
            g.c = 1.f;
            g.open = false;
        }
    }
    return g;
}

// The same for one sphere and two points, one per half of every float2, in the
// packed float32x2 instructions (identical arithmetic per half).  ic = 1 / c.
struct PairGeom2 {
    float2 dx, dy, dz, invD, invD2, s2, c, ic;
    bool open0, open1;
};

template <bool CULL>
__device__ __forceinline__ PairGeom2 pair_geometry2(float2 px, float2 py, float2 pz, float4 sp, const float2* u) {
    const float2 one = make_float2(1.f, 1.f), mone = make_float2(-1.f, -1.f);
    PairGeom2 g;
    g.dx = make_float2(sp.x - px.x, sp.x - px.y);
    g.dy = make_float2(sp.y - py.x, sp.y - py.y);
    g.dz = make_float2(sp.z - pz.x, sp.z - pz.y);
    const float2 D2 = __ffma2_rn(g.dx, g.dx, __ffma2_rn(g.dy, g.dy, __fmul2_rn(g.dz, g.dz)));
    g.invD = make_float2(D2.x > 0.f ? rsqrtf(D2.x) : 0.f, D2.y > 0.f ? rsqrtf(D2.y) : 0.f);
    g.invD2 = __fmul2_rn(g.invD, g.invD);
    const float r2 = sp.w * sp.w;
    const float2 r2i = __fmul2_rn(make_float2(r2, r2), g.invD2);
    g.open0 = r2i.x < 1.f;
    g.open1 = r2i.y < 1.f;
    g.s2 = make_float2(fminf(r2i.x, 1.f), fminf(r2i.y, 1.f));
    const float2 om = __ffma2_rn(g.s2, mone, one);
    g.ic = make_float2(rsqrtf(fmaxf(om.x, 1e-30f)), rsqrtf(fmaxf(om.y, 1e-30f)));
    g.c = __fmul2_rn(om, g.ic);
    if constexpr (CULL) {   // u: the points' unit normals
        const float2 h = __ffma2_rn(g.dx, u[0], __ffma2_rn(g.dy, u[1], __fmul2_rn(g.dz, u[2])));
        if (h.x < -sp.w) {
            g.s2.x = 0.f;
            g.c.x = 1.f;
            g.open0 = false;
        }
        if (h.y < -sp.w) {
            g.s2.y = 0.f;
            g.c.y = 1.f;
            g.open1 = false;
        }
    }
    return g;
}

// dPsi/dd and dPsi/dr of two pairs from s_hat, s_hat's gradient a (its radial
// part is removed here) and ga = -dPsi/dc.
__device__ __forceinline__ void pair_finish2(const PairGeom2& g, float r, float2 sx, float2 sy, float2 sz, float2 ax,
                                             float2 ay, float2 az, float2 ga, float2* d) {
    const float2 mone = make_float2(-1.f, -1.f);
    // c = sqrt(1 - s2): d c / d s2 = -1 / (2 c); clamped caps carry no gradient
    const float2 h = __fmul2_rn(ga, g.ic);
    const float2 t = __fmul2_rn(make_float2(g.open0 ? h.x : 0.f, g.open1 ? h.y : 0.f), g.invD2);   // 2 dPsi/ds2 / D^2
    const float2 coef = __fmul2_rn(__fmul2_rn(t, mone), g.s2);                                     // 2 dPsi/dD^2
    const float2 nrad = __fmul2_rn(mone, __ffma2_rn(sx, ax, __ffma2_rn(sy, ay, __fmul2_rn(sz, az))));
    d[0] = __ffma2_rn(__ffma2_rn(nrad, sx, ax), g.invD, __fmul2_rn(coef, g.dx));
    d[1] = __ffma2_rn(__ffma2_rn(nrad, sy, ay), g.invD, __fmul2_rn(coef, g.dy));
    d[2] = __ffma2_rn(__ffma2_rn(nrad, sz, az), g.invD, __fmul2_rn(coef, g.dz));
    d[3] = __fmul2_rn(t, make_float2(r, r));                                                       // s2 = r^2 / D^2
}

__device__ __forceinline__ float load_or(const float* p, int64_t i, bool live) {
    return live ? __ldg(p + i) : 0.f;
}

// Parts of the forward pass a kernel runs: everything; the log-visibility f
// only, stored; or, from a stored f, the exponential and shading.
constexpr int kFwdFull = 0, kFwdPairs = 1, kFwdTail = 2;

// Adds the tile's total of entry e to a batch request's accumulator.  The
// loss, a sum of a thousand terms of one sign and more, is added in float64:
// in float32 its error grows with the number of tiles (2e-6 at 16k tiles).
__device__ __forceinline__ void add_tile_sum(const BwdArgs& a, int e, float v) {
    if (e == 3 * K) {
        if (a.loss) atomicAdd(a.loss_sum, static_cast<double>(v));
    } else {
        atomicAdd(a.partials + e, v);
    }
}

// The last contributor copies the accumulated scene-level sums to the
// outputs and re-zeroes the accumulator and its counter for the next launch.
__device__ void finish_scene_sums(const BwdArgs& a, int E) {
    __threadfence();
    for (int e = threadIdx.x; e < E; e += kBlock) {
        float v = __ldcg(a.partials + e);
        a.partials[e] = 0.f;
        if (e == 3 * K && a.loss_sum) {
            v = static_cast<float>(__ldcg(a.loss_sum));
            *a.loss_sum = 0.0;
        }
        if (e < 3 * K) {
            if (a.d_light) a.d_light[e] = v;
        } else if (e == 3 * K) {
            if (a.loss) *a.loss = v;
        } else {
            const int s = e - (3 * K + 1), j = s >> 2, comp = s & 3;
            if (comp < 3) {
                if (a.d_centers) a.d_centers[3 * j + comp] = v;
            } else if (a.d_radii) {
                a.d_radii[j] = v;
            }
        }
    }
    if (threadIdx.x == 0) *a.counter = 0u;
}

__device__ __forceinline__ int find_request(const int64_t* tb, int n, int64_t tile) {
    int r = 0;
    while (r + 1 < n && tile >= tb[r + 1]) ++r;
    return r;
}

// Deterministic finish: fixed-order sum of the blocks' partial rows (the
// lighting and loss entries and the sphere entries may come from launches with
// different grids).  One block per 8 entries (a 32-byte sector of a row); its
// 64 slices of rows take at most eight loads each up to 512 rows, all issued
// before any is added: one trip to the L2 instead of the four of 32 slices
// that each held 32 entries (the sum is latency-bound: 456 rows x 449 entries
// 6.6 -> 3.7 us).
constexpr int kReduceEntries = 8, kReduceThreads = 512, kReduceSlices = kReduceThreads / kReduceEntries;
inline int reduce_blocks(int entries) { return (entries + kReduceEntries - 1) / kReduceEntries; }

__global__ void __launch_bounds__(kReduceThreads) reduce_partials_kernel(BwdArgs a, int light_rows, int sphere_rows) {
    __shared__ float s[kReduceThreads / 32][kReduceEntries];
    const int N = a.sc.n_spheres;
    const int E = 3 * K + 1 + 4 * N;
    const int slice = threadIdx.x / kReduceEntries, e = blockIdx.x * kReduceEntries + threadIdx.x % kReduceEntries;
    const int nblk = e <= 3 * K ? light_rows : sphere_rows;
    float t = 0.f;
    if (e < E) {
        const float* col = a.partials + e;
        const size_t st = static_cast<size_t>(a.partial_stride);
        for (int b = slice; b < nblk; b += 8 * kReduceSlices) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                v[u] = b + u * kReduceSlices < nblk ? __ldcg(col + (b + u * kReduceSlices) * st) : 0.f;
            t += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
        }
    }
    t += __shfl_xor_sync(0xffffffffu, t, 8);
    t += __shfl_xor_sync(0xffffffffu, t, 16);
    if ((threadIdx.x & 31) < kReduceEntries) s[threadIdx.x >> 5][threadIdx.x & 31] = t;
    __syncthreads();
    if (threadIdx.x >= kReduceEntries || e >= E) return;
    t = 0.f;
#pragma unroll
    for (int w = 0; w < kReduceThreads / 32; ++w) t += s[w][threadIdx.x];
    if (e < 3 * K) {
        if (a.d_light) a.d_light[e] = t;
    } else if (e == 3 * K) {
        if (a.loss) *a.loss = t;
    } else {
        const int q = e - (3 * K + 1), j = q >> 2, comp = q & 3;
        if (comp < 3) {
            if (a.d_centers) a.d_centers[3 * j + comp] = t;
        } else if (a.d_radii) {
            a.d_radii[j] = t;
        }
    }
}

}  // namespace
}  // namespace shs
