// Generated by gen_tables.py -- do not edit.
// Real SH polynomials, their reverse-mode gradients, and the truncated
// SH triple product (Sec. 3.2, Eq. 3 and Eq. 6-7), unrolled per band count
// (from 6 bands, lane-pair quadrature tables for the triple product instead).
#pragma once

namespace shsgen {

template <int NB> struct SH;

#if defined(SHS_NB) && SHS_NB == 1
static __constant__ float kExpLeg1[2] = {0.282094806432724f, 0.282094806432724f};
static __constant__ float kExpTrig1[4] = {1.0f, 1.0f, 1.0f, 1.0f};
static __constant__ float kExpW1[2] = {1.5707963705062866f, 1.5707963705062866f};
#endif
template <> struct SH<1> {
    static constexpr int K = 1;
    static constexpr int NNZ_SYM = 1;   // entries (i, j <= k)
    static constexpr int EZ = 2;    // projected-exponential rule: Gauss-Legendre nodes
    static constexpr int EP = 4;    // projected-exponential rule: uniform azimuths
#if defined(SHS_NB) && SHS_NB == 1
    __device__ __forceinline__ static const float* eleg() { return kExpLeg1; }
    __device__ __forceinline__ static const float* etrig() { return kExpTrig1; }
    __device__ __forceinline__ static const float* ew() { return kExpW1; }
#endif
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static void ybar(float x, float y, float z, float* Y) {
        (void)x; (void)y; (void)z;
        Y[0] = 1.0f;
    }
    __device__ __forceinline__ static void ybar_vjp(float x, float y, float z, const float* w,
                                                    float& gx, float& gy, float& gz) {
        (void)x; (void)y; (void)z; (void)w;
        gx = 0.0f;
        gy = 0.0f;
        gz = 0.0f;
    }
    static constexpr int NA = 1;   // monomials of degree < n
    static constexpr int NG = 0;   // symmetric tensor entries, bands >= 1
    __device__ __forceinline__ static void accumulate(const float* G, float x, float y, float z, float* acc) {
        (void)x; (void)y; (void)z;
        acc[0] = fmaf(G[0], 1.0f, acc[0]);
    }
    // the same for two pairs at once, one per half of each float2
    __device__ __forceinline__ static void accumulate2(const float2* G, float2 x, float2 y, float2 z,
                                                       float2* acc) {
        (void)x; (void)y; (void)z;
        acc[0] = __fadd2_rn(G[0], acc[0]);
    }
    __device__ __forceinline__ static void mono_to_f(const float* acc, float* f) {
        f[0] = 1.0f * acc[0];
    }
    __device__ __forceinline__ static void grad_coeffs(const float* w, float* gq) {
        (void)w; (void)gq;

    }
    template <class Q>
    __device__ __forceinline__ static void grad_eval2(float2 x, float2 y, float2 z, Q&& gq,
                                                      float2* gx, float2* gy, float2* gz) {
        (void)x; (void)y; (void)z; (void)gq; (void)gx; (void)gy; (void)gz;

    }
    __device__ __forceinline__ static void mul(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = 0.282094806432724f * a[0] * b[0];
    }
    __device__ __forceinline__ static void mul_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = 0.282094806432724f * a[0] * b[0];
    }
    __device__ __forceinline__ static void mul_onto_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = 0.282094806432724f * a[0] * b[0];
    }
    __device__ __forceinline__ static void sqr(const float* __restrict__ a, float* __restrict__ o) {
        o[0] = 0.282094806432724f * a[0] * a[0];
    }
};

#if defined(SHS_NB) && SHS_NB == 2
static __constant__ float kExpLeg2[16] = {0.282094806432724f, 0.24839287996292114f, -0.4207533597946167f, 0.24839287996292114f, 0.282094806432724f, 0.4594975709915161f, -0.16611559689044952f, 0.4594975709915161f, 0.282094806432724f, 0.4594975709915161f, 0.16611559689044952f, 0.4594975709915161f, 0.282094806432724f, 0.24839287996292114f, 0.4207533597946167f, 0.24839287996292114f};
static __constant__ float kExpTrig2[24] = {1.0f, 0.9238795042037964f, 0.3826834261417389f, 1.0f, 0.3826834261417389f, 0.9238795042037964f, 1.0f, -0.3826834261417389f, 0.9238795042037964f, 1.0f, -0.9238795042037964f, 0.3826834261417389f, 1.0f, -0.9238795042037964f, -0.3826834261417389f, 1.0f, -0.3826834261417389f, -0.9238795042037964f, 1.0f, 0.3826834261417389f, -0.9238795042037964f, 1.0f, 0.9238795042037964f, -0.3826834261417389f};
static __constant__ float kExpW2[4] = {0.2732045650482178f, 0.5121936202049255f, 0.5121936202049255f, 0.2732045650482178f};
#endif
template <> struct SH<2> {
    static constexpr int K = 4;
    static constexpr int NNZ_SYM = 7;   // entries (i, j <= k)
    static constexpr int EZ = 4;    // projected-exponential rule: Gauss-Legendre nodes
    static constexpr int EP = 8;    // projected-exponential rule: uniform azimuths
#if defined(SHS_NB) && SHS_NB == 2
    __device__ __forceinline__ static const float* eleg() { return kExpLeg2; }
    __device__ __forceinline__ static const float* etrig() { return kExpTrig2; }
    __device__ __forceinline__ static const float* ew() { return kExpW2; }
#endif
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static void ybar(float x, float y, float z, float* Y) {
        (void)x; (void)y; (void)z;
        Y[0] = 1.0f;
        Y[1] = y;
        Y[2] = z;
        Y[3] = x;
    }
    __device__ __forceinline__ static void ybar_vjp(float x, float y, float z, const float* w,
                                                    float& gx, float& gy, float& gz) {
        (void)x; (void)y; (void)z; (void)w;
        gx = w[3];
        gy = w[1];
        gz = w[2];
    }
    static constexpr int NA = 4;   // monomials of degree < n
    static constexpr int NG = 3;   // symmetric tensor entries, bands >= 1
    __device__ __forceinline__ static void accumulate(const float* G, float x, float y, float z, float* acc) {
        (void)x; (void)y; (void)z;
        const float m1_0_0 = x;
        const float m0_1_0 = y;
        const float m0_0_1 = z;
        acc[0] = fmaf(G[0], 1.0f, acc[0]);
        acc[1] = fmaf(G[1], m1_0_0, acc[1]);
        acc[2] = fmaf(G[1], m0_1_0, acc[2]);
        acc[3] = fmaf(G[1], m0_0_1, acc[3]);
    }
    // the same for two pairs at once, one per half of each float2
    __device__ __forceinline__ static void accumulate2(const float2* G, float2 x, float2 y, float2 z,
                                                       float2* acc) {
        (void)x; (void)y; (void)z;
        const float2 m1_0_0 = x;
        const float2 m0_1_0 = y;
        const float2 m0_0_1 = z;
        acc[0] = __fadd2_rn(G[0], acc[0]);
        acc[1] = __ffma2_rn(G[1], m1_0_0, acc[1]);
        acc[2] = __ffma2_rn(G[1], m0_1_0, acc[2]);
        acc[3] = __ffma2_rn(G[1], m0_0_1, acc[3]);
    }
    __device__ __forceinline__ static void mono_to_f(const float* acc, float* f) {
        f[0] = 1.0f * acc[0];
        f[1] = 1.0f * acc[2];
        f[2] = 1.0f * acc[3];
        f[3] = 1.0f * acc[1];
    }
    __device__ __forceinline__ static void grad_coeffs(const float* w, float* gq) {
        (void)w; (void)gq;
        gq[0] = 1.0f * w[3];
        gq[1] = 1.0f * w[1];
        gq[2] = 1.0f * w[2];
    }
    template <class Q>
    __device__ __forceinline__ static void grad_eval2(float2 x, float2 y, float2 z, Q&& gq,
                                                      float2* gx, float2* gy, float2* gz) {
        (void)x; (void)y; (void)z; (void)gq; (void)gx; (void)gy; (void)gz;
        gx[0] = gq(0);
        gy[0] = gq(1);
        gz[0] = gq(2);
    }
    __device__ __forceinline__ static void mul(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((0.282094806432724f * a[0] * b[0] + 0.282094806432724f * a[1] * b[1]) + (0.282094806432724f * a[2] * b[2] + 0.282094806432724f * a[3] * b[3]));
        o[1] = 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]);
        o[2] = 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]);
        o[3] = 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]);
    }
    __device__ __forceinline__ static void mul_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((0.282094806432724f * a[0] * b[0] + 0.282094806432724f * a[1] * b[1]) + (0.282094806432724f * a[2] * b[2] + 0.282094806432724f * a[3] * b[3]));
        o[1] = 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]);
        o[2] = 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]);
        o[3] = 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]);
    }
    __device__ __forceinline__ static void mul_onto_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((0.282094806432724f * a[0] * b[0] + 0.282094806432724f * a[1] * b[1]) + (0.282094806432724f * a[2] * b[2] + 0.282094806432724f * a[3] * b[3]));
        o[1] = 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]);
        o[2] = 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]);
        o[3] = 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]);
    }
    __device__ __forceinline__ static void sqr(const float* __restrict__ a, float* __restrict__ o) {
        o[0] = ((0.282094806432724f * a[0] * a[0] + 0.282094806432724f * a[1] * a[1]) + (0.282094806432724f * a[2] * a[2] + 0.282094806432724f * a[3] * a[3]));
        o[1] = 0.564189612865448f * a[0] * a[1];
        o[2] = 0.564189612865448f * a[0] * a[2];
        o[3] = 0.564189612865448f * a[0] * a[3];
    }
};

#if defined(SHS_NB) && SHS_NB == 3
static __constant__ float kExpLeg3[54] = {0.282094806432724f, 0.17650701105594635f, -0.45560693740844727f, 0.17650701105594635f, 0.07128911465406418f, -0.3680286407470703f, 0.5073067545890808f, -0.3680286407470703f, 0.07128911465406418f, 0.282094806432724f, 0.3665502965450287f, -0.3230685591697693f, 0.3665502965450287f, 0.307444304227829f, -0.5419479608535767f, 0.09827397763729095f, -0.5419479608535767f, 0.307444304227829f, 0.282094806432724f, 0.47448834776878357f, -0.11658993363380432f, 0.47448834776878357f, 0.5151698589324951f, -0.2531721591949463f, -0.2615172266960144f, -0.2531721591949463f, 0.5151698589324951f, 0.282094806432724f, 0.47448834776878357f, 0.11658993363380432f, 0.47448834776878357f, 0.5151698589324951f, 0.2531721591949463f, -0.2615172266960144f, 0.2531721591949463f, 0.5151698589324951f, 0.282094806432724f, 0.3665502965450287f, 0.3230685591697693f, 0.3665502965450287f, 0.307444304227829f, 0.5419479608535767f, 0.09827397763729095f, 0.5419479608535767f, 0.307444304227829f, 0.282094806432724f, 0.17650701105594635f, 0.45560693740844727f, 0.17650701105594635f, 0.07128911465406418f, 0.3680286407470703f, 0.5073067545890808f, 0.3680286407470703f, 0.07128911465406418f};
static __constant__ float kExpTrig3[60] = {1.0f, 0.9659258127212524f, 0.258819043636322f, 0.8660253882408142f, 0.5f, 1.0f, 0.7071067690849304f, 0.7071067690849304f, 6.123234262925839e-17f, 1.0f, 1.0f, 0.258819043636322f, 0.9659258127212524f, -0.8660253882408142f, 0.5f, 1.0f, -0.258819043636322f, 0.9659258127212524f, -0.8660253882408142f, -0.5f, 1.0f, -0.7071067690849304f, 0.7071067690849304f, -1.8369701465288538e-16f, -1.0f, 1.0f, -0.9659258127212524f, 0.258819043636322f, 0.8660253882408142f, -0.5f, 1.0f, -0.9659258127212524f, -0.258819043636322f, 0.8660253882408142f, 0.5f, 1.0f, -0.7071067690849304f, -0.7071067690849304f, 1.1943400666719682e-15f, 1.0f, 1.0f, -0.258819043636322f, -0.9659258127212524f, -0.8660253882408142f, 0.5f, 1.0f, 0.258819043636322f, -0.9659258127212524f, -0.8660253882408142f, -0.5f, 1.0f, 0.7071067690849304f, -0.7071067690849304f, -4.2862638516991895e-16f, -1.0f, 1.0f, 0.9659258127212524f, -0.258819043636322f, 0.8660253882408142f, -0.5f};
static __constant__ float kExpW3[6] = {0.08970529586076736f, 0.18889431655406952f, 0.24499917030334473f, 0.24499917030334473f, 0.18889431655406952f, 0.08970529586076736f};
#endif
template <> struct SH<3> {
    static constexpr int K = 9;
    static constexpr int NNZ_SYM = 52;   // entries (i, j <= k)
    static constexpr int EZ = 6;    // projected-exponential rule: Gauss-Legendre nodes
    static constexpr int EP = 12;    // projected-exponential rule: uniform azimuths
#if defined(SHS_NB) && SHS_NB == 3
    __device__ __forceinline__ static const float* eleg() { return kExpLeg3; }
    __device__ __forceinline__ static const float* etrig() { return kExpTrig3; }
    __device__ __forceinline__ static const float* ew() { return kExpW3; }
#endif
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static void ybar(float x, float y, float z, float* Y) {
        (void)x; (void)y; (void)z;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = z * z;
        const float t7 = t6 * 1.5f;
        const float t8 = t7 - 0.5f;
        const float t9 = z * 3.0f;
        const float t10 = t9 * x;
        const float t11 = t9 * y;
        const float t12 = t2 * 3.0f;
        const float t13 = t5 * 3.0f;
        Y[0] = 1.0f;
        Y[1] = y;
        Y[2] = z;
        Y[3] = x;
        Y[4] = t13;
        Y[5] = t11;
        Y[6] = t8;
        Y[7] = t10;
        Y[8] = t12;
    }
    __device__ __forceinline__ static void ybar_vjp(float x, float y, float z, const float* w,
                                                    float& gx, float& gy, float& gz) {
        (void)x; (void)y; (void)z; (void)w;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = z * z;
        const float t7 = t6 * 1.5f;
        const float t8 = t7 - 0.5f;
        const float t9 = z * 3.0f;
        const float t10 = t9 * x;
        const float t11 = t9 * y;
        const float t12 = t2 * 3.0f;
        const float t13 = t5 * 3.0f;
        const float a_t13 = w[4];
        const float a_t12 = w[8];
        const float a_t11 = w[5];
        const float a_t10 = w[7];
        const float a_t9 = y * a_t11 + x * a_t10;
        const float a_t8 = w[6];
        const float a_t7 = a_t8;
        const float a_t6 = 1.5f * a_t7;
        const float a_t5 = 3.0f * a_t13;
        const float a_t4 = a_t5;
        const float a_t3 = a_t5;
        const float a_t2 = 3.0f * a_t12;
        const float a_t1 = -a_t2;
        const float a_t0 = a_t2;
        gx = w[3] + t9 * a_t10 + y * a_t4 + y * a_t3 + x * a_t0 + x * a_t0;
        gy = w[1] + t9 * a_t11 + x * a_t4 + x * a_t3 + y * a_t1 + y * a_t1;
        gz = w[2] + 3.0f * a_t9 + z * a_t6 + z * a_t6;
    }
    static constexpr int NA = 10;   // monomials of degree < n
    static constexpr int NG = 9;   // symmetric tensor entries, bands >= 1
    __device__ __forceinline__ static void accumulate(const float* G, float x, float y, float z, float* acc) {
        (void)x; (void)y; (void)z;
        const float m1_0_0 = x;
        const float m0_1_0 = y;
        const float m0_0_1 = z;
        const float gtx = G[2] * x;
        const float gty = G[2] * y;
        const float gtz = G[2] * z;
        acc[0] = fmaf(G[0], 1.0f, acc[0]);
        acc[1] = fmaf(G[1], m1_0_0, acc[1]);
        acc[2] = fmaf(G[1], m0_1_0, acc[2]);
        acc[3] = fmaf(G[1], m0_0_1, acc[3]);
        acc[4] = fmaf(gtx, m1_0_0, acc[4]);
        acc[5] = fmaf(gtx, m0_1_0, acc[5]);
        acc[6] = fmaf(gtx, m0_0_1, acc[6]);
        acc[7] = fmaf(gty, m0_1_0, acc[7]);
        acc[8] = fmaf(gty, m0_0_1, acc[8]);
        acc[9] = fmaf(gtz, m0_0_1, acc[9]);
    }
    // the same for two pairs at once, one per half of each float2
    __device__ __forceinline__ static void accumulate2(const float2* G, float2 x, float2 y, float2 z,
                                                       float2* acc) {
        (void)x; (void)y; (void)z;
        const float2 m1_0_0 = x;
        const float2 m0_1_0 = y;
        const float2 m0_0_1 = z;
        const float2 gtx = __fmul2_rn(G[2], x);
        const float2 gty = __fmul2_rn(G[2], y);
        const float2 gtz = __fmul2_rn(G[2], z);
        acc[0] = __fadd2_rn(G[0], acc[0]);
        acc[1] = __ffma2_rn(G[1], m1_0_0, acc[1]);
        acc[2] = __ffma2_rn(G[1], m0_1_0, acc[2]);
        acc[3] = __ffma2_rn(G[1], m0_0_1, acc[3]);
        acc[4] = __ffma2_rn(gtx, m1_0_0, acc[4]);
        acc[5] = __ffma2_rn(gtx, m0_1_0, acc[5]);
        acc[6] = __ffma2_rn(gtx, m0_0_1, acc[6]);
        acc[7] = __ffma2_rn(gty, m0_1_0, acc[7]);
        acc[8] = __ffma2_rn(gty, m0_0_1, acc[8]);
        acc[9] = __ffma2_rn(gtz, m0_0_1, acc[9]);
    }
    __device__ __forceinline__ static void mono_to_f(const float* acc, float* f) {
        f[0] = 1.0f * acc[0];
        f[1] = 1.0f * acc[2];
        f[2] = 1.0f * acc[3];
        f[3] = 1.0f * acc[1];
        f[4] = 6.0f * acc[5];
        f[5] = 3.0f * acc[8];
        f[6] = ((1.0f * acc[9] + -0.5f * acc[7]) + -0.5f * acc[4]);
        f[7] = 3.0f * acc[6];
        f[8] = (-3.0f * acc[7] + 3.0f * acc[4]);
    }
    __device__ __forceinline__ static void grad_coeffs(const float* w, float* gq) {
        (void)w; (void)gq;
        gq[0] = 1.0f * w[3];
        gq[1] = 1.0f * w[1];
        gq[2] = 1.0f * w[2];
        gq[3] = (-1.0f * w[6] + 6.0f * w[8]);
        gq[4] = 6.0f * w[4];
        gq[5] = 3.0f * w[7];
        gq[6] = (-1.0f * w[6] + -6.0f * w[8]);
        gq[7] = 3.0f * w[5];
        gq[8] = 2.0f * w[6];
    }
    template <class Q>
    __device__ __forceinline__ static void grad_eval2(float2 x, float2 y, float2 z, Q&& gq,
                                                      float2* gx, float2* gy, float2* gz) {
        (void)x; (void)y; (void)z; (void)gq; (void)gx; (void)gy; (void)gz;
        gx[0] = gq(0);
        gy[0] = gq(1);
        gz[0] = gq(2);
        gx[1] = __ffma2_rn(gq(5), z, __ffma2_rn(gq(4), y, __fmul2_rn(gq(3), x)));
        gy[1] = __ffma2_rn(gq(7), z, __ffma2_rn(gq(6), y, __fmul2_rn(gq(4), x)));
        gz[1] = __ffma2_rn(gq(8), z, __ffma2_rn(gq(7), y, __fmul2_rn(gq(5), x)));
    }
    __device__ __forceinline__ static void mul(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])) + fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])) + (fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]) + fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])));
        o[1] = ((fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])) + -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])) + (-0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]) + 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])));
        o[2] = ((0.282094806432724f * (a[0] * b[2] + a[2] * b[0]) + 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1])) + (0.2523132562637329f * (a[2] * b[6] + a[6] * b[2]) + 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3])));
        o[3] = ((fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])) + 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])) + (0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]) + -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])));
        o[4] = ((0.282094806432724f * (a[0] * b[4] + a[4] * b[0]) + 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])) + (-0.180223748087883f * (a[4] * b[6] + a[6] * b[4]) + 0.15607835352420807f * (a[5] * b[7] + a[7] * b[5])));
        o[5] = ((fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])) + 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1])) + (0.15607835352420807f * (a[4] * b[7] + a[7] * b[4]) + 0.0901118740439415f * (a[5] * b[6] + a[6] * b[5])));
        o[6] = ((fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))) + fmaf(0.0901118740439415f, a[5] * b[5], -0.12615662813186646f * a[1] * b[1])) + (fmaf(0.180223748087883f, a[6] * b[6], 0.2523132562637329f * a[2] * b[2]) + fmaf(0.0901118740439415f, a[7] * b[7], -0.12615662813186646f * a[3] * b[3])));
        o[7] = ((fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])) + 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2])) + (0.15607835352420807f * (a[4] * b[5] + a[5] * b[4]) + 0.0901118740439415f * (a[6] * b[7] + a[7] * b[6])));
        o[8] = ((fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])) + fmaf(0.15607835352420807f, a[7] * b[7], -0.21850968897342682f * a[1] * b[1])) + (0.21850968897342682f * a[3] * b[3] + -0.15607835352420807f * a[5] * b[5]));
    }
    __device__ __forceinline__ static void mul_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])) + fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])) + (fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]) + fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])));
        o[1] = ((fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])) + -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])) + (-0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]) + 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])));
        o[2] = ((0.282094806432724f * (a[0] * b[2] + a[2] * b[0]) + 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1])) + (0.2523132562637329f * (a[2] * b[6] + a[6] * b[2]) + 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3])));
        o[3] = ((fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])) + 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])) + (0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]) + -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])));
        o[4] = ((0.282094806432724f * (a[0] * b[4] + a[4] * b[0]) + 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])) + (-0.180223748087883f * (a[4] * b[6] + a[6] * b[4]) + 0.15607835352420807f * (a[5] * b[7] + a[7] * b[5])));
        o[5] = ((fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])) + 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1])) + (0.15607835352420807f * (a[4] * b[7] + a[7] * b[4]) + 0.0901118740439415f * (a[5] * b[6] + a[6] * b[5])));
        o[6] = ((fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))) + fmaf(0.0901118740439415f, a[5] * b[5], -0.12615662813186646f * a[1] * b[1])) + (fmaf(0.180223748087883f, a[6] * b[6], 0.2523132562637329f * a[2] * b[2]) + fmaf(0.0901118740439415f, a[7] * b[7], -0.12615662813186646f * a[3] * b[3])));
        o[7] = ((fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])) + 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2])) + (0.15607835352420807f * (a[4] * b[5] + a[5] * b[4]) + 0.0901118740439415f * (a[6] * b[7] + a[7] * b[6])));
        o[8] = ((fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])) + fmaf(0.15607835352420807f, a[7] * b[7], -0.21850968897342682f * a[1] * b[1])) + (0.21850968897342682f * a[3] * b[3] + -0.15607835352420807f * a[5] * b[5]));
    }
    __device__ __forceinline__ static void mul_onto_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])) + fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])) + (fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]) + fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])));
        o[1] = ((fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])) + -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])) + (-0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]) + 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])));
        o[2] = ((0.282094806432724f * (a[0] * b[2] + a[2] * b[0]) + 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1])) + (0.2523132562637329f * (a[2] * b[6] + a[6] * b[2]) + 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3])));
        o[3] = ((fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])) + 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])) + (0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]) + -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])));
        o[4] = ((0.282094806432724f * (a[0] * b[4] + a[4] * b[0]) + 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])) + (-0.180223748087883f * (a[4] * b[6] + a[6] * b[4]) + 0.15607835352420807f * (a[5] * b[7] + a[7] * b[5])));
        o[5] = ((fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])) + 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1])) + (0.15607835352420807f * (a[4] * b[7] + a[7] * b[4]) + 0.0901118740439415f * (a[5] * b[6] + a[6] * b[5])));
        o[6] = ((fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))) + fmaf(0.0901118740439415f, a[5] * b[5], -0.12615662813186646f * a[1] * b[1])) + (fmaf(0.180223748087883f, a[6] * b[6], 0.2523132562637329f * a[2] * b[2]) + fmaf(0.0901118740439415f, a[7] * b[7], -0.12615662813186646f * a[3] * b[3])));
        o[7] = ((fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])) + 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2])) + (0.15607835352420807f * (a[4] * b[5] + a[5] * b[4]) + 0.0901118740439415f * (a[6] * b[7] + a[7] * b[6])));
        o[8] = ((fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])) + fmaf(0.15607835352420807f, a[7] * b[7], -0.21850968897342682f * a[1] * b[1])) + (0.21850968897342682f * a[3] * b[3] + -0.15607835352420807f * a[5] * b[5]));
    }
    __device__ __forceinline__ static void sqr(const float* __restrict__ a, float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[8] * a[8], fmaf(0.282094806432724f, a[4] * a[4], 0.282094806432724f * a[0] * a[0])) + fmaf(0.282094806432724f, a[5] * a[5], 0.282094806432724f * a[1] * a[1])) + (fmaf(0.282094806432724f, a[6] * a[6], 0.282094806432724f * a[2] * a[2]) + fmaf(0.282094806432724f, a[7] * a[7], 0.282094806432724f * a[3] * a[3])));
        o[1] = ((fmaf(0.43701937794685364f, a[3] * a[4], 0.564189612865448f * a[0] * a[1]) + -0.2523132562637329f * a[1] * a[6]) + (-0.43701937794685364f * a[1] * a[8] + 0.43701937794685364f * a[2] * a[5]));
        o[2] = ((0.564189612865448f * a[0] * a[2] + 0.43701937794685364f * a[1] * a[5]) + (0.5046265125274658f * a[2] * a[6] + 0.43701937794685364f * a[3] * a[7]));
        o[3] = ((fmaf(0.43701937794685364f, a[3] * a[8], 0.564189612865448f * a[0] * a[3]) + 0.43701937794685364f * a[1] * a[4]) + (0.43701937794685364f * a[2] * a[7] + -0.2523132562637329f * a[3] * a[6]));
        o[4] = ((0.564189612865448f * a[0] * a[4] + 0.43701937794685364f * a[1] * a[3]) + (-0.360447496175766f * a[4] * a[6] + 0.31215670704841614f * a[5] * a[7]));
        o[5] = ((fmaf(-0.31215670704841614f, a[5] * a[8], 0.564189612865448f * a[0] * a[5]) + 0.43701937794685364f * a[1] * a[2]) + (0.31215670704841614f * a[4] * a[7] + 0.180223748087883f * a[5] * a[6]));
        o[6] = ((fmaf(-0.180223748087883f, a[8] * a[8], fmaf(-0.180223748087883f, a[4] * a[4], 0.564189612865448f * a[0] * a[6])) + fmaf(0.0901118740439415f, a[5] * a[5], -0.12615662813186646f * a[1] * a[1])) + (fmaf(0.180223748087883f, a[6] * a[6], 0.2523132562637329f * a[2] * a[2]) + fmaf(0.0901118740439415f, a[7] * a[7], -0.12615662813186646f * a[3] * a[3])));
        o[7] = ((fmaf(0.31215670704841614f, a[7] * a[8], 0.564189612865448f * a[0] * a[7]) + 0.43701937794685364f * a[2] * a[3]) + (0.31215670704841614f * a[4] * a[5] + 0.180223748087883f * a[6] * a[7]));
        o[8] = ((fmaf(-0.360447496175766f, a[6] * a[8], 0.564189612865448f * a[0] * a[8]) + fmaf(0.15607835352420807f, a[7] * a[7], -0.21850968897342682f * a[1] * a[1])) + (0.21850968897342682f * a[3] * a[3] + -0.15607835352420807f * a[5] * a[5]));
    }
};

#if defined(SHS_NB) && SHS_NB == 4
static __constant__ float kExpLeg4[128] = {0.282094806432724f, 0.13632220029830933f, -0.4692000448703766f, 0.13632220029830933f, 0.042523838579654694f, -0.2927210330963135f, 0.5571296811103821f, -0.2927210330963135f, 0.042523838579654694f, 0.012814944609999657f, -0.10803981125354767f, 0.46043887734413147f, -0.5772361159324646f, 0.46043887734413147f, -0.10803981125354767f, 0.012814944609999657f, 0.282094806432724f, 0.2953207194805145f, -0.3892532289028168f, 0.2953207194805145f, 0.19956627488136292f, -0.5260844230651855f, 0.2851242125034332f, -0.5260844230651855f, 0.19956627488136292f, 0.130286306142807f, -0.42064207792282104f, 0.6003922820091248f, -0.05154756084084511f, 0.6003922820091248f, -0.42064207792282104f, 0.130286306142807f, 0.282094806432724f, 0.4156900942325592f, -0.25677645206451416f, 0.4156900942325592f, 0.39540183544158936f, -0.4884883463382721f, -0.05407295748591423f, -0.4884883463382721f, 0.39540183544158936f, 0.3633507788181305f, -0.5497778058052063f, 0.1481184959411621f, 0.3175275921821594f, 0.1481184959411621f, -0.5497778058052063f, 0.3633507788181305f, 0.282094806432724f, 0.48031187057495117f, -0.08962662518024445f, 0.48031187057495117f, 0.5278930068016052f, -0.19701063632965088f, -0.28355443477630615f, -0.19701063632965088f, 0.5278930068016052f, 0.5605146288871765f, -0.25619834661483765f, -0.3737013638019562f, 0.19384369254112244f, -0.3737013638019562f, -0.25619834661483765f, 0.5605146288871765f, 0.282094806432724f, 0.48031187057495117f, 0.08962662518024445f, 0.48031187057495117f, 0.5278930068016052f, 0.19701063632965088f, -0.28355443477630615f, 0.19701063632965088f, 0.5278930068016052f, 0.5605146288871765f, 0.25619834661483765f, -0.3737013638019562f, -0.19384369254112244f, -0.3737013638019562f, 0.25619834661483765f, 0.5605146288871765f, 0.282094806432724f, 0.4156900942325592f, 0.25677645206451416f, 0.4156900942325592f, 0.39540183544158936f, 0.4884883463382721f, -0.05407295748591423f, 0.4884883463382721f, 0.39540183544158936f, 0.3633507788181305f, 0.5497778058052063f, 0.1481184959411621f, -0.3175275921821594f, 0.1481184959411621f, 0.5497778058052063f, 0.3633507788181305f, 0.282094806432724f, 0.2953207194805145f, 0.3892532289028168f, 0.2953207194805145f, 0.19956627488136292f, 0.5260844230651855f, 0.2851242125034332f, 0.5260844230651855f, 0.19956627488136292f, 0.130286306142807f, 0.42064207792282104f, 0.6003922820091248f, 0.05154756084084511f, 0.6003922820091248f, 0.42064207792282104f, 0.130286306142807f, 0.282094806432724f, 0.13632220029830933f, 0.4692000448703766f, 0.13632220029830933f, 0.042523838579654694f, 0.2927210330963135f, 0.5571296811103821f, 0.2927210330963135f, 0.042523838579654694f, 0.012814944609999657f, 0.10803981125354767f, 0.46043887734413147f, 0.5772361159324646f, 0.46043887734413147f, 0.10803981125354767f, 0.012814944609999657f};
static __constant__ float kExpTrig4[112] = {1.0f, 0.9807852506637573f, 0.19509032368659973f, 0.9238795042037964f, 0.3826834261417389f, 0.8314695954322815f, 0.5555702447891235f, 1.0f, 0.8314695954322815f, 0.5555702447891235f, 0.3826834261417389f, 0.9238795042037964f, -0.19509032368659973f, 0.9807852506637573f, 1.0f, 0.5555702447891235f, 0.8314695954322815f, -0.3826834261417389f, 0.9238795042037964f, -0.9807852506637573f, 0.19509032368659973f, 1.0f, 0.19509032368659973f, 0.9807852506637573f, -0.9238795042037964f, 0.3826834261417389f, -0.5555702447891235f, -0.8314695954322815f, 1.0f, -0.19509032368659973f, 0.9807852506637573f, -0.9238795042037964f, -0.3826834261417389f, 0.5555702447891235f, -0.8314695954322815f, 1.0f, -0.5555702447891235f, 0.8314695954322815f, -0.3826834261417389f, -0.9238795042037964f, 0.9807852506637573f, 0.19509032368659973f, 1.0f, -0.8314695954322815f, 0.5555702447891235f, 0.3826834261417389f, -0.9238795042037964f, 0.19509032368659973f, 0.9807852506637573f, 1.0f, -0.9807852506637573f, 0.19509032368659973f, 0.9238795042037964f, -0.3826834261417389f, -0.8314695954322815f, 0.5555702447891235f, 1.0f, -0.9807852506637573f, -0.19509032368659973f, 0.9238795042037964f, 0.3826834261417389f, -0.8314695954322815f, -0.5555702447891235f, 1.0f, -0.8314695954322815f, -0.5555702447891235f, 0.3826834261417389f, 0.9238795042037964f, 0.19509032368659973f, -0.9807852506637573f, 1.0f, -0.5555702447891235f, -0.8314695954322815f, -0.3826834261417389f, 0.9238795042037964f, 0.9807852506637573f, -0.19509032368659973f, 1.0f, -0.19509032368659973f, -0.9807852506637573f, -0.9238795042037964f, 0.3826834261417389f, 0.5555702447891235f, 0.8314695954322815f, 1.0f, 0.19509032368659973f, -0.9807852506637573f, -0.9238795042037964f, -0.3826834261417389f, -0.5555702447891235f, 0.8314695954322815f, 1.0f, 0.5555702447891235f, -0.8314695954322815f, -0.3826834261417389f, -0.9238795042037964f, -0.9807852506637573f, -0.19509032368659973f, 1.0f, 0.8314695954322815f, -0.5555702447891235f, 0.3826834261417389f, -0.9238795042037964f, -0.19509032368659973f, -0.9807852506637573f, 1.0f, 0.9807852506637573f, -0.19509032368659973f, 0.9238795042037964f, -0.3826834261417389f, 0.8314695954322815f, -0.5555702447891235f};
static __constant__ float kExpW4[8] = {0.039752352982759476f, 0.08732882887125015f, 0.12319231033325195f, 0.14242558181285858f, 0.14242558181285858f, 0.12319231033325195f, 0.08732882887125015f, 0.039752352982759476f};
#endif
template <> struct SH<4> {
    static constexpr int K = 16;
    static constexpr int NNZ_SYM = 194;   // entries (i, j <= k)
    static constexpr int EZ = 8;    // projected-exponential rule: Gauss-Legendre nodes
    static constexpr int EP = 16;    // projected-exponential rule: uniform azimuths
#if defined(SHS_NB) && SHS_NB == 4
    __device__ __forceinline__ static const float* eleg() { return kExpLeg4; }
    __device__ __forceinline__ static const float* etrig() { return kExpTrig4; }
    __device__ __forceinline__ static const float* ew() { return kExpW4; }
#endif
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            case 9: return 0.03933623805642128f;
            case 10: return 0.09635371714830399f;
            case 11: return 0.304697185754776f;
            case 12: return 0.7463526725769043f;
            case 13: return 0.304697185754776f;
            case 14: return 0.09635371714830399f;
            case 15: return 0.03933623805642128f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            case 3: return 0.0f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static void ybar(float x, float y, float z, float* Y) {
        (void)x; (void)y; (void)z;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = x * t2;
        const float t7 = y * t5;
        const float t8 = t6 - t7;
        const float t9 = x * t5;
        const float t10 = y * t2;
        const float t11 = t9 + t10;
        const float t12 = z * z;
        const float t13 = t12 * 1.5f;
        const float t14 = t13 - 0.5f;
        const float t15 = z * t14;
        const float t16 = t15 * 1.6666666269302368f;
        const float t17 = z * 0.6666666865348816f;
        const float t18 = t16 - t17;
        const float t19 = z * 3.0f;
        const float t20 = z * t19;
        const float t21 = t20 * 2.5f;
        const float t22 = t21 - 1.5f;
        const float t23 = z * 3.0f;
        const float t24 = t23 * 5.0f;
        const float t25 = t19 * x;
        const float t26 = t19 * y;
        const float t27 = t2 * 3.0f;
        const float t28 = t5 * 3.0f;
        const float t29 = t22 * x;
        const float t30 = t22 * y;
        const float t31 = t24 * t2;
        const float t32 = t24 * t5;
        const float t33 = t8 * 15.0f;
        const float t34 = t11 * 15.0f;
        Y[0] = 1.0f;
        Y[1] = y;
        Y[2] = z;
        Y[3] = x;
        Y[4] = t28;
        Y[5] = t26;
        Y[6] = t14;
        Y[7] = t25;
        Y[8] = t27;
        Y[9] = t34;
        Y[10] = t32;
        Y[11] = t30;
        Y[12] = t18;
        Y[13] = t29;
        Y[14] = t31;
        Y[15] = t33;
    }
    __device__ __forceinline__ static void ybar_vjp(float x, float y, float z, const float* w,
                                                    float& gx, float& gy, float& gz) {
        (void)x; (void)y; (void)z; (void)w;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = x * t2;
        const float t7 = y * t5;
        const float t8 = t6 - t7;
        const float t9 = x * t5;
        const float t10 = y * t2;
        const float t11 = t9 + t10;
        const float t12 = z * z;
        const float t13 = t12 * 1.5f;
        const float t14 = t13 - 0.5f;
        const float t15 = z * t14;
        const float t16 = t15 * 1.6666666269302368f;
        const float t17 = z * 0.6666666865348816f;
        const float t18 = t16 - t17;
        const float t19 = z * 3.0f;
        const float t20 = z * t19;
        const float t21 = t20 * 2.5f;
        const float t22 = t21 - 1.5f;
        const float t23 = z * 3.0f;
        const float t24 = t23 * 5.0f;
        const float t25 = t19 * x;
        const float t26 = t19 * y;
        const float t27 = t2 * 3.0f;
        const float t28 = t5 * 3.0f;
        const float t29 = t22 * x;
        const float t30 = t22 * y;
        const float t31 = t24 * t2;
        const float t32 = t24 * t5;
        const float t33 = t8 * 15.0f;
        const float t34 = t11 * 15.0f;
        const float a_t34 = w[9];
        const float a_t33 = w[15];
        const float a_t32 = w[10];
        const float a_t31 = w[14];
        const float a_t30 = w[11];
        const float a_t29 = w[13];
        const float a_t28 = w[4];
        const float a_t27 = w[8];
        const float a_t26 = w[5];
        const float a_t25 = w[7];
        const float a_t24 = t5 * a_t32 + t2 * a_t31;
        const float a_t23 = 5.0f * a_t24;
        const float a_t22 = y * a_t30 + x * a_t29;
        const float a_t21 = a_t22;
        const float a_t20 = 2.5f * a_t21;
        const float a_t19 = y * a_t26 + x * a_t25 + z * a_t20;
        const float a_t18 = w[12];
        const float a_t17 = -a_t18;
        const float a_t16 = a_t18;
        const float a_t15 = 1.6666666269302368f * a_t16;
        const float a_t14 = w[6] + z * a_t15;
        const float a_t13 = a_t14;
        const float a_t12 = 1.5f * a_t13;
        const float a_t11 = 15.0f * a_t34;
        const float a_t10 = a_t11;
        const float a_t9 = a_t11;
        const float a_t8 = 15.0f * a_t33;
        const float a_t7 = -a_t8;
        const float a_t6 = a_t8;
        const float a_t5 = t24 * a_t32 + 3.0f * a_t28 + x * a_t9 + y * a_t7;
        const float a_t4 = a_t5;
        const float a_t3 = a_t5;
        const float a_t2 = t24 * a_t31 + 3.0f * a_t27 + y * a_t10 + x * a_t6;
        const float a_t1 = -a_t2;
        const float a_t0 = a_t2;
        gx = w[3] + t22 * a_t29 + t19 * a_t25 + t5 * a_t9 + t2 * a_t6 + y * a_t4 + y * a_t3 + x * a_t0 + x * a_t0;
        gy = w[1] + t22 * a_t30 + t19 * a_t26 + t2 * a_t10 + t5 * a_t7 + x * a_t4 + x * a_t3 + y * a_t1 + y * a_t1;
        gz = w[2] + 3.0f * a_t23 + t19 * a_t20 + 3.0f * a_t19 + 0.6666666865348816f * a_t17 + t14 * a_t15 + z * a_t12 + z * a_t12;
    }
    static constexpr int NA = 20;   // monomials of degree < n
    static constexpr int NG = 19;   // symmetric tensor entries, bands >= 1
    __device__ __forceinline__ static void accumulate(const float* G, float x, float y, float z, float* acc) {
        (void)x; (void)y; (void)z;
        const float m1_0_0 = x;
        const float m0_1_0 = y;
        const float m0_0_1 = z;
        const float m2_0_0 = x * m1_0_0;
        const float m1_1_0 = x * m0_1_0;
        const float m1_0_1 = x * m0_0_1;
        const float m0_2_0 = y * m0_1_0;
        const float m0_1_1 = y * m0_0_1;
        const float m0_0_2 = z * m0_0_1;
        const float gtx = G[3] * x;
        const float gty = G[3] * y;
        const float gtz = G[3] * z;
        acc[0] = fmaf(G[0], 1.0f, acc[0]);
        acc[1] = fmaf(G[1], m1_0_0, acc[1]);
        acc[2] = fmaf(G[1], m0_1_0, acc[2]);
        acc[3] = fmaf(G[1], m0_0_1, acc[3]);
        acc[4] = fmaf(G[2], m2_0_0, acc[4]);
        acc[5] = fmaf(G[2], m1_1_0, acc[5]);
        acc[6] = fmaf(G[2], m1_0_1, acc[6]);
        acc[7] = fmaf(G[2], m0_2_0, acc[7]);
        acc[8] = fmaf(G[2], m0_1_1, acc[8]);
        acc[9] = fmaf(G[2], m0_0_2, acc[9]);
        acc[10] = fmaf(gtx, m2_0_0, acc[10]);
        acc[11] = fmaf(gtx, m1_1_0, acc[11]);
        acc[12] = fmaf(gtx, m1_0_1, acc[12]);
        acc[13] = fmaf(gtx, m0_2_0, acc[13]);
        acc[14] = fmaf(gtx, m0_1_1, acc[14]);
        acc[15] = fmaf(gtx, m0_0_2, acc[15]);
        acc[16] = fmaf(gty, m0_2_0, acc[16]);
        acc[17] = fmaf(gty, m0_1_1, acc[17]);
        acc[18] = fmaf(gty, m0_0_2, acc[18]);
        acc[19] = fmaf(gtz, m0_0_2, acc[19]);
    }
    // the same for two pairs at once, one per half of each float2
    __device__ __forceinline__ static void accumulate2(const float2* G, float2 x, float2 y, float2 z,
                                                       float2* acc) {
        (void)x; (void)y; (void)z;
        const float2 m1_0_0 = x;
        const float2 m0_1_0 = y;
        const float2 m0_0_1 = z;
        const float2 m2_0_0 = __fmul2_rn(x, m1_0_0);
        const float2 m1_1_0 = __fmul2_rn(x, m0_1_0);
        const float2 m1_0_1 = __fmul2_rn(x, m0_0_1);
        const float2 m0_2_0 = __fmul2_rn(y, m0_1_0);
        const float2 m0_1_1 = __fmul2_rn(y, m0_0_1);
        const float2 m0_0_2 = __fmul2_rn(z, m0_0_1);
        const float2 gtx = __fmul2_rn(G[3], x);
        const float2 gty = __fmul2_rn(G[3], y);
        const float2 gtz = __fmul2_rn(G[3], z);
        acc[0] = __fadd2_rn(G[0], acc[0]);
        acc[1] = __ffma2_rn(G[1], m1_0_0, acc[1]);
        acc[2] = __ffma2_rn(G[1], m0_1_0, acc[2]);
        acc[3] = __ffma2_rn(G[1], m0_0_1, acc[3]);
        acc[4] = __ffma2_rn(G[2], m2_0_0, acc[4]);
        acc[5] = __ffma2_rn(G[2], m1_1_0, acc[5]);
        acc[6] = __ffma2_rn(G[2], m1_0_1, acc[6]);
        acc[7] = __ffma2_rn(G[2], m0_2_0, acc[7]);
        acc[8] = __ffma2_rn(G[2], m0_1_1, acc[8]);
        acc[9] = __ffma2_rn(G[2], m0_0_2, acc[9]);
        acc[10] = __ffma2_rn(gtx, m2_0_0, acc[10]);
        acc[11] = __ffma2_rn(gtx, m1_1_0, acc[11]);
        acc[12] = __ffma2_rn(gtx, m1_0_1, acc[12]);
        acc[13] = __ffma2_rn(gtx, m0_2_0, acc[13]);
        acc[14] = __ffma2_rn(gtx, m0_1_1, acc[14]);
        acc[15] = __ffma2_rn(gtx, m0_0_2, acc[15]);
        acc[16] = __ffma2_rn(gty, m0_2_0, acc[16]);
        acc[17] = __ffma2_rn(gty, m0_1_1, acc[17]);
        acc[18] = __ffma2_rn(gty, m0_0_2, acc[18]);
        acc[19] = __ffma2_rn(gtz, m0_0_2, acc[19]);
    }
    __device__ __forceinline__ static void mono_to_f(const float* acc, float* f) {
        f[0] = 1.0f * acc[0];
        f[1] = 1.0f * acc[2];
        f[2] = 1.0f * acc[3];
        f[3] = 1.0f * acc[1];
        f[4] = 6.0f * acc[5];
        f[5] = 3.0f * acc[8];
        f[6] = ((1.0f * acc[9] + -0.5f * acc[7]) + -0.5f * acc[4]);
        f[7] = 3.0f * acc[6];
        f[8] = (-3.0f * acc[7] + 3.0f * acc[4]);
        f[9] = (-15.0f * acc[16] + 45.0f * acc[11]);
        f[10] = 30.0f * acc[14];
        f[11] = ((6.0f * acc[18] + -1.5f * acc[16]) + -1.5f * acc[11]);
        f[12] = ((1.0f * acc[19] + -1.5f * acc[17]) + -1.5f * acc[12]);
        f[13] = ((6.0f * acc[15] + -1.5f * acc[13]) + -1.5f * acc[10]);
        f[14] = (-15.0f * acc[17] + 15.0f * acc[12]);
        f[15] = (-45.0f * acc[13] + 15.0f * acc[10]);
    }
    __device__ __forceinline__ static void grad_coeffs(const float* w, float* gq) {
        (void)w; (void)gq;
        gq[0] = 1.0f * w[3];
        gq[1] = 1.0f * w[1];
        gq[2] = 1.0f * w[2];
        gq[3] = (-1.0f * w[6] + 6.0f * w[8]);
        gq[4] = 6.0f * w[4];
        gq[5] = 3.0f * w[7];
        gq[6] = (-1.0f * w[6] + -6.0f * w[8]);
        gq[7] = 3.0f * w[5];
        gq[8] = 2.0f * w[6];
        gq[9] = (-4.5f * w[13] + 45.0f * w[15]);
        gq[10] = (45.0f * w[9] + -1.5f * w[11]);
        gq[11] = (-1.5f * w[12] + 15.0f * w[14]);
        gq[12] = (-1.5f * w[13] + -45.0f * w[15]);
        gq[13] = 15.0f * w[10];
        gq[14] = 6.0f * w[13];
        gq[15] = (-45.0f * w[9] + -4.5f * w[11]);
        gq[16] = (-1.5f * w[12] + -15.0f * w[14]);
        gq[17] = 6.0f * w[11];
        gq[18] = 3.0f * w[12];
    }
    template <class Q>
    __device__ __forceinline__ static void grad_eval2(float2 x, float2 y, float2 z, Q&& gq,
                                                      float2* gx, float2* gy, float2* gz) {
        (void)x; (void)y; (void)z; (void)gq; (void)gx; (void)gy; (void)gz;
        const float2 x2 = __fmul2_rn(make_float2(2.0f, 2.0f), x);
        const float2 y2 = __fmul2_rn(make_float2(2.0f, 2.0f), y);
        const float2 z2 = __fmul2_rn(make_float2(2.0f, 2.0f), z);
        const float2 u2_0_0 = __fmul2_rn(x, x);
        const float2 u1_1_0 = __fmul2_rn(y, x2);
        const float2 u1_0_1 = __fmul2_rn(z, x2);
        const float2 u0_2_0 = __fmul2_rn(y, y);
        const float2 u0_1_1 = __fmul2_rn(z, y2);
        const float2 u0_0_2 = __fmul2_rn(z, z);
        gx[0] = gq(0);
        gy[0] = gq(1);
        gz[0] = gq(2);
        gx[1] = __ffma2_rn(gq(5), z, __ffma2_rn(gq(4), y, __fmul2_rn(gq(3), x)));
        gy[1] = __ffma2_rn(gq(7), z, __ffma2_rn(gq(6), y, __fmul2_rn(gq(4), x)));
        gz[1] = __ffma2_rn(gq(8), z, __ffma2_rn(gq(7), y, __fmul2_rn(gq(5), x)));
        gx[2] = __ffma2_rn(gq(14), u0_0_2, __ffma2_rn(gq(13), u0_1_1, __ffma2_rn(gq(12), u0_2_0, __ffma2_rn(gq(11), u1_0_1, __ffma2_rn(gq(10), u1_1_0, __fmul2_rn(gq(9), u2_0_0))))));
        gy[2] = __ffma2_rn(gq(17), u0_0_2, __ffma2_rn(gq(16), u0_1_1, __ffma2_rn(gq(15), u0_2_0, __ffma2_rn(gq(13), u1_0_1, __ffma2_rn(gq(12), u1_1_0, __fmul2_rn(gq(10), u2_0_0))))));
        gz[2] = __ffma2_rn(gq(18), u0_0_2, __ffma2_rn(gq(17), u0_1_1, __ffma2_rn(gq(16), u0_2_0, __ffma2_rn(gq(14), u1_0_1, __ffma2_rn(gq(13), u1_1_0, __fmul2_rn(gq(11), u2_0_0))))));
    }
    __device__ __forceinline__ static void mul(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[12] * b[12], fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0]))) + fmaf(0.282094806432724f, a[13] * b[13], fmaf(0.282094806432724f, a[9] * b[9], fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])))) + (fmaf(0.282094806432724f, a[14] * b[14], fmaf(0.282094806432724f, a[10] * b[10], fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]))) + fmaf(0.282094806432724f, a[15] * b[15], fmaf(0.282094806432724f, a[11] * b[11], fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])))));
        o[1] = ((fmaf(0.05839917063713074f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.18467439711093903f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])))) + fmaf(0.20230065286159515f, (a[6] * b[11] + a[11] * b[6]), fmaf(-0.05839917063713074f, (a[4] * b[13] + a[13] * b[4]), -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])))) + (fmaf(0.18467439711093903f, (a[7] * b[10] + a[10] * b[7]), fmaf(-0.22617901861667633f, (a[4] * b[15] + a[15] * b[4]), -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]))) + fmaf(0.22617901861667633f, (a[8] * b[9] + a[9] * b[8]), fmaf(-0.14304816722869873f, (a[5] * b[12] + a[12] * b[5]), 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])))));
        o[2] = ((fmaf(0.18467439711093903f, (a[8] * b[14] + a[14] * b[8]), fmaf(0.18467439711093903f, (a[4] * b[10] + a[10] * b[4]), 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]))) + fmaf(0.23359668254852295f, (a[5] * b[11] + a[11] * b[5]), 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.24776668846607208f, (a[6] * b[12] + a[12] * b[6]), 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])) + fmaf(0.23359668254852295f, (a[7] * b[13] + a[13] * b[7]), 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))));
        o[3] = ((fmaf(0.22617901861667633f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.20230065286159515f, (a[6] * b[13] + a[13] * b[6]), fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])))) + fmaf(-0.14304816722869873f, (a[7] * b[12] + a[12] * b[7]), fmaf(0.22617901861667633f, (a[4] * b[9] + a[9] * b[4]), 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])))) + (fmaf(0.18467439711093903f, (a[7] * b[14] + a[14] * b[7]), fmaf(-0.05839917063713074f, (a[4] * b[11] + a[11] * b[4]), 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]))) + fmaf(-0.05839917063713074f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.18467439711093903f, (a[5] * b[10] + a[10] * b[5]), -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])))));
        o[4] = ((fmaf(0.09403159469366074f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.18467439711093903f, (a[2] * b[10] + a[10] * b[2]), 0.282094806432724f * (a[0] * b[4] + a[4] * b[0])))) + fmaf(-0.09403159469366074f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.22617901861667633f, (a[3] * b[9] + a[9] * b[3]), 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])))) + (fmaf(-0.18806318938732147f, (a[10] * b[12] + a[12] * b[10]), fmaf(-0.05839917063713074f, (a[3] * b[11] + a[11] * b[3]), -0.05839917063713074f * (a[1] * b[13] + a[13] * b[1]))) + fmaf(0.14567312598228455f, (a[11] * b[13] + a[13] * b[11]), fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * (a[1] * b[15] + a[15] * b[1])))));
        o[5] = ((fmaf(0.059470802545547485f, (a[11] * b[12] + a[12] * b[11]), fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.23359668254852295f, (a[2] * b[11] + a[11] * b[2]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])))) + fmaf(-0.11516471952199936f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.1486770063638687f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.18467439711093903f, (a[3] * b[10] + a[10] * b[3]), 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1]))))) + (fmaf(0.11516471952199936f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * (a[1] * b[12] + a[12] * b[1]))) + fmaf(-0.1486770063638687f, (a[10] * b[15] + a[15] * b[10]), fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), -0.18467439711093903f * (a[1] * b[14] + a[14] * b[1])))));
        o[6] = ((fmaf(-0.2102610468864441f, a[15] * b[15], fmaf(-0.2102610468864441f, a[9] * b[9], fmaf(0.0901118740439415f, a[5] * b[5], fmaf(0.24776668846607208f, (a[2] * b[12] + a[12] * b[2]), 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))))) + fmaf(0.12615662813186646f, a[11] * b[11], fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1])))) + (fmaf(0.16820883750915527f, a[12] * b[12], fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.20230065286159515f, (a[3] * b[13] + a[13] * b[3]), 0.20230065286159515f * (a[1] * b[11] + a[11] * b[1])))) + fmaf(0.12615662813186646f, a[13] * b[13], fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2])))));
        o[7] = ((fmaf(0.11516471952199936f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.14304816722869873f, (a[3] * b[12] + a[12] * b[3]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])))) + fmaf(0.1486770063638687f, (a[14] * b[15] + a[15] * b[14]), fmaf(0.1486770063638687f, (a[9] * b[10] + a[10] * b[9]), fmaf(0.18467439711093903f, (a[3] * b[14] + a[14] * b[3]), 0.18467439711093903f * (a[1] * b[10] + a[10] * b[1]))))) + (fmaf(0.11516471952199936f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2]))) + fmaf(0.059470802545547485f, (a[12] * b[13] + a[13] * b[12]), fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), 0.23359668254852295f * (a[2] * b[13] + a[13] * b[2])))));
        o[8] = ((fmaf(-0.14567312598228455f, a[11] * b[11], fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.18467439711093903f, (a[2] * b[14] + a[14] * b[2]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])))) + fmaf(-0.18806318938732147f, (a[12] * b[14] + a[14] * b[12]), fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1])))) + (fmaf(0.14567312598228455f, a[13] * b[13], fmaf(0.15607835352420807f, a[7] * b[7], fmaf(-0.05839917063713074f, (a[3] * b[13] + a[13] * b[3]), 0.22617901861667633f * (a[1] * b[9] + a[9] * b[1])))) + fmaf(-0.09403159469366074f, (a[13] * b[15] + a[15] * b[13]), fmaf(-0.09403159469366074f, (a[9] * b[11] + a[11] * b[9]), fmaf(0.22617901861667633f, (a[3] * b[15] + a[15] * b[3]), 0.05839917063713074f * (a[1] * b[11] + a[11] * b[1]))))));
        o[9] = ((fmaf(0.1486770063638687f, (a[5] * b[14] + a[14] * b[5]), 0.282094806432724f * (a[0] * b[9] + a[9] * b[0])) + fmaf(-0.2102610468864441f, (a[6] * b[9] + a[9] * b[6]), 0.22617901861667633f * (a[1] * b[8] + a[8] * b[1]))) + (fmaf(0.1486770063638687f, (a[7] * b[10] + a[10] * b[7]), 0.22617901861667633f * (a[3] * b[4] + a[4] * b[3])) + fmaf(-0.09403159469366074f, (a[8] * b[11] + a[11] * b[8]), -0.09403159469366074f * (a[4] * b[13] + a[13] * b[4]))));
        o[10] = ((fmaf(0.11516471952199936f, (a[7] * b[11] + a[11] * b[7]), fmaf(-0.18806318938732147f, (a[4] * b[12] + a[12] * b[4]), 0.282094806432724f * (a[0] * b[10] + a[10] * b[0]))) + fmaf(0.11516471952199936f, (a[5] * b[13] + a[13] * b[5]), 0.18467439711093903f * (a[1] * b[7] + a[7] * b[1]))) + (fmaf(-0.1486770063638687f, (a[5] * b[15] + a[15] * b[5]), 0.18467439711093903f * (a[2] * b[4] + a[4] * b[2])) + fmaf(0.1486770063638687f, (a[7] * b[9] + a[9] * b[7]), 0.18467439711093903f * (a[3] * b[5] + a[5] * b[3]))));
        o[11] = ((fmaf(-0.14567312598228455f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.11516471952199936f, (a[5] * b[14] + a[14] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[11] + a[11] * b[0])))) + fmaf(0.12615662813186646f, (a[6] * b[11] + a[11] * b[6]), fmaf(0.14567312598228455f, (a[4] * b[13] + a[13] * b[4]), 0.20230065286159515f * (a[1] * b[6] + a[6] * b[1])))) + (fmaf(0.11516471952199936f, (a[7] * b[10] + a[10] * b[7]), fmaf(0.09403159469366074f, (a[4] * b[15] + a[15] * b[4]), 0.05839917063713074f * (a[1] * b[8] + a[8] * b[1]))) + fmaf(-0.09403159469366074f, (a[8] * b[9] + a[9] * b[8]), fmaf(0.059470802545547485f, (a[5] * b[12] + a[12] * b[5]), 0.23359668254852295f * (a[2] * b[5] + a[5] * b[2])))));
        o[12] = ((fmaf(-0.18806318938732147f, (a[8] * b[14] + a[14] * b[8]), fmaf(-0.18806318938732147f, (a[4] * b[10] + a[10] * b[4]), 0.282094806432724f * (a[0] * b[12] + a[12] * b[0]))) + fmaf(0.059470802545547485f, (a[5] * b[11] + a[11] * b[5]), -0.14304816722869873f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.16820883750915527f, (a[6] * b[12] + a[12] * b[6]), 0.24776668846607208f * (a[2] * b[6] + a[6] * b[2])) + fmaf(0.059470802545547485f, (a[7] * b[13] + a[13] * b[7]), -0.14304816722869873f * (a[3] * b[7] + a[7] * b[3]))));
        o[13] = ((fmaf(-0.09403159469366074f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.12615662813186646f, (a[6] * b[13] + a[13] * b[6]), fmaf(-0.05839917063713074f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[13] + a[13] * b[0])))) + fmaf(0.059470802545547485f, (a[7] * b[12] + a[12] * b[7]), fmaf(-0.09403159469366074f, (a[4] * b[9] + a[9] * b[4]), -0.05839917063713074f * (a[1] * b[4] + a[4] * b[1])))) + (fmaf(0.11516471952199936f, (a[7] * b[14] + a[14] * b[7]), fmaf(0.14567312598228455f, (a[4] * b[11] + a[11] * b[4]), 0.23359668254852295f * (a[2] * b[7] + a[7] * b[2]))) + fmaf(0.14567312598228455f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.11516471952199936f, (a[5] * b[10] + a[10] * b[5]), 0.20230065286159515f * (a[3] * b[6] + a[6] * b[3])))));
        o[14] = ((fmaf(-0.18806318938732147f, (a[8] * b[12] + a[12] * b[8]), fmaf(0.1486770063638687f, (a[5] * b[9] + a[9] * b[5]), 0.282094806432724f * (a[0] * b[14] + a[14] * b[0]))) + fmaf(-0.11516471952199936f, (a[5] * b[11] + a[11] * b[5]), -0.18467439711093903f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.11516471952199936f, (a[7] * b[13] + a[13] * b[7]), 0.18467439711093903f * (a[2] * b[8] + a[8] * b[2])) + fmaf(0.1486770063638687f, (a[7] * b[15] + a[15] * b[7]), 0.18467439711093903f * (a[3] * b[7] + a[7] * b[3]))));
        o[15] = ((fmaf(-0.1486770063638687f, (a[5] * b[10] + a[10] * b[5]), 0.282094806432724f * (a[0] * b[15] + a[15] * b[0])) + fmaf(-0.2102610468864441f, (a[6] * b[15] + a[15] * b[6]), -0.22617901861667633f * (a[1] * b[4] + a[4] * b[1]))) + (fmaf(0.1486770063638687f, (a[7] * b[14] + a[14] * b[7]), 0.22617901861667633f * (a[3] * b[8] + a[8] * b[3])) + fmaf(-0.09403159469366074f, (a[8] * b[13] + a[13] * b[8]), 0.09403159469366074f * (a[4] * b[11] + a[11] * b[4]))));
    }
    __device__ __forceinline__ static void mul_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])) + fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])) + (fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]) + fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])));
        o[1] = ((fmaf(0.05839917063713074f, a[11] * b[8], fmaf(-0.18467439711093903f, a[14] * b[5], fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])))) + fmaf(0.20230065286159515f, a[11] * b[6], fmaf(-0.05839917063713074f, a[13] * b[4], -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])))) + (fmaf(0.18467439711093903f, a[10] * b[7], fmaf(-0.22617901861667633f, a[15] * b[4], -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]))) + fmaf(0.22617901861667633f, a[9] * b[8], fmaf(-0.14304816722869873f, a[12] * b[5], 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])))));
        o[2] = ((fmaf(0.18467439711093903f, a[14] * b[8], fmaf(0.18467439711093903f, a[10] * b[4], 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]))) + fmaf(0.23359668254852295f, a[11] * b[5], 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.24776668846607208f, a[12] * b[6], 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])) + fmaf(0.23359668254852295f, a[13] * b[7], 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))));
        o[3] = ((fmaf(0.22617901861667633f, a[15] * b[8], fmaf(0.20230065286159515f, a[13] * b[6], fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])))) + fmaf(-0.14304816722869873f, a[12] * b[7], fmaf(0.22617901861667633f, a[9] * b[4], 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])))) + (fmaf(0.18467439711093903f, a[14] * b[7], fmaf(-0.05839917063713074f, a[11] * b[4], 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]))) + fmaf(-0.05839917063713074f, a[13] * b[8], fmaf(0.18467439711093903f, a[10] * b[5], -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])))));
        o[4] = ((fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.18467439711093903f, a[10] * b[2], 0.282094806432724f * (a[0] * b[4] + a[4] * b[0]))) + fmaf(0.22617901861667633f, a[9] * b[3], 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1]))) + (fmaf(-0.05839917063713074f, a[11] * b[3], -0.05839917063713074f * a[13] * b[1]) + fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * a[15] * b[1])));
        o[5] = ((fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.23359668254852295f, a[11] * b[2], 0.282094806432724f * (a[0] * b[5] + a[5] * b[0]))) + fmaf(0.18467439711093903f, a[10] * b[3], 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1]))) + (fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * a[12] * b[1]) + fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), -0.18467439711093903f * a[14] * b[1])));
        o[6] = ((fmaf(0.0901118740439415f, a[5] * b[5], fmaf(0.24776668846607208f, a[12] * b[2], 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))) + fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1]))) + (fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.20230065286159515f, a[13] * b[3], 0.20230065286159515f * a[11] * b[1])) + fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2]))));
        o[7] = ((fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.14304816722869873f, a[12] * b[3], 0.282094806432724f * (a[0] * b[7] + a[7] * b[0]))) + fmaf(0.18467439711093903f, a[14] * b[3], 0.18467439711093903f * a[10] * b[1])) + (fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2])) + fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), 0.23359668254852295f * a[13] * b[2])));
        o[8] = ((fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.18467439711093903f, a[14] * b[2], 0.282094806432724f * (a[0] * b[8] + a[8] * b[0]))) + fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1]))) + (fmaf(0.15607835352420807f, a[7] * b[7], fmaf(-0.05839917063713074f, a[13] * b[3], 0.22617901861667633f * a[9] * b[1])) + fmaf(0.22617901861667633f, a[15] * b[3], 0.05839917063713074f * a[11] * b[1])));
        o[9] = ((fmaf(0.1486770063638687f, a[14] * b[5], 0.282094806432724f * a[9] * b[0]) + fmaf(-0.2102610468864441f, a[9] * b[6], 0.22617901861667633f * (a[1] * b[8] + a[8] * b[1]))) + (fmaf(0.1486770063638687f, a[10] * b[7], 0.22617901861667633f * (a[3] * b[4] + a[4] * b[3])) + fmaf(-0.09403159469366074f, a[11] * b[8], -0.09403159469366074f * a[13] * b[4])));
        o[10] = ((fmaf(0.11516471952199936f, a[11] * b[7], fmaf(-0.18806318938732147f, a[12] * b[4], 0.282094806432724f * a[10] * b[0])) + fmaf(0.11516471952199936f, a[13] * b[5], 0.18467439711093903f * (a[1] * b[7] + a[7] * b[1]))) + (fmaf(-0.1486770063638687f, a[15] * b[5], 0.18467439711093903f * (a[2] * b[4] + a[4] * b[2])) + fmaf(0.1486770063638687f, a[9] * b[7], 0.18467439711093903f * (a[3] * b[5] + a[5] * b[3]))));
        o[11] = ((fmaf(-0.14567312598228455f, a[11] * b[8], fmaf(-0.11516471952199936f, a[14] * b[5], fmaf(-0.05839917063713074f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * a[11] * b[0]))) + fmaf(0.12615662813186646f, a[11] * b[6], fmaf(0.14567312598228455f, a[13] * b[4], 0.20230065286159515f * (a[1] * b[6] + a[6] * b[1])))) + (fmaf(0.11516471952199936f, a[10] * b[7], fmaf(0.09403159469366074f, a[15] * b[4], 0.05839917063713074f * (a[1] * b[8] + a[8] * b[1]))) + fmaf(-0.09403159469366074f, a[9] * b[8], fmaf(0.059470802545547485f, a[12] * b[5], 0.23359668254852295f * (a[2] * b[5] + a[5] * b[2])))));
        o[12] = ((fmaf(-0.18806318938732147f, a[14] * b[8], fmaf(-0.18806318938732147f, a[10] * b[4], 0.282094806432724f * a[12] * b[0])) + fmaf(0.059470802545547485f, a[11] * b[5], -0.14304816722869873f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.16820883750915527f, a[12] * b[6], 0.24776668846607208f * (a[2] * b[6] + a[6] * b[2])) + fmaf(0.059470802545547485f, a[13] * b[7], -0.14304816722869873f * (a[3] * b[7] + a[7] * b[3]))));
        o[13] = ((fmaf(-0.09403159469366074f, a[15] * b[8], fmaf(0.12615662813186646f, a[13] * b[6], fmaf(-0.05839917063713074f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * a[13] * b[0]))) + fmaf(0.059470802545547485f, a[12] * b[7], fmaf(-0.09403159469366074f, a[9] * b[4], -0.05839917063713074f * (a[1] * b[4] + a[4] * b[1])))) + (fmaf(0.11516471952199936f, a[14] * b[7], fmaf(0.14567312598228455f, a[11] * b[4], 0.23359668254852295f * (a[2] * b[7] + a[7] * b[2]))) + fmaf(0.14567312598228455f, a[13] * b[8], fmaf(0.11516471952199936f, a[10] * b[5], 0.20230065286159515f * (a[3] * b[6] + a[6] * b[3])))));
        o[14] = ((fmaf(-0.18806318938732147f, a[12] * b[8], fmaf(0.1486770063638687f, a[9] * b[5], 0.282094806432724f * a[14] * b[0])) + fmaf(-0.11516471952199936f, a[11] * b[5], -0.18467439711093903f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.11516471952199936f, a[13] * b[7], 0.18467439711093903f * (a[2] * b[8] + a[8] * b[2])) + fmaf(0.1486770063638687f, a[15] * b[7], 0.18467439711093903f * (a[3] * b[7] + a[7] * b[3]))));
        o[15] = ((fmaf(-0.1486770063638687f, a[10] * b[5], 0.282094806432724f * a[15] * b[0]) + fmaf(-0.2102610468864441f, a[15] * b[6], -0.22617901861667633f * (a[1] * b[4] + a[4] * b[1]))) + (fmaf(0.1486770063638687f, a[14] * b[7], 0.22617901861667633f * (a[3] * b[8] + a[8] * b[3])) + fmaf(-0.09403159469366074f, a[13] * b[8], 0.09403159469366074f * a[11] * b[4])));
    }
    __device__ __forceinline__ static void mul_onto_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[12] * b[12], fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0]))) + fmaf(0.282094806432724f, a[13] * b[13], fmaf(0.282094806432724f, a[9] * b[9], fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])))) + (fmaf(0.282094806432724f, a[14] * b[14], fmaf(0.282094806432724f, a[10] * b[10], fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]))) + fmaf(0.282094806432724f, a[15] * b[15], fmaf(0.282094806432724f, a[11] * b[11], fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])))));
        o[1] = ((fmaf(0.05839917063713074f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.18467439711093903f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0])))) + fmaf(0.20230065286159515f, (a[6] * b[11] + a[11] * b[6]), fmaf(-0.05839917063713074f, (a[4] * b[13] + a[13] * b[4]), -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1])))) + (fmaf(0.18467439711093903f, (a[7] * b[10] + a[10] * b[7]), fmaf(-0.22617901861667633f, (a[4] * b[15] + a[15] * b[4]), -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1]))) + fmaf(0.22617901861667633f, (a[8] * b[9] + a[9] * b[8]), fmaf(-0.14304816722869873f, (a[5] * b[12] + a[12] * b[5]), 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2])))));
        o[2] = ((fmaf(0.18467439711093903f, (a[8] * b[14] + a[14] * b[8]), fmaf(0.18467439711093903f, (a[4] * b[10] + a[10] * b[4]), 0.282094806432724f * (a[0] * b[2] + a[2] * b[0]))) + fmaf(0.23359668254852295f, (a[5] * b[11] + a[11] * b[5]), 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))) + (fmaf(0.24776668846607208f, (a[6] * b[12] + a[12] * b[6]), 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])) + fmaf(0.23359668254852295f, (a[7] * b[13] + a[13] * b[7]), 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))));
        o[3] = ((fmaf(0.22617901861667633f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.20230065286159515f, (a[6] * b[13] + a[13] * b[6]), fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0])))) + fmaf(-0.14304816722869873f, (a[7] * b[12] + a[12] * b[7]), fmaf(0.22617901861667633f, (a[4] * b[9] + a[9] * b[4]), 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1])))) + (fmaf(0.18467439711093903f, (a[7] * b[14] + a[14] * b[7]), fmaf(-0.05839917063713074f, (a[4] * b[11] + a[11] * b[4]), 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2]))) + fmaf(-0.05839917063713074f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.18467439711093903f, (a[5] * b[10] + a[10] * b[5]), -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3])))));
        o[4] = ((fmaf(0.09403159469366074f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.18467439711093903f, (a[2] * b[10] + a[10] * b[2]), 0.282094806432724f * (a[0] * b[4] + a[4] * b[0])))) + fmaf(-0.09403159469366074f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.22617901861667633f, (a[3] * b[9] + a[9] * b[3]), 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])))) + (fmaf(-0.18806318938732147f, (a[10] * b[12] + a[12] * b[10]), fmaf(-0.05839917063713074f, (a[3] * b[11] + a[11] * b[3]), -0.05839917063713074f * (a[1] * b[13] + a[13] * b[1]))) + fmaf(0.14567312598228455f, (a[11] * b[13] + a[13] * b[11]), fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * (a[1] * b[15] + a[15] * b[1])))));
        o[5] = ((fmaf(0.059470802545547485f, (a[11] * b[12] + a[12] * b[11]), fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.23359668254852295f, (a[2] * b[11] + a[11] * b[2]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])))) + fmaf(-0.11516471952199936f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.1486770063638687f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.18467439711093903f, (a[3] * b[10] + a[10] * b[3]), 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1]))))) + (fmaf(0.11516471952199936f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * (a[1] * b[12] + a[12] * b[1]))) + fmaf(-0.1486770063638687f, (a[10] * b[15] + a[15] * b[10]), fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), -0.18467439711093903f * (a[1] * b[14] + a[14] * b[1])))));
        o[6] = ((fmaf(-0.2102610468864441f, a[15] * b[15], fmaf(-0.2102610468864441f, a[9] * b[9], fmaf(0.0901118740439415f, a[5] * b[5], fmaf(0.24776668846607208f, (a[2] * b[12] + a[12] * b[2]), 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))))) + fmaf(0.12615662813186646f, a[11] * b[11], fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1])))) + (fmaf(0.16820883750915527f, a[12] * b[12], fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.20230065286159515f, (a[3] * b[13] + a[13] * b[3]), 0.20230065286159515f * (a[1] * b[11] + a[11] * b[1])))) + fmaf(0.12615662813186646f, a[13] * b[13], fmaf(-0.180223748087883f, a[8] * b[8], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2])))));
        o[7] = ((fmaf(0.11516471952199936f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.14304816722869873f, (a[3] * b[12] + a[12] * b[3]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])))) + fmaf(0.1486770063638687f, (a[14] * b[15] + a[15] * b[14]), fmaf(0.1486770063638687f, (a[9] * b[10] + a[10] * b[9]), fmaf(0.18467439711093903f, (a[3] * b[14] + a[14] * b[3]), 0.18467439711093903f * (a[1] * b[10] + a[10] * b[1]))))) + (fmaf(0.11516471952199936f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2]))) + fmaf(0.059470802545547485f, (a[12] * b[13] + a[13] * b[12]), fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), 0.23359668254852295f * (a[2] * b[13] + a[13] * b[2])))));
        o[8] = ((fmaf(-0.14567312598228455f, a[11] * b[11], fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.18467439711093903f, (a[2] * b[14] + a[14] * b[2]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])))) + fmaf(-0.18806318938732147f, (a[12] * b[14] + a[14] * b[12]), fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1])))) + (fmaf(0.14567312598228455f, a[13] * b[13], fmaf(0.15607835352420807f, a[7] * b[7], fmaf(-0.05839917063713074f, (a[3] * b[13] + a[13] * b[3]), 0.22617901861667633f * (a[1] * b[9] + a[9] * b[1])))) + fmaf(-0.09403159469366074f, (a[13] * b[15] + a[15] * b[13]), fmaf(-0.09403159469366074f, (a[9] * b[11] + a[11] * b[9]), fmaf(0.22617901861667633f, (a[3] * b[15] + a[15] * b[3]), 0.05839917063713074f * (a[1] * b[11] + a[11] * b[1]))))));
        o[9] = 0.0f;
        o[10] = 0.0f;
        o[11] = 0.0f;
        o[12] = 0.0f;
        o[13] = 0.0f;
        o[14] = 0.0f;
        o[15] = 0.0f;
    }
    __device__ __forceinline__ static void sqr(const float* __restrict__ a, float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[12] * a[12], fmaf(0.282094806432724f, a[8] * a[8], fmaf(0.282094806432724f, a[4] * a[4], 0.282094806432724f * a[0] * a[0]))) + fmaf(0.282094806432724f, a[13] * a[13], fmaf(0.282094806432724f, a[9] * a[9], fmaf(0.282094806432724f, a[5] * a[5], 0.282094806432724f * a[1] * a[1])))) + (fmaf(0.282094806432724f, a[14] * a[14], fmaf(0.282094806432724f, a[10] * a[10], fmaf(0.282094806432724f, a[6] * a[6], 0.282094806432724f * a[2] * a[2]))) + fmaf(0.282094806432724f, a[15] * a[15], fmaf(0.282094806432724f, a[11] * a[11], fmaf(0.282094806432724f, a[7] * a[7], 0.282094806432724f * a[3] * a[3])))));
        o[1] = ((fmaf(0.11679834127426147f, a[8] * a[11], fmaf(-0.36934879422187805f, a[5] * a[14], fmaf(0.43701937794685364f, a[3] * a[4], 0.564189612865448f * a[0] * a[1]))) + fmaf(0.4046013057231903f, a[6] * a[11], fmaf(-0.11679834127426147f, a[4] * a[13], -0.2523132562637329f * a[1] * a[6]))) + (fmaf(0.36934879422187805f, a[7] * a[10], fmaf(-0.45235803723335266f, a[4] * a[15], -0.43701937794685364f * a[1] * a[8])) + fmaf(0.45235803723335266f, a[8] * a[9], fmaf(-0.28609633445739746f, a[5] * a[12], 0.43701937794685364f * a[2] * a[5]))));
        o[2] = ((fmaf(0.36934879422187805f, a[8] * a[14], fmaf(0.36934879422187805f, a[4] * a[10], 0.564189612865448f * a[0] * a[2])) + fmaf(0.4671933650970459f, a[5] * a[11], 0.43701937794685364f * a[1] * a[5])) + (fmaf(0.49553337693214417f, a[6] * a[12], 0.5046265125274658f * a[2] * a[6]) + fmaf(0.4671933650970459f, a[7] * a[13], 0.43701937794685364f * a[3] * a[7])));
        o[3] = ((fmaf(0.45235803723335266f, a[8] * a[15], fmaf(0.4046013057231903f, a[6] * a[13], fmaf(0.43701937794685364f, a[3] * a[8], 0.564189612865448f * a[0] * a[3]))) + fmaf(-0.28609633445739746f, a[7] * a[12], fmaf(0.45235803723335266f, a[4] * a[9], 0.43701937794685364f * a[1] * a[4]))) + (fmaf(0.36934879422187805f, a[7] * a[14], fmaf(-0.11679834127426147f, a[4] * a[11], 0.43701937794685364f * a[2] * a[7])) + fmaf(-0.11679834127426147f, a[8] * a[13], fmaf(0.36934879422187805f, a[5] * a[10], -0.2523132562637329f * a[3] * a[6]))));
        o[4] = ((fmaf(0.18806318938732147f, a[11] * a[15], fmaf(0.31215670704841614f, a[5] * a[7], fmaf(0.36934879422187805f, a[2] * a[10], 0.564189612865448f * a[0] * a[4]))) + fmaf(-0.18806318938732147f, a[9] * a[13], fmaf(0.45235803723335266f, a[3] * a[9], 0.43701937794685364f * a[1] * a[3]))) + (fmaf(-0.37612637877464294f, a[10] * a[12], fmaf(-0.11679834127426147f, a[3] * a[11], -0.11679834127426147f * a[1] * a[13])) + fmaf(0.2913462519645691f, a[11] * a[13], fmaf(-0.360447496175766f, a[4] * a[6], -0.45235803723335266f * a[1] * a[15]))));
        o[5] = ((fmaf(0.11894160509109497f, a[11] * a[12], fmaf(-0.31215670704841614f, a[5] * a[8], fmaf(0.4671933650970459f, a[2] * a[11], 0.564189612865448f * a[0] * a[5]))) + fmaf(-0.23032943904399872f, a[11] * a[14], fmaf(0.2973540127277374f, a[9] * a[14], fmaf(0.36934879422187805f, a[3] * a[10], 0.43701937794685364f * a[1] * a[2])))) + (fmaf(0.23032943904399872f, a[10] * a[13], fmaf(0.31215670704841614f, a[4] * a[7], -0.28609633445739746f * a[1] * a[12])) + fmaf(-0.2973540127277374f, a[10] * a[15], fmaf(0.180223748087883f, a[5] * a[6], -0.36934879422187805f * a[1] * a[14]))));
        o[6] = ((fmaf(-0.2102610468864441f, a[15] * a[15], fmaf(-0.2102610468864441f, a[9] * a[9], fmaf(0.0901118740439415f, a[5] * a[5], fmaf(0.49553337693214417f, a[2] * a[12], 0.564189612865448f * a[0] * a[6])))) + fmaf(0.12615662813186646f, a[11] * a[11], fmaf(0.180223748087883f, a[6] * a[6], fmaf(-0.12615662813186646f, a[3] * a[3], -0.12615662813186646f * a[1] * a[1])))) + (fmaf(0.16820883750915527f, a[12] * a[12], fmaf(0.0901118740439415f, a[7] * a[7], fmaf(0.4046013057231903f, a[3] * a[13], 0.4046013057231903f * a[1] * a[11]))) + fmaf(0.12615662813186646f, a[13] * a[13], fmaf(-0.180223748087883f, a[8] * a[8], fmaf(-0.180223748087883f, a[4] * a[4], 0.2523132562637329f * a[2] * a[2])))));
        o[7] = ((fmaf(0.23032943904399872f, a[13] * a[14], fmaf(0.31215670704841614f, a[7] * a[8], fmaf(-0.28609633445739746f, a[3] * a[12], 0.564189612865448f * a[0] * a[7]))) + fmaf(0.2973540127277374f, a[14] * a[15], fmaf(0.2973540127277374f, a[9] * a[10], fmaf(0.36934879422187805f, a[3] * a[14], 0.36934879422187805f * a[1] * a[10])))) + (fmaf(0.23032943904399872f, a[10] * a[11], fmaf(0.31215670704841614f, a[4] * a[5], 0.43701937794685364f * a[2] * a[3])) + fmaf(0.11894160509109497f, a[12] * a[13], fmaf(0.180223748087883f, a[6] * a[7], 0.4671933650970459f * a[2] * a[13]))));
        o[8] = ((fmaf(-0.14567312598228455f, a[11] * a[11], fmaf(-0.15607835352420807f, a[5] * a[5], fmaf(0.36934879422187805f, a[2] * a[14], 0.564189612865448f * a[0] * a[8]))) + fmaf(-0.37612637877464294f, a[12] * a[14], fmaf(-0.360447496175766f, a[6] * a[8], fmaf(0.21850968897342682f, a[3] * a[3], -0.21850968897342682f * a[1] * a[1])))) + (fmaf(0.14567312598228455f, a[13] * a[13], fmaf(0.15607835352420807f, a[7] * a[7], fmaf(-0.11679834127426147f, a[3] * a[13], 0.45235803723335266f * a[1] * a[9]))) + fmaf(-0.18806318938732147f, a[13] * a[15], fmaf(-0.18806318938732147f, a[9] * a[11], fmaf(0.45235803723335266f, a[3] * a[15], 0.11679834127426147f * a[1] * a[11])))));
        o[9] = ((fmaf(0.2973540127277374f, a[5] * a[14], 0.564189612865448f * a[0] * a[9]) + fmaf(-0.4205220937728882f, a[6] * a[9], 0.45235803723335266f * a[1] * a[8])) + (fmaf(0.2973540127277374f, a[7] * a[10], 0.45235803723335266f * a[3] * a[4]) + fmaf(-0.18806318938732147f, a[8] * a[11], -0.18806318938732147f * a[4] * a[13])));
        o[10] = ((fmaf(0.23032943904399872f, a[7] * a[11], fmaf(-0.37612637877464294f, a[4] * a[12], 0.564189612865448f * a[0] * a[10])) + fmaf(0.23032943904399872f, a[5] * a[13], 0.36934879422187805f * a[1] * a[7])) + (fmaf(-0.2973540127277374f, a[5] * a[15], 0.36934879422187805f * a[2] * a[4]) + fmaf(0.2973540127277374f, a[7] * a[9], 0.36934879422187805f * a[3] * a[5])));
        o[11] = ((fmaf(-0.2913462519645691f, a[8] * a[11], fmaf(-0.23032943904399872f, a[5] * a[14], fmaf(-0.11679834127426147f, a[3] * a[4], 0.564189612865448f * a[0] * a[11]))) + fmaf(0.2523132562637329f, a[6] * a[11], fmaf(0.2913462519645691f, a[4] * a[13], 0.4046013057231903f * a[1] * a[6]))) + (fmaf(0.23032943904399872f, a[7] * a[10], fmaf(0.18806318938732147f, a[4] * a[15], 0.11679834127426147f * a[1] * a[8])) + fmaf(-0.18806318938732147f, a[8] * a[9], fmaf(0.11894160509109497f, a[5] * a[12], 0.4671933650970459f * a[2] * a[5]))));
        o[12] = ((fmaf(-0.37612637877464294f, a[8] * a[14], fmaf(-0.37612637877464294f, a[4] * a[10], 0.564189612865448f * a[0] * a[12])) + fmaf(0.11894160509109497f, a[5] * a[11], -0.28609633445739746f * a[1] * a[5])) + (fmaf(0.33641767501831055f, a[6] * a[12], 0.49553337693214417f * a[2] * a[6]) + fmaf(0.11894160509109497f, a[7] * a[13], -0.28609633445739746f * a[3] * a[7])));
        o[13] = ((fmaf(-0.18806318938732147f, a[8] * a[15], fmaf(0.2523132562637329f, a[6] * a[13], fmaf(-0.11679834127426147f, a[3] * a[8], 0.564189612865448f * a[0] * a[13]))) + fmaf(0.11894160509109497f, a[7] * a[12], fmaf(-0.18806318938732147f, a[4] * a[9], -0.11679834127426147f * a[1] * a[4]))) + (fmaf(0.23032943904399872f, a[7] * a[14], fmaf(0.2913462519645691f, a[4] * a[11], 0.4671933650970459f * a[2] * a[7])) + fmaf(0.2913462519645691f, a[8] * a[13], fmaf(0.23032943904399872f, a[5] * a[10], 0.4046013057231903f * a[3] * a[6]))));
        o[14] = ((fmaf(-0.37612637877464294f, a[8] * a[12], fmaf(0.2973540127277374f, a[5] * a[9], 0.564189612865448f * a[0] * a[14])) + fmaf(-0.23032943904399872f, a[5] * a[11], -0.36934879422187805f * a[1] * a[5])) + (fmaf(0.23032943904399872f, a[7] * a[13], 0.36934879422187805f * a[2] * a[8]) + fmaf(0.2973540127277374f, a[7] * a[15], 0.36934879422187805f * a[3] * a[7])));
        o[15] = ((fmaf(-0.2973540127277374f, a[5] * a[10], 0.564189612865448f * a[0] * a[15]) + fmaf(-0.4205220937728882f, a[6] * a[15], -0.45235803723335266f * a[1] * a[4])) + (fmaf(0.2973540127277374f, a[7] * a[14], 0.45235803723335266f * a[3] * a[8]) + fmaf(-0.18806318938732147f, a[8] * a[13], 0.18806318938732147f * a[4] * a[11])));
    }
};

#if defined(SHS_NB) && SHS_NB == 5
static __constant__ float kExpLeg5[250] = {0.282094806432724f, 0.11088809370994568f, -0.47585317492485046f, 0.11088809370994568f, 0.028136439621448517f, -0.24148334562778473f, 0.5820493698120117f, -0.24148334562778473f, 0.028136439621448517f, 0.006897183135151863f, -0.07249957323074341f, 0.3881925940513611f, -0.6332811713218689f, 0.3881925940513611f, -0.07249957323074341f, 0.006897183135151863f, 0.0016602643299847841f, -0.020151635631918907f, 0.13741593062877655f, -0.5381947755813599f, 0.6381627321243286f, -0.5381947755813599f, 0.13741593062877655f, -0.020151635631918907f, 0.0016602643299847841f, 0.282094806432724f, 0.24511361122131348f, -0.4226721227169037f, 0.24511361122131348f, 0.137478306889534f, -0.4741331934928894f, 0.39266371726989746f, -0.4741331934928894f, 0.137478306889534f, 0.0744936540722847f, -0.3146524429321289f, 0.6286184787750244f, -0.23942779004573822f, 0.6286184787750244f, -0.3146524429321289f, 0.0744936540722847f, 0.039637595415115356f, -0.1933251917362213f, 0.5046157836914062f, -0.6498939394950867f, 0.015881182625889778f, -0.6498939394950867f, 0.5046157836914062f, -0.1933251917362213f, 0.039637595415115356f, 0.282094806432724f, 0.3585166037082672f, -0.3319612145423889f, 0.3585166037082672f, 0.29411548376083374f, -0.5446605682373047f, 0.1213601753115654f, -0.5446605682373047f, 0.29411548376083374f, 0.23310139775276184f, -0.5286869406700134f, 0.438648521900177f, 0.17545272409915924f, 0.438648521900177f, -0.5286869406700134f, 0.23310139775276184f, 0.1814156323671341f, -0.47511395812034607f, 0.5683075189590454f, -0.07710716128349304f, -0.3586549460887909f, -0.07710716128349304f, 0.5683075189590454f, -0.47511395812034607f, 0.1814156323671341f, 0.282094806432724f, 0.44033047556877136f, -0.2117580771446228f, 0.44033047556877136f, 0.4436666667461395f, -0.42672494053840637f, -0.13767008483409882f, -0.42672494053840637f, 0.4436666667461395f, 0.4318702220916748f, -0.5087332725524902f, -0.025060366839170456f, 0.3333059847354889f, -0.025060366839170456f, -0.5087332725524902f, 0.4318702220916748f, 0.4128122329711914f, -0.5615116953849792f, 0.12096259742975235f, 0.440361887216568f, -0.1481127291917801f, 0.440361887216568f, 0.12096259742975235f, -0.5615116953849792f, 0.4128122329711914f, 0.282094806432724f, 0.48315757513046265f, -0.07274037599563599f, 0.48315757513046265f, 0.5341668128967285f, -0.16083984076976776f, -0.2944209575653076f, -0.16083984076976776f, 0.5341668128967285f, 0.5705364942550659f, -0.21040001511573792f, -0.40186813473701477f, 0.1605125069618225f, -0.40186813473701477f, -0.21040001511573792f, 0.5705364942550659f, 0.598401665687561f, -0.2548147141933441f, -0.3908316493034363f, 0.2802008390426636f, 0.24883784353733063f, 0.2802008390426636f, -0.3908316493034363f, -0.2548147141933441f, 0.598401665687561f, 0.282094806432724f, 0.48315757513046265f, 0.07274037599563599f, 0.48315757513046265f, 0.5341668128967285f, 0.16083984076976776f, -0.2944209575653076f, 0.16083984076976776f, 0.5341668128967285f, 0.5705364942550659f, 0.21040001511573792f, -0.40186813473701477f, -0.1605125069618225f, -0.40186813473701477f, 0.21040001511573792f, 0.5705364942550659f, 0.598401665687561f, 0.2548147141933441f, -0.3908316493034363f, -0.2802008390426636f, 0.24883784353733063f, -0.2802008390426636f, -0.3908316493034363f, 0.2548147141933441f, 0.598401665687561f, 0.282094806432724f, 0.44033047556877136f, 0.2117580771446228f, 0.44033047556877136f, 0.4436666667461395f, 0.42672494053840637f, -0.13767008483409882f, 0.42672494053840637f, 0.4436666667461395f, 0.4318702220916748f, 0.5087332725524902f, -0.025060366839170456f, -0.3333059847354889f, -0.025060366839170456f, 0.5087332725524902f, 0.4318702220916748f, 0.4128122329711914f, 0.5615116953849792f, 0.12096259742975235f, -0.440361887216568f, -0.1481127291917801f, -0.440361887216568f, 0.12096259742975235f, 0.5615116953849792f, 0.4128122329711914f, 0.282094806432724f, 0.3585166037082672f, 0.3319612145423889f, 0.3585166037082672f, 0.29411548376083374f, 0.5446605682373047f, 0.1213601753115654f, 0.5446605682373047f, 0.29411548376083374f, 0.23310139775276184f, 0.5286869406700134f, 0.438648521900177f, -0.17545272409915924f, 0.438648521900177f, 0.5286869406700134f, 0.23310139775276184f, 0.1814156323671341f, 0.47511395812034607f, 0.5683075189590454f, 0.07710716128349304f, -0.3586549460887909f, 0.07710716128349304f, 0.5683075189590454f, 0.47511395812034607f, 0.1814156323671341f, 0.282094806432724f, 0.24511361122131348f, 0.4226721227169037f, 0.24511361122131348f, 0.137478306889534f, 0.4741331934928894f, 0.39266371726989746f, 0.4741331934928894f, 0.137478306889534f, 0.0744936540722847f, 0.3146524429321289f, 0.6286184787750244f, 0.23942779004573822f, 0.6286184787750244f, 0.3146524429321289f, 0.0744936540722847f, 0.039637595415115356f, 0.1933251917362213f, 0.5046157836914062f, 0.6498939394950867f, 0.015881182625889778f, 0.6498939394950867f, 0.5046157836914062f, 0.1933251917362213f, 0.039637595415115356f, 0.282094806432724f, 0.11088809370994568f, 0.47585317492485046f, 0.11088809370994568f, 0.028136439621448517f, 0.24148334562778473f, 0.5820493698120117f, 0.24148334562778473f, 0.028136439621448517f, 0.006897183135151863f, 0.07249957323074341f, 0.3881925940513611f, 0.6332811713218689f, 0.3881925940513611f, 0.07249957323074341f, 0.006897183135151863f, 0.0016602643299847841f, 0.020151635631918907f, 0.13741593062877655f, 0.5381947755813599f, 0.6381627321243286f, 0.5381947755813599f, 0.13741593062877655f, 0.020151635631918907f, 0.0016602643299847841f};
static __constant__ float kExpTrig5[180] = {1.0f, 0.9876883625984192f, 0.15643446147441864f, 0.9510565400123596f, 0.30901700258255005f, 0.8910065293312073f, 0.45399048924446106f, 0.80901700258255f, 0.5877852439880371f, 1.0f, 0.8910065293312073f, 0.45399048924446106f, 0.5877852439880371f, 0.80901700258255f, 0.15643446147441864f, 0.9876883625984192f, -0.30901700258255005f, 0.9510565400123596f, 1.0f, 0.7071067690849304f, 0.7071067690849304f, 6.123234262925839e-17f, 1.0f, -0.7071067690849304f, 0.7071067690849304f, -1.0f, 1.2246468525851679e-16f, 1.0f, 0.45399048924446106f, 0.8910065293312073f, -0.5877852439880371f, 0.80901700258255f, -0.9876883625984192f, -0.15643446147441864f, -0.30901700258255005f, -0.9510565400123596f, 1.0f, 0.15643446147441864f, 0.9876883625984192f, -0.9510565400123596f, 0.30901700258255005f, -0.45399048924446106f, -0.8910065293312073f, 0.80901700258255f, -0.5877852439880371f, 1.0f, -0.15643446147441864f, 0.9876883625984192f, -0.9510565400123596f, -0.30901700258255005f, 0.45399048924446106f, -0.8910065293312073f, 0.80901700258255f, 0.5877852439880371f, 1.0f, -0.45399048924446106f, 0.8910065293312073f, -0.5877852439880371f, -0.80901700258255f, 0.9876883625984192f, -0.15643446147441864f, -0.30901700258255005f, 0.9510565400123596f, 1.0f, -0.7071067690849304f, 0.7071067690849304f, -1.8369701465288538e-16f, -1.0f, 0.7071067690849304f, 0.7071067690849304f, -1.0f, 3.6739402930577075e-16f, 1.0f, -0.8910065293312073f, 0.45399048924446106f, 0.5877852439880371f, -0.80901700258255f, -0.15643446147441864f, 0.9876883625984192f, -0.30901700258255005f, -0.9510565400123596f, 1.0f, -0.9876883625984192f, 0.15643446147441864f, 0.9510565400123596f, -0.30901700258255005f, -0.8910065293312073f, 0.45399048924446106f, 0.80901700258255f, -0.5877852439880371f, 1.0f, -0.9876883625984192f, -0.15643446147441864f, 0.9510565400123596f, 0.30901700258255005f, -0.8910065293312073f, -0.45399048924446106f, 0.80901700258255f, 0.5877852439880371f, 1.0f, -0.8910065293312073f, -0.45399048924446106f, 0.5877852439880371f, 0.80901700258255f, -0.15643446147441864f, -0.9876883625984192f, -0.30901700258255005f, 0.9510565400123596f, 1.0f, -0.7071067690849304f, -0.7071067690849304f, 3.0616169991140216e-16f, 1.0f, 0.7071067690849304f, -0.7071067690849304f, -1.0f, 6.123233998228043e-16f, 1.0f, -0.45399048924446106f, -0.8910065293312073f, -0.5877852439880371f, 0.80901700258255f, 0.9876883625984192f, 0.15643446147441864f, -0.30901700258255005f, -0.9510565400123596f, 1.0f, -0.15643446147441864f, -0.9876883625984192f, -0.9510565400123596f, 0.30901700258255005f, 0.45399048924446106f, 0.8910065293312073f, 0.80901700258255f, -0.5877852439880371f, 1.0f, 0.15643446147441864f, -0.9876883625984192f, -0.9510565400123596f, -0.30901700258255005f, -0.45399048924446106f, 0.8910065293312073f, 0.80901700258255f, 0.5877852439880371f, 1.0f, 0.45399048924446106f, -0.8910065293312073f, -0.5877852439880371f, -0.80901700258255f, -0.9876883625984192f, 0.15643446147441864f, -0.30901700258255005f, 0.9510565400123596f, 1.0f, 0.7071067690849304f, -0.7071067690849304f, -4.2862638516991895e-16f, -1.0f, -0.7071067690849304f, -0.7071067690849304f, -1.0f, 8.572527703398379e-16f, 1.0f, 0.8910065293312073f, -0.45399048924446106f, 0.5877852439880371f, -0.80901700258255f, 0.15643446147441864f, -0.9876883625984192f, -0.30901700258255005f, -0.9510565400123596f, 1.0f, 0.9876883625984192f, -0.15643446147441864f, 0.9510565400123596f, -0.30901700258255005f, 0.8910065293312073f, -0.45399048924446106f, 0.80901700258255f, -0.5877852439880371f};
static __constant__ float kExpW5[10] = {0.020945420488715172f, 0.046951524913311005f, 0.06882800906896591f, 0.08459263294935226f, 0.09284166991710663f, 0.09284166991710663f, 0.08459263294935226f, 0.06882800906896591f, 0.046951524913311005f, 0.020945420488715172f};
#endif
template <> struct SH<5> {
    static constexpr int K = 25;
    static constexpr int NNZ_SYM = 623;   // entries (i, j <= k)
    static constexpr int EZ = 10;    // projected-exponential rule: Gauss-Legendre nodes
    static constexpr int EP = 20;    // projected-exponential rule: uniform azimuths
#if defined(SHS_NB) && SHS_NB == 5
    __device__ __forceinline__ static const float* eleg() { return kExpLeg5; }
    __device__ __forceinline__ static const float* etrig() { return kExpTrig5; }
    __device__ __forceinline__ static const float* ew() { return kExpW5; }
#endif
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            case 9: return 0.03933623805642128f;
            case 10: return 0.09635371714830399f;
            case 11: return 0.304697185754776f;
            case 12: return 0.7463526725769043f;
            case 13: return 0.304697185754776f;
            case 14: return 0.09635371714830399f;
            case 15: return 0.03933623805642128f;
            case 16: return 0.005960340145975351f;
            case 17: return 0.016858387738466263f;
            case 18: return 0.06307831406593323f;
            case 19: return 0.2676186263561249f;
            case 20: return 0.8462843894958496f;
            case 21: return 0.2676186263561249f;
            case 22: return 0.06307831406593323f;
            case 23: return 0.016858387738466263f;
            case 24: return 0.005960340145975351f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            case 3: return 0.0f;
            case 4: return -0.13089969754219055f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static void ybar(float x, float y, float z, float* Y) {
        (void)x; (void)y; (void)z;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = x * t2;
        const float t7 = y * t5;
        const float t8 = t6 - t7;
        const float t9 = x * t5;
        const float t10 = y * t2;
        const float t11 = t9 + t10;
        const float t12 = x * t8;
        const float t13 = y * t11;
        const float t14 = t12 - t13;
        const float t15 = x * t11;
        const float t16 = y * t8;
        const float t17 = t15 + t16;
        const float t18 = z * z;
        const float t19 = t18 * 1.5f;
        const float t20 = t19 - 0.5f;
        const float t21 = z * t20;
        const float t22 = t21 * 1.6666666269302368f;
        const float t23 = z * 0.6666666865348816f;
        const float t24 = t22 - t23;
        const float t25 = z * t24;
        const float t26 = t25 * 1.75f;
        const float t27 = t20 * 0.75f;
        const float t28 = t26 - t27;
        const float t29 = z * 3.0f;
        const float t30 = z * t29;
        const float t31 = t30 * 2.5f;
        const float t32 = t31 - 1.5f;
        const float t33 = z * t32;
        const float t34 = t33 * 2.3333332538604736f;
        const float t35 = t29 * 1.3333333730697632f;
        const float t36 = t34 - t35;
        const float t37 = z * 3.0f;
        const float t38 = t37 * 5.0f;
        const float t39 = z * t38;
        const float t40 = t39 * 3.5f;
        const float t41 = t40 - 7.5f;
        const float t42 = z * 15.0f;
        const float t43 = t42 * 7.0f;
        const float t44 = t29 * x;
        const float t45 = t29 * y;
        const float t46 = t2 * 3.0f;
        const float t47 = t5 * 3.0f;
        const float t48 = t32 * x;
        const float t49 = t32 * y;
        const float t50 = t38 * t2;
        const float t51 = t38 * t5;
        const float t52 = t8 * 15.0f;
        const float t53 = t11 * 15.0f;
        const float t54 = t36 * x;
        const float t55 = t36 * y;
        const float t56 = t41 * t2;
        const float t57 = t41 * t5;
        const float t58 = t43 * t8;
        const float t59 = t43 * t11;
        const float t60 = t14 * 105.0f;
        const float t61 = t17 * 105.0f;
        Y[0] = 1.0f;
        Y[1] = y;
        Y[2] = z;
        Y[3] = x;
        Y[4] = t47;
        Y[5] = t45;
        Y[6] = t20;
        Y[7] = t44;
        Y[8] = t46;
        Y[9] = t53;
        Y[10] = t51;
        Y[11] = t49;
        Y[12] = t24;
        Y[13] = t48;
        Y[14] = t50;
        Y[15] = t52;
        Y[16] = t61;
        Y[17] = t59;
        Y[18] = t57;
        Y[19] = t55;
        Y[20] = t28;
        Y[21] = t54;
        Y[22] = t56;
        Y[23] = t58;
        Y[24] = t60;
    }
    __device__ __forceinline__ static void ybar_vjp(float x, float y, float z, const float* w,
                                                    float& gx, float& gy, float& gz) {
        (void)x; (void)y; (void)z; (void)w;
        const float t0 = x * x;
        const float t1 = y * y;
        const float t2 = t0 - t1;
        const float t3 = x * y;
        const float t4 = y * x;
        const float t5 = t3 + t4;
        const float t6 = x * t2;
        const float t7 = y * t5;
        const float t8 = t6 - t7;
        const float t9 = x * t5;
        const float t10 = y * t2;
        const float t11 = t9 + t10;
        const float t12 = x * t8;
        const float t13 = y * t11;
        const float t14 = t12 - t13;
        const float t15 = x * t11;
        const float t16 = y * t8;
        const float t17 = t15 + t16;
        const float t18 = z * z;
        const float t19 = t18 * 1.5f;
        const float t20 = t19 - 0.5f;
        const float t21 = z * t20;
        const float t22 = t21 * 1.6666666269302368f;
        const float t23 = z * 0.6666666865348816f;
        const float t24 = t22 - t23;
        const float t25 = z * t24;
        const float t26 = t25 * 1.75f;
        const float t27 = t20 * 0.75f;
        const float t28 = t26 - t27;
        const float t29 = z * 3.0f;
        const float t30 = z * t29;
        const float t31 = t30 * 2.5f;
        const float t32 = t31 - 1.5f;
        const float t33 = z * t32;
        const float t34 = t33 * 2.3333332538604736f;
        const float t35 = t29 * 1.3333333730697632f;
        const float t36 = t34 - t35;
        const float t37 = z * 3.0f;
        const float t38 = t37 * 5.0f;
        const float t39 = z * t38;
        const float t40 = t39 * 3.5f;
        const float t41 = t40 - 7.5f;
        const float t42 = z * 15.0f;
        const float t43 = t42 * 7.0f;
        const float t44 = t29 * x;
        const float t45 = t29 * y;
        const float t46 = t2 * 3.0f;
        const float t47 = t5 * 3.0f;
        const float t48 = t32 * x;
        const float t49 = t32 * y;
        const float t50 = t38 * t2;
        const float t51 = t38 * t5;
        const float t52 = t8 * 15.0f;
        const float t53 = t11 * 15.0f;
        const float t54 = t36 * x;
        const float t55 = t36 * y;
        const float t56 = t41 * t2;
        const float t57 = t41 * t5;
        const float t58 = t43 * t8;
        const float t59 = t43 * t11;
        const float t60 = t14 * 105.0f;
        const float t61 = t17 * 105.0f;
        const float a_t61 = w[16];
        const float a_t60 = w[24];
        const float a_t59 = w[17];
        const float a_t58 = w[23];
        const float a_t57 = w[18];
        const float a_t56 = w[22];
        const float a_t55 = w[19];
        const float a_t54 = w[21];
        const float a_t53 = w[9];
        const float a_t52 = w[15];
        const float a_t51 = w[10];
        const float a_t50 = w[14];
        const float a_t49 = w[11];
        const float a_t48 = w[13];
        const float a_t47 = w[4];
        const float a_t46 = w[8];
        const float a_t45 = w[5];
        const float a_t44 = w[7];
        const float a_t43 = t11 * a_t59 + t8 * a_t58;
        const float a_t42 = 7.0f * a_t43;
        const float a_t41 = t5 * a_t57 + t2 * a_t56;
        const float a_t40 = a_t41;
        const float a_t39 = 3.5f * a_t40;
        const float a_t38 = t5 * a_t51 + t2 * a_t50 + z * a_t39;
        const float a_t37 = 5.0f * a_t38;
        const float a_t36 = y * a_t55 + x * a_t54;
        const float a_t35 = -a_t36;
        const float a_t34 = a_t36;
        const float a_t33 = 2.3333332538604736f * a_t34;
        const float a_t32 = y * a_t49 + x * a_t48 + z * a_t33;
        const float a_t31 = a_t32;
        const float a_t30 = 2.5f * a_t31;
        const float a_t29 = y * a_t45 + x * a_t44 + 1.3333333730697632f * a_t35 + z * a_t30;
        const float a_t28 = w[20];
        const float a_t27 = -a_t28;
        const float a_t26 = a_t28;
        const float a_t25 = 1.75f * a_t26;
        const float a_t24 = w[12] + z * a_t25;
        const float a_t23 = -a_t24;
        const float a_t22 = a_t24;
        const float a_t21 = 1.6666666269302368f * a_t22;
        const float a_t20 = w[6] + 0.75f * a_t27 + z * a_t21;
        const float a_t19 = a_t20;
        const float a_t18 = 1.5f * a_t19;
        const float a_t17 = 105.0f * a_t61;
        const float a_t16 = a_t17;
        const float a_t15 = a_t17;
        const float a_t14 = 105.0f * a_t60;
        const float a_t13 = -a_t14;
        const float a_t12 = a_t14;
        const float a_t11 = t43 * a_t59 + 15.0f * a_t53 + x * a_t15 + y * a_t13;
        const float a_t10 = a_t11;
        const float a_t9 = a_t11;
        const float a_t8 = t43 * a_t58 + 15.0f * a_t52 + y * a_t16 + x * a_t12;
        const float a_t7 = -a_t8;
        const float a_t6 = a_t8;
        const float a_t5 = t41 * a_t57 + t38 * a_t51 + 3.0f * a_t47 + x * a_t9 + y * a_t7;
        const float a_t4 = a_t5;
        const float a_t3 = a_t5;
        const float a_t2 = t41 * a_t56 + t38 * a_t50 + 3.0f * a_t46 + y * a_t10 + x * a_t6;
        const float a_t1 = -a_t2;
        const float a_t0 = a_t2;
        gx = w[3] + t36 * a_t54 + t32 * a_t48 + t29 * a_t44 + t11 * a_t15 + t8 * a_t12 + t5 * a_t9 + t2 * a_t6 + y * a_t4 + y * a_t3 + x * a_t0 + x * a_t0;
        gy = w[1] + t36 * a_t55 + t32 * a_t49 + t29 * a_t45 + t8 * a_t16 + t11 * a_t13 + t2 * a_t10 + t5 * a_t7 + x * a_t4 + x * a_t3 + y * a_t1 + y * a_t1;
        gz = w[2] + 15.0f * a_t42 + t38 * a_t39 + 3.0f * a_t37 + t32 * a_t33 + t29 * a_t30 + 3.0f * a_t29 + t24 * a_t25 + 0.6666666865348816f * a_t23 + t20 * a_t21 + z * a_t18 + z * a_t18;
    }
    static constexpr int NA = 35;   // monomials of degree < n
    static constexpr int NG = 34;   // symmetric tensor entries, bands >= 1
    __device__ __forceinline__ static void accumulate(const float* G, float x, float y, float z, float* acc) {
        (void)x; (void)y; (void)z;
        const float m1_0_0 = x;
        const float m0_1_0 = y;
        const float m0_0_1 = z;
        const float m2_0_0 = x * m1_0_0;
        const float m1_1_0 = x * m0_1_0;
        const float m1_0_1 = x * m0_0_1;
        const float m0_2_0 = y * m0_1_0;
        const float m0_1_1 = y * m0_0_1;
        const float m0_0_2 = z * m0_0_1;
        const float m3_0_0 = x * m2_0_0;
        const float m2_1_0 = x * m1_1_0;
        const float m2_0_1 = x * m1_0_1;
        const float m1_2_0 = x * m0_2_0;
        const float m1_1_1 = x * m0_1_1;
        const float m1_0_2 = x * m0_0_2;
        const float m0_3_0 = y * m0_2_0;
        const float m0_2_1 = y * m0_1_1;
        const float m0_1_2 = y * m0_0_2;
        const float m0_0_3 = z * m0_0_2;
        const float gtx = G[4] * x;
        const float gty = G[4] * y;
        const float gtz = G[4] * z;
        acc[0] = fmaf(G[0], 1.0f, acc[0]);
        acc[1] = fmaf(G[1], m1_0_0, acc[1]);
        acc[2] = fmaf(G[1], m0_1_0, acc[2]);
        acc[3] = fmaf(G[1], m0_0_1, acc[3]);
        acc[4] = fmaf(G[2], m2_0_0, acc[4]);
        acc[5] = fmaf(G[2], m1_1_0, acc[5]);
        acc[6] = fmaf(G[2], m1_0_1, acc[6]);
        acc[7] = fmaf(G[2], m0_2_0, acc[7]);
        acc[8] = fmaf(G[2], m0_1_1, acc[8]);
        acc[9] = fmaf(G[2], m0_0_2, acc[9]);
        acc[10] = fmaf(G[3], m3_0_0, acc[10]);
        acc[11] = fmaf(G[3], m2_1_0, acc[11]);
        acc[12] = fmaf(G[3], m2_0_1, acc[12]);
        acc[13] = fmaf(G[3], m1_2_0, acc[13]);
        acc[14] = fmaf(G[3], m1_1_1, acc[14]);
        acc[15] = fmaf(G[3], m1_0_2, acc[15]);
        acc[16] = fmaf(G[3], m0_3_0, acc[16]);
        acc[17] = fmaf(G[3], m0_2_1, acc[17]);
        acc[18] = fmaf(G[3], m0_1_2, acc[18]);
        acc[19] = fmaf(G[3], m0_0_3, acc[19]);
        acc[20] = fmaf(gtx, m3_0_0, acc[20]);
        acc[21] = fmaf(gtx, m2_1_0, acc[21]);
        acc[22] = fmaf(gtx, m2_0_1, acc[22]);
        acc[23] = fmaf(gtx, m1_2_0, acc[23]);
        acc[24] = fmaf(gtx, m1_1_1, acc[24]);
        acc[25] = fmaf(gtx, m1_0_2, acc[25]);
        acc[26] = fmaf(gtx, m0_3_0, acc[26]);
        acc[27] = fmaf(gtx, m0_2_1, acc[27]);
        acc[28] = fmaf(gtx, m0_1_2, acc[28]);
        acc[29] = fmaf(gtx, m0_0_3, acc[29]);
        acc[30] = fmaf(gty, m0_3_0, acc[30]);
        acc[31] = fmaf(gty, m0_2_1, acc[31]);
        acc[32] = fmaf(gty, m0_1_2, acc[32]);
        acc[33] = fmaf(gty, m0_0_3, acc[33]);
        acc[34] = fmaf(gtz, m0_0_3, acc[34]);
    }
    // the same for two pairs at once, one per half of each float2
    __device__ __forceinline__ static void accumulate2(const float2* G, float2 x, float2 y, float2 z,
                                                       float2* acc) {
        (void)x; (void)y; (void)z;
        const float2 m1_0_0 = x;
        const float2 m0_1_0 = y;
        const float2 m0_0_1 = z;
        const float2 m2_0_0 = __fmul2_rn(x, m1_0_0);
        const float2 m1_1_0 = __fmul2_rn(x, m0_1_0);
        const float2 m1_0_1 = __fmul2_rn(x, m0_0_1);
        const float2 m0_2_0 = __fmul2_rn(y, m0_1_0);
        const float2 m0_1_1 = __fmul2_rn(y, m0_0_1);
        const float2 m0_0_2 = __fmul2_rn(z, m0_0_1);
        const float2 m3_0_0 = __fmul2_rn(x, m2_0_0);
        const float2 m2_1_0 = __fmul2_rn(x, m1_1_0);
        const float2 m2_0_1 = __fmul2_rn(x, m1_0_1);
        const float2 m1_2_0 = __fmul2_rn(x, m0_2_0);
        const float2 m1_1_1 = __fmul2_rn(x, m0_1_1);
        const float2 m1_0_2 = __fmul2_rn(x, m0_0_2);
        const float2 m0_3_0 = __fmul2_rn(y, m0_2_0);
        const float2 m0_2_1 = __fmul2_rn(y, m0_1_1);
        const float2 m0_1_2 = __fmul2_rn(y, m0_0_2);
        const float2 m0_0_3 = __fmul2_rn(z, m0_0_2);
        const float2 gtx = __fmul2_rn(G[4], x);
        const float2 gty = __fmul2_rn(G[4], y);
        const float2 gtz = __fmul2_rn(G[4], z);
        acc[0] = __fadd2_rn(G[0], acc[0]);
        acc[1] = __ffma2_rn(G[1], m1_0_0, acc[1]);
        acc[2] = __ffma2_rn(G[1], m0_1_0, acc[2]);
        acc[3] = __ffma2_rn(G[1], m0_0_1, acc[3]);
        acc[4] = __ffma2_rn(G[2], m2_0_0, acc[4]);
        acc[5] = __ffma2_rn(G[2], m1_1_0, acc[5]);
        acc[6] = __ffma2_rn(G[2], m1_0_1, acc[6]);
        acc[7] = __ffma2_rn(G[2], m0_2_0, acc[7]);
        acc[8] = __ffma2_rn(G[2], m0_1_1, acc[8]);
        acc[9] = __ffma2_rn(G[2], m0_0_2, acc[9]);
        acc[10] = __ffma2_rn(G[3], m3_0_0, acc[10]);
        acc[11] = __ffma2_rn(G[3], m2_1_0, acc[11]);
        acc[12] = __ffma2_rn(G[3], m2_0_1, acc[12]);
        acc[13] = __ffma2_rn(G[3], m1_2_0, acc[13]);
        acc[14] = __ffma2_rn(G[3], m1_1_1, acc[14]);
        acc[15] = __ffma2_rn(G[3], m1_0_2, acc[15]);
        acc[16] = __ffma2_rn(G[3], m0_3_0, acc[16]);
        acc[17] = __ffma2_rn(G[3], m0_2_1, acc[17]);
        acc[18] = __ffma2_rn(G[3], m0_1_2, acc[18]);
        acc[19] = __ffma2_rn(G[3], m0_0_3, acc[19]);
        acc[20] = __ffma2_rn(gtx, m3_0_0, acc[20]);
        acc[21] = __ffma2_rn(gtx, m2_1_0, acc[21]);
        acc[22] = __ffma2_rn(gtx, m2_0_1, acc[22]);
        acc[23] = __ffma2_rn(gtx, m1_2_0, acc[23]);
        acc[24] = __ffma2_rn(gtx, m1_1_1, acc[24]);
        acc[25] = __ffma2_rn(gtx, m1_0_2, acc[25]);
        acc[26] = __ffma2_rn(gtx, m0_3_0, acc[26]);
        acc[27] = __ffma2_rn(gtx, m0_2_1, acc[27]);
        acc[28] = __ffma2_rn(gtx, m0_1_2, acc[28]);
        acc[29] = __ffma2_rn(gtx, m0_0_3, acc[29]);
        acc[30] = __ffma2_rn(gty, m0_3_0, acc[30]);
        acc[31] = __ffma2_rn(gty, m0_2_1, acc[31]);
        acc[32] = __ffma2_rn(gty, m0_1_2, acc[32]);
        acc[33] = __ffma2_rn(gty, m0_0_3, acc[33]);
        acc[34] = __ffma2_rn(gtz, m0_0_3, acc[34]);
    }
    __device__ __forceinline__ static void mono_to_f(const float* acc, float* f) {
        f[0] = 1.0f * acc[0];
        f[1] = 1.0f * acc[2];
        f[2] = 1.0f * acc[3];
        f[3] = 1.0f * acc[1];
        f[4] = 6.0f * acc[5];
        f[5] = 3.0f * acc[8];
        f[6] = ((1.0f * acc[9] + -0.5f * acc[7]) + -0.5f * acc[4]);
        f[7] = 3.0f * acc[6];
        f[8] = (-3.0f * acc[7] + 3.0f * acc[4]);
        f[9] = (-15.0f * acc[16] + 45.0f * acc[11]);
        f[10] = 30.0f * acc[14];
        f[11] = ((6.0f * acc[18] + -1.5f * acc[16]) + -1.5f * acc[11]);
        f[12] = ((1.0f * acc[19] + -1.5f * acc[17]) + -1.5f * acc[12]);
        f[13] = ((6.0f * acc[15] + -1.5f * acc[13]) + -1.5f * acc[10]);
        f[14] = (-15.0f * acc[17] + 15.0f * acc[12]);
        f[15] = (-45.0f * acc[13] + 15.0f * acc[10]);
        f[16] = (-420.0f * acc[26] + 420.0f * acc[21]);
        f[17] = (-105.0f * acc[31] + 315.0f * acc[24]);
        f[18] = ((90.0f * acc[28] + -15.0f * acc[26]) + -15.0f * acc[21]);
        f[19] = ((10.0f * acc[33] + -7.5f * acc[31]) + -7.5f * acc[24]);
        f[20] = ((fmaf(0.75f, acc[23], 1.0f * acc[34]) + fmaf(0.375f, acc[20], -3.0f * acc[32])) + (0.375f * acc[30] + -3.0f * acc[25]));
        f[21] = ((10.0f * acc[29] + -7.5f * acc[27]) + -7.5f * acc[22]);
        f[22] = ((-45.0f * acc[32] + 7.5f * acc[30]) + (45.0f * acc[25] + -7.5f * acc[20]));
        f[23] = (-315.0f * acc[27] + 105.0f * acc[22]);
        f[24] = ((105.0f * acc[30] + -630.0f * acc[23]) + 105.0f * acc[20]);
    }
    __device__ __forceinline__ static void grad_coeffs(const float* w, float* gq) {
        (void)w; (void)gq;
        gq[0] = 1.0f * w[3];
        gq[1] = 1.0f * w[1];
        gq[2] = 1.0f * w[2];
        gq[3] = (-1.0f * w[6] + 6.0f * w[8]);
        gq[4] = 6.0f * w[4];
        gq[5] = 3.0f * w[7];
        gq[6] = (-1.0f * w[6] + -6.0f * w[8]);
        gq[7] = 3.0f * w[5];
        gq[8] = 2.0f * w[6];
        gq[9] = (-4.5f * w[13] + 45.0f * w[15]);
        gq[10] = (45.0f * w[9] + -1.5f * w[11]);
        gq[11] = (-1.5f * w[12] + 15.0f * w[14]);
        gq[12] = (-1.5f * w[13] + -45.0f * w[15]);
        gq[13] = 15.0f * w[10];
        gq[14] = 6.0f * w[13];
        gq[15] = (-45.0f * w[9] + -4.5f * w[11]);
        gq[16] = (-1.5f * w[12] + -15.0f * w[14]);
        gq[17] = 6.0f * w[11];
        gq[18] = 3.0f * w[12];
        gq[19] = ((1.5f * w[20] + -30.0f * w[22]) + 420.0f * w[24]);
        gq[20] = (420.0f * w[16] + -15.0f * w[18]);
        gq[21] = (-7.5f * w[21] + 105.0f * w[23]);
        gq[22] = (0.5f * w[20] + -420.0f * w[24]);
        gq[23] = (105.0f * w[17] + -2.5f * w[19]);
        gq[24] = (-2.0f * w[20] + 30.0f * w[22]);
        gq[25] = (-420.0f * w[16] + -15.0f * w[18]);
        gq[26] = (-2.5f * w[21] + -105.0f * w[23]);
        gq[27] = 30.0f * w[18];
        gq[28] = 10.0f * w[21];
        gq[29] = ((1.5f * w[20] + 30.0f * w[22]) + 420.0f * w[24]);
        gq[30] = (-105.0f * w[17] + -7.5f * w[19]);
        gq[31] = (-2.0f * w[20] + -30.0f * w[22]);
        gq[32] = 10.0f * w[19];
        gq[33] = 4.0f * w[20];
    }
    template <class Q>
    __device__ __forceinline__ static void grad_eval2(float2 x, float2 y, float2 z, Q&& gq,
                                                      float2* gx, float2* gy, float2* gz) {
        (void)x; (void)y; (void)z; (void)gq; (void)gx; (void)gy; (void)gz;
        const float2 x2 = __fmul2_rn(make_float2(2.0f, 2.0f), x);
        const float2 y2 = __fmul2_rn(make_float2(2.0f, 2.0f), y);
        const float2 z2 = __fmul2_rn(make_float2(2.0f, 2.0f), z);
        const float2 u2_0_0 = __fmul2_rn(x, x);
        const float2 u1_1_0 = __fmul2_rn(y, x2);
        const float2 u1_0_1 = __fmul2_rn(z, x2);
        const float2 u0_2_0 = __fmul2_rn(y, y);
        const float2 u0_1_1 = __fmul2_rn(z, y2);
        const float2 u0_0_2 = __fmul2_rn(z, z);
        const float2 x3 = __fmul2_rn(make_float2(3.0f, 3.0f), x);
        const float2 y3 = __fmul2_rn(make_float2(3.0f, 3.0f), y);
        const float2 z3 = __fmul2_rn(make_float2(3.0f, 3.0f), z);
        const float2 u3_0_0 = __fmul2_rn(u2_0_0, x);
        const float2 u2_1_0 = __fmul2_rn(u2_0_0, y3);
        const float2 u2_0_1 = __fmul2_rn(u2_0_0, z3);
        const float2 u1_2_0 = __fmul2_rn(u0_2_0, x3);
        const float2 u1_1_1 = __fmul2_rn(u0_1_1, x3);
        const float2 u1_0_2 = __fmul2_rn(u0_0_2, x3);
        const float2 u0_3_0 = __fmul2_rn(u0_2_0, y);
        const float2 u0_2_1 = __fmul2_rn(u0_2_0, z3);
        const float2 u0_1_2 = __fmul2_rn(u0_0_2, y3);
        const float2 u0_0_3 = __fmul2_rn(u0_0_2, z);
        gx[0] = gq(0);
        gy[0] = gq(1);
        gz[0] = gq(2);
        gx[1] = __ffma2_rn(gq(5), z, __ffma2_rn(gq(4), y, __fmul2_rn(gq(3), x)));
        gy[1] = __ffma2_rn(gq(7), z, __ffma2_rn(gq(6), y, __fmul2_rn(gq(4), x)));
        gz[1] = __ffma2_rn(gq(8), z, __ffma2_rn(gq(7), y, __fmul2_rn(gq(5), x)));
        gx[2] = __ffma2_rn(gq(14), u0_0_2, __ffma2_rn(gq(13), u0_1_1, __ffma2_rn(gq(12), u0_2_0, __ffma2_rn(gq(11), u1_0_1, __ffma2_rn(gq(10), u1_1_0, __fmul2_rn(gq(9), u2_0_0))))));
        gy[2] = __ffma2_rn(gq(17), u0_0_2, __ffma2_rn(gq(16), u0_1_1, __ffma2_rn(gq(15), u0_2_0, __ffma2_rn(gq(13), u1_0_1, __ffma2_rn(gq(12), u1_1_0, __fmul2_rn(gq(10), u2_0_0))))));
        gz[2] = __ffma2_rn(gq(18), u0_0_2, __ffma2_rn(gq(17), u0_1_1, __ffma2_rn(gq(16), u0_2_0, __ffma2_rn(gq(14), u1_0_1, __ffma2_rn(gq(13), u1_1_0, __fmul2_rn(gq(11), u2_0_0))))));
        gx[3] = __ffma2_rn(gq(28), u0_0_3, __ffma2_rn(gq(27), u0_1_2, __ffma2_rn(gq(26), u0_2_1, __ffma2_rn(gq(25), u0_3_0, __ffma2_rn(gq(24), u1_0_2, __ffma2_rn(gq(23), u1_1_1, __ffma2_rn(gq(22), u1_2_0, __ffma2_rn(gq(21), u2_0_1, __ffma2_rn(gq(20), u2_1_0, __fmul2_rn(gq(19), u3_0_0))))))))));
        gy[3] = __ffma2_rn(gq(32), u0_0_3, __ffma2_rn(gq(31), u0_1_2, __ffma2_rn(gq(30), u0_2_1, __ffma2_rn(gq(29), u0_3_0, __ffma2_rn(gq(27), u1_0_2, __ffma2_rn(gq(26), u1_1_1, __ffma2_rn(gq(25), u1_2_0, __ffma2_rn(gq(23), u2_0_1, __ffma2_rn(gq(22), u2_1_0, __fmul2_rn(gq(20), u3_0_0))))))))));
        gz[3] = __ffma2_rn(gq(33), u0_0_3, __ffma2_rn(gq(32), u0_1_2, __ffma2_rn(gq(31), u0_2_1, __ffma2_rn(gq(30), u0_3_0, __ffma2_rn(gq(28), u1_0_2, __ffma2_rn(gq(27), u1_1_1, __ffma2_rn(gq(26), u1_2_0, __ffma2_rn(gq(24), u2_0_1, __ffma2_rn(gq(23), u2_1_0, __fmul2_rn(gq(21), u3_0_0))))))))));
    }
    __device__ __forceinline__ static void mul(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[24] * b[24], fmaf(0.282094806432724f, a[20] * b[20], fmaf(0.282094806432724f, a[16] * b[16], fmaf(0.282094806432724f, a[12] * b[12], fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])))))) + fmaf(0.282094806432724f, a[21] * b[21], fmaf(0.282094806432724f, a[17] * b[17], fmaf(0.282094806432724f, a[13] * b[13], fmaf(0.282094806432724f, a[9] * b[9], fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])))))) + (fmaf(0.282094806432724f, a[22] * b[22], fmaf(0.282094806432724f, a[18] * b[18], fmaf(0.282094806432724f, a[14] * b[14], fmaf(0.282094806432724f, a[10] * b[10], fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]))))) + fmaf(0.282094806432724f, a[23] * b[23], fmaf(0.282094806432724f, a[19] * b[19], fmaf(0.282094806432724f, a[15] * b[15], fmaf(0.282094806432724f, a[11] * b[11], fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])))))));
        o[1] = ((fmaf(0.04352817311882973f, (a[15] * b[18] + a[18] * b[15]), fmaf(0.16858388483524323f, (a[13] * b[18] + a[18] * b[13]), fmaf(-0.1994711458683014f, (a[10] * b[23] + a[23] * b[10]), fmaf(0.05839917063713074f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.18467439711093903f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]))))))) + fmaf(0.1994711458683014f, (a[14] * b[17] + a[17] * b[14]), fmaf(-0.15078601241111755f, (a[11] * b[20] + a[20] * b[11]), fmaf(-0.04352817311882973f, (a[9] * b[22] + a[22] * b[9]), fmaf(0.20230065286159515f, (a[6] * b[11] + a[11] * b[6]), fmaf(-0.05839917063713074f, (a[4] * b[13] + a[13] * b[4]), -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1]))))))) + (fmaf(0.07539300620555878f, (a[14] * b[19] + a[19] * b[14]), fmaf(-0.16858388483524323f, (a[11] * b[22] + a[22] * b[11]), fmaf(-0.23032943904399872f, (a[9] * b[24] + a[24] * b[9]), fmaf(0.18467439711093903f, (a[7] * b[10] + a[10] * b[7]), fmaf(-0.22617901861667633f, (a[4] * b[15] + a[15] * b[4]), -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1])))))) + fmaf(0.23032943904399872f, (a[15] * b[16] + a[16] * b[15]), fmaf(0.1946638971567154f, (a[12] * b[19] + a[19] * b[12]), fmaf(-0.07539300620555878f, (a[10] * b[21] + a[21] * b[10]), fmaf(0.22617901861667633f, (a[8] * b[9] + a[9] * b[8]), fmaf(-0.14304816722869873f, (a[5] * b[12] + a[12] * b[5]), 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2]))))))));
        o[2] = ((fmaf(0.2462325245141983f, (a[12] * b[20] + a[20] * b[12]), fmaf(0.18467439711093903f, (a[8] * b[14] + a[14] * b[8]), fmaf(0.18467439711093903f, (a[4] * b[10] + a[10] * b[4]), 0.282094806432724f * (a[0] * b[2] + a[2] * b[0])))) + fmaf(0.23841361701488495f, (a[13] * b[21] + a[21] * b[13]), fmaf(0.1628675013780594f, (a[9] * b[17] + a[17] * b[9]), fmaf(0.23359668254852295f, (a[5] * b[11] + a[11] * b[5]), 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))))) + (fmaf(0.21324361860752106f, (a[14] * b[22] + a[22] * b[14]), fmaf(0.21324361860752106f, (a[10] * b[18] + a[18] * b[10]), fmaf(0.24776668846607208f, (a[6] * b[12] + a[12] * b[6]), 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])))) + fmaf(0.1628675013780594f, (a[15] * b[23] + a[23] * b[15]), fmaf(0.23841361701488495f, (a[11] * b[19] + a[19] * b[11]), fmaf(0.23359668254852295f, (a[7] * b[13] + a[13] * b[7]), 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))))));
        o[3] = ((fmaf(0.23032943904399872f, (a[15] * b[24] + a[24] * b[15]), fmaf(0.16858388483524323f, (a[13] * b[22] + a[22] * b[13]), fmaf(-0.07539300620555878f, (a[10] * b[19] + a[19] * b[10]), fmaf(0.22617901861667633f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.20230065286159515f, (a[6] * b[13] + a[13] * b[6]), fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]))))))) + fmaf(-0.07539300620555878f, (a[14] * b[21] + a[21] * b[14]), fmaf(0.16858388483524323f, (a[11] * b[18] + a[18] * b[11]), fmaf(0.23032943904399872f, (a[9] * b[16] + a[16] * b[9]), fmaf(-0.14304816722869873f, (a[7] * b[12] + a[12] * b[7]), fmaf(0.22617901861667633f, (a[4] * b[9] + a[9] * b[4]), 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1]))))))) + (fmaf(0.1994711458683014f, (a[14] * b[23] + a[23] * b[14]), fmaf(0.1946638971567154f, (a[12] * b[21] + a[21] * b[12]), fmaf(-0.04352817311882973f, (a[9] * b[18] + a[18] * b[9]), fmaf(0.18467439711093903f, (a[7] * b[14] + a[14] * b[7]), fmaf(-0.05839917063713074f, (a[4] * b[11] + a[11] * b[4]), 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2])))))) + fmaf(-0.04352817311882973f, (a[15] * b[22] + a[22] * b[15]), fmaf(-0.15078601241111755f, (a[13] * b[20] + a[20] * b[13]), fmaf(0.1994711458683014f, (a[10] * b[17] + a[17] * b[10]), fmaf(-0.05839917063713074f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.18467439711093903f, (a[5] * b[10] + a[10] * b[5]), -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3]))))))));
        o[4] = ((fmaf(0.07508081942796707f, (a[18] * b[24] + a[24] * b[18]), fmaf(0.09403159469366074f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.23841361701488495f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.16858388483524323f, (a[5] * b[23] + a[23] * b[5]), fmaf(0.04029925540089607f, (a[4] * b[20] + a[20] * b[4]), fmaf(0.18467439711093903f, (a[2] * b[10] + a[10] * b[2]), 0.282094806432724f * (a[0] * b[4] + a[4] * b[0]))))))) + fmaf(0.14188940823078156f, (a[19] * b[21] + a[21] * b[19]), fmaf(-0.07508081942796707f, (a[16] * b[22] + a[22] * b[16]), fmaf(-0.09403159469366074f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.15607835352420807f, (a[6] * b[18] + a[18] * b[6]), fmaf(-0.23841361701488495f, (a[4] * b[24] + a[24] * b[4]), fmaf(0.22617901861667633f, (a[3] * b[9] + a[9] * b[3]), 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])))))))) + (fmaf(0.11262122541666031f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.11262122541666031f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.18806318938732147f, (a[10] * b[12] + a[12] * b[10]), fmaf(0.16858388483524323f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[11] + a[11] * b[3]), -0.05839917063713074f * (a[1] * b[13] + a[13] * b[1]))))))) + fmaf(-0.19036461412906647f, (a[18] * b[20] + a[20] * b[18]), fmaf(0.14567312598228455f, (a[11] * b[13] + a[13] * b[11]), fmaf(-0.06371872127056122f, (a[7] * b[19] + a[19] * b[7]), fmaf(-0.06371872127056122f, (a[5] * b[21] + a[21] * b[5]), fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * (a[1] * b[15] + a[15] * b[1]))))))));
        o[5] = ((fmaf(-0.09029786288738251f, (a[19] * b[22] + a[22] * b[19]), fmaf(-0.14046335220336914f, (a[17] * b[24] + a[24] * b[17]), fmaf(0.059470802545547485f, (a[11] * b[12] + a[12] * b[11]), fmaf(0.06371872127056122f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.180223748087883f, (a[5] * b[22] + a[22] * b[5]), fmaf(-0.16858388483524323f, (a[4] * b[23] + a[23] * b[4]), fmaf(0.23359668254852295f, (a[2] * b[11] + a[11] * b[2]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])))))))) + fmaf(0.09029786288738251f, (a[18] * b[21] + a[21] * b[18]), fmaf(-0.11516471952199936f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.1486770063638687f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.22072811424732208f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[10] + a[10] * b[3]), 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1])))))))) + (fmaf(-0.13272538781166077f, (a[18] * b[23] + a[23] * b[18]), fmaf(0.14046335220336914f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.11516471952199936f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.180223748087883f, (a[7] * b[18] + a[18] * b[7]), fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * (a[1] * b[12] + a[12] * b[1]))))))) + fmaf(0.04486937075853348f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.13272538781166077f, (a[17] * b[22] + a[22] * b[17]), fmaf(-0.1486770063638687f, (a[10] * b[15] + a[15] * b[10]), fmaf(0.16858388483524323f, (a[8] * b[17] + a[17] * b[8]), fmaf(-0.1611970216035843f, (a[5] * b[20] + a[20] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[21] + a[21] * b[4]), -0.18467439711093903f * (a[1] * b[14] + a[14] * b[1])))))))));
        o[6] = ((fmaf(0.06553591042757034f, a[22] * b[22], fmaf(0.06553591042757034f, a[18] * b[18], fmaf(0.12615662813186646f, a[13] * b[13], fmaf(0.15607835352420807f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.24179553985595703f, (a[6] * b[20] + a[20] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[18] + a[18] * b[4]), fmaf(0.24776668846607208f, (a[2] * b[12] + a[12] * b[2]), 0.282094806432724f * (a[0] * b[6] + a[6] * b[0])))))))) + fmaf(-0.057343922555446625f, a[23] * b[23], fmaf(0.1392638087272644f, a[19] * b[19], fmaf(-0.2102610468864441f, a[15] * b[15], fmaf(-0.2102610468864441f, a[9] * b[9], fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.0901118740439415f, a[5] * b[5], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1])))))))) + (fmaf(-0.2293756902217865f, a[24] * b[24], fmaf(0.16383977234363556f, a[20] * b[20], fmaf(-0.2293756902217865f, a[16] * b[16], fmaf(0.12615662813186646f, a[11] * b[11], fmaf(0.22072811424732208f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.22072811424732208f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.20230065286159515f, (a[3] * b[13] + a[13] * b[3]), 0.20230065286159515f * (a[1] * b[11] + a[11] * b[1])))))))) + fmaf(0.1392638087272644f, a[21] * b[21], fmaf(-0.057343922555446625f, a[17] * b[17], fmaf(0.16820883750915527f, a[12] * b[12], fmaf(-0.180223748087883f, a[8] * b[8], fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2]))))))));
        o[7] = ((fmaf(0.14046335220336914f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.09029786288738251f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.11516471952199936f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.16858388483524323f, (a[8] * b[23] + a[23] * b[8]), fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.06371872127056122f, (a[4] * b[19] + a[19] * b[4]), fmaf(-0.14304816722869873f, (a[3] * b[12] + a[12] * b[3]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])))))))) + fmaf(0.04486937075853348f, (a[20] * b[21] + a[21] * b[20]), fmaf(0.1486770063638687f, (a[14] * b[15] + a[15] * b[14]), fmaf(0.1486770063638687f, (a[9] * b[10] + a[10] * b[9]), fmaf(-0.1611970216035843f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.180223748087883f, (a[5] * b[18] + a[18] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[14] + a[14] * b[3]), 0.18467439711093903f * (a[1] * b[10] + a[10] * b[1])))))))) + (fmaf(0.09029786288738251f, (a[21] * b[22] + a[22] * b[21]), fmaf(0.14046335220336914f, (a[16] * b[17] + a[17] * b[16]), fmaf(0.11516471952199936f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.180223748087883f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2]))))))) + fmaf(0.13272538781166077f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.13272538781166077f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.059470802545547485f, (a[12] * b[13] + a[13] * b[12]), fmaf(-0.06371872127056122f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.22072811424732208f, (a[6] * b[21] + a[21] * b[6]), fmaf(0.16858388483524323f, (a[4] * b[17] + a[17] * b[4]), 0.23359668254852295f * (a[2] * b[13] + a[13] * b[2])))))))));
        o[8] = ((fmaf(0.14188940823078156f, a[21] * b[21], fmaf(-0.07508081942796707f, (a[16] * b[18] + a[18] * b[16]), fmaf(-0.14567312598228455f, a[11] * b[11], fmaf(0.16858388483524323f, (a[7] * b[23] + a[23] * b[7]), fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.23841361701488495f, (a[4] * b[16] + a[16] * b[4]), fmaf(0.18467439711093903f, (a[2] * b[14] + a[14] * b[2]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])))))))) + fmaf(-0.11262122541666031f, (a[21] * b[23] + a[23] * b[21]), fmaf(-0.11262122541666031f, (a[17] * b[19] + a[19] * b[17]), fmaf(-0.18806318938732147f, (a[12] * b[14] + a[14] * b[12]), fmaf(0.04029925540089607f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.15607835352420807f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1])))))))) + (fmaf(-0.07508081942796707f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.14188940823078156f, a[19] * b[19], fmaf(0.14567312598228455f, a[13] * b[13], fmaf(0.23841361701488495f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.15607835352420807f, a[7] * b[7], fmaf(0.16858388483524323f, (a[5] * b[17] + a[17] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[13] + a[13] * b[3]), 0.22617901861667633f * (a[1] * b[9] + a[9] * b[1])))))))) + fmaf(-0.19036461412906647f, (a[20] * b[22] + a[22] * b[20]), fmaf(-0.09403159469366074f, (a[13] * b[15] + a[15] * b[13]), fmaf(-0.09403159469366074f, (a[9] * b[11] + a[11] * b[9]), fmaf(-0.06371872127056122f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.22617901861667633f, (a[3] * b[15] + a[15] * b[3]), 0.05839917063713074f * (a[1] * b[11] + a[11] * b[1])))))))));
        o[9] = ((fmaf(-0.09932258725166321f, (a[14] * b[19] + a[19] * b[14]), fmaf(0.11752006411552429f, (a[11] * b[24] + a[24] * b[11]), fmaf(-0.09403159469366074f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.09403159469366074f, (a[4] * b[13] + a[13] * b[4]), fmaf(0.1628675013780594f, (a[2] * b[17] + a[17] * b[2]), 0.282094806432724f * (a[0] * b[9] + a[9] * b[0])))))) + fmaf(-0.20355072617530823f, (a[12] * b[17] + a[17] * b[12]), fmaf(0.07693494111299515f, (a[9] * b[20] + a[20] * b[9]), fmaf(0.1486770063638687f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.22617901861667633f, (a[3] * b[4] + a[4] * b[3]), 0.22617901861667633f * (a[1] * b[8] + a[8] * b[1])))))) + (fmaf(-0.11752006411552429f, (a[13] * b[16] + a[16] * b[13]), fmaf(-0.09932258725166321f, (a[10] * b[21] + a[21] * b[10]), fmaf(-0.2102610468864441f, (a[6] * b[9] + a[9] * b[6]), fmaf(0.23032943904399872f, (a[3] * b[16] + a[16] * b[3]), -0.04352817311882973f * (a[1] * b[22] + a[22] * b[1]))))) + fmaf(0.1332552284002304f, (a[13] * b[18] + a[18] * b[13]), fmaf(0.1332552284002304f, (a[11] * b[22] + a[22] * b[11]), fmaf(0.1486770063638687f, (a[7] * b[10] + a[10] * b[7]), fmaf(-0.04352817311882973f, (a[3] * b[18] + a[18] * b[3]), -0.23032943904399872f * (a[1] * b[24] + a[24] * b[1])))))));
        o[10] = ((fmaf(0.06785023957490921f, (a[13] * b[17] + a[17] * b[13]), fmaf(-0.15171775221824646f, (a[10] * b[24] + a[24] * b[10]), fmaf(0.1486770063638687f, (a[7] * b[9] + a[9] * b[7]), fmaf(-0.07539300620555878f, (a[3] * b[19] + a[19] * b[3]), fmaf(0.18467439711093903f, (a[2] * b[4] + a[4] * b[2]), 0.282094806432724f * (a[0] * b[10] + a[10] * b[0])))))) + fmaf(0.10257992148399353f, (a[13] * b[19] + a[19] * b[13]), fmaf(0.10257992148399353f, (a[11] * b[21] + a[21] * b[11]), fmaf(0.11516471952199936f, (a[7] * b[11] + a[11] * b[7]), fmaf(-0.18806318938732147f, (a[4] * b[12] + a[12] * b[4]), fmaf(0.21324361860752106f, (a[2] * b[18] + a[18] * b[2]), 0.18467439711093903f * (a[1] * b[7] + a[7] * b[1]))))))) + (fmaf(0.15171775221824646f, (a[14] * b[16] + a[16] * b[14]), fmaf(-0.06785023957490921f, (a[11] * b[23] + a[23] * b[11]), fmaf(-0.09932258725166321f, (a[9] * b[21] + a[21] * b[9]), fmaf(0.11516471952199936f, (a[5] * b[13] + a[13] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[5] + a[5] * b[3]), -0.07539300620555878f * (a[1] * b[21] + a[21] * b[1])))))) + fmaf(0.09932258725166321f, (a[15] * b[19] + a[19] * b[15]), fmaf(-0.04441840946674347f, (a[12] * b[18] + a[18] * b[12]), fmaf(-0.17951487004756927f, (a[10] * b[20] + a[20] * b[10]), fmaf(-0.1486770063638687f, (a[5] * b[15] + a[15] * b[5]), fmaf(0.1994711458683014f, (a[3] * b[17] + a[17] * b[3]), -0.1994711458683014f * (a[1] * b[23] + a[23] * b[1]))))))));
        o[11] = ((fmaf(-0.1332552284002304f, (a[15] * b[18] + a[18] * b[15]), fmaf(0.11468784511089325f, (a[13] * b[18] + a[18] * b[13]), fmaf(-0.06785023957490921f, (a[10] * b[23] + a[23] * b[10]), fmaf(-0.14567312598228455f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.11516471952199936f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.16858388483524323f, (a[3] * b[18] + a[18] * b[3]), fmaf(-0.16858388483524323f, (a[1] * b[22] + a[22] * b[1]), 0.282094806432724f * (a[0] * b[11] + a[11] * b[0])))))))) + fmaf(0.06785023957490921f, (a[14] * b[17] + a[17] * b[14]), fmaf(0.025644980370998383f, (a[11] * b[20] + a[20] * b[11]), fmaf(0.1332552284002304f, (a[9] * b[22] + a[22] * b[9]), fmaf(0.12615662813186646f, (a[6] * b[11] + a[11] * b[6]), fmaf(0.14567312598228455f, (a[4] * b[13] + a[13] * b[4]), fmaf(0.23359668254852295f, (a[2] * b[5] + a[5] * b[2]), 0.20230065286159515f * (a[1] * b[6] + a[6] * b[1])))))))) + (fmaf(-0.10257992148399353f, (a[14] * b[19] + a[19] * b[14]), fmaf(-0.11468784511089325f, (a[11] * b[22] + a[22] * b[11]), fmaf(0.11752006411552429f, (a[9] * b[24] + a[24] * b[9]), fmaf(0.11516471952199936f, (a[7] * b[10] + a[10] * b[7]), fmaf(0.09403159469366074f, (a[4] * b[15] + a[15] * b[4]), fmaf(0.23841361701488495f, (a[2] * b[19] + a[19] * b[2]), 0.05839917063713074f * (a[1] * b[8] + a[8] * b[1]))))))) + fmaf(-0.11752006411552429f, (a[15] * b[16] + a[16] * b[15]), fmaf(0.09932258725166321f, (a[12] * b[19] + a[19] * b[12]), fmaf(0.10257992148399353f, (a[10] * b[21] + a[21] * b[10]), fmaf(-0.09403159469366074f, (a[8] * b[9] + a[9] * b[8]), fmaf(0.059470802545547485f, (a[5] * b[12] + a[12] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[4] + a[4] * b[3]), -0.15078601241111755f * (a[1] * b[20] + a[20] * b[1])))))))));
        o[12] = ((fmaf(0.09932258725166321f, (a[13] * b[21] + a[21] * b[13]), fmaf(-0.20355072617530823f, (a[9] * b[17] + a[17] * b[9]), fmaf(0.059470802545547485f, (a[5] * b[11] + a[11] * b[5]), fmaf(0.2462325245141983f, (a[2] * b[20] + a[20] * b[2]), 0.282094806432724f * (a[0] * b[12] + a[12] * b[0]))))) + fmaf(-0.04441840946674347f, (a[14] * b[22] + a[22] * b[14]), fmaf(-0.04441840946674347f, (a[10] * b[18] + a[18] * b[10]), fmaf(0.16820883750915527f, (a[6] * b[12] + a[12] * b[6]), fmaf(-0.14304816722869873f, (a[3] * b[7] + a[7] * b[3]), -0.14304816722869873f * (a[1] * b[5] + a[5] * b[1])))))) + (fmaf(-0.20355072617530823f, (a[15] * b[23] + a[23] * b[15]), fmaf(0.09932258725166321f, (a[11] * b[19] + a[19] * b[11]), fmaf(0.059470802545547485f, (a[7] * b[13] + a[13] * b[7]), fmaf(0.1946638971567154f, (a[3] * b[21] + a[21] * b[3]), 0.1946638971567154f * (a[1] * b[19] + a[19] * b[1]))))) + fmaf(0.1538698822259903f, (a[12] * b[20] + a[20] * b[12]), fmaf(-0.18806318938732147f, (a[8] * b[14] + a[14] * b[8]), fmaf(-0.18806318938732147f, (a[4] * b[10] + a[10] * b[4]), 0.24776668846607208f * (a[2] * b[6] + a[6] * b[2]))))));
        o[13] = ((fmaf(-0.11752006411552429f, (a[15] * b[24] + a[24] * b[15]), fmaf(0.11468784511089325f, (a[13] * b[22] + a[22] * b[13]), fmaf(0.10257992148399353f, (a[10] * b[19] + a[19] * b[10]), fmaf(-0.09403159469366074f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.12615662813186646f, (a[6] * b[13] + a[13] * b[6]), fmaf(0.16858388483524323f, (a[3] * b[22] + a[22] * b[3]), fmaf(0.23841361701488495f, (a[2] * b[21] + a[21] * b[2]), 0.282094806432724f * (a[0] * b[13] + a[13] * b[0])))))))) + fmaf(0.10257992148399353f, (a[14] * b[21] + a[21] * b[14]), fmaf(0.11468784511089325f, (a[11] * b[18] + a[18] * b[11]), fmaf(-0.11752006411552429f, (a[9] * b[16] + a[16] * b[9]), fmaf(0.059470802545547485f, (a[7] * b[12] + a[12] * b[7]), fmaf(-0.09403159469366074f, (a[4] * b[9] + a[9] * b[4]), fmaf(0.20230065286159515f, (a[3] * b[6] + a[6] * b[3]), -0.05839917063713074f * (a[1] * b[4] + a[4] * b[1])))))))) + (fmaf(0.06785023957490921f, (a[14] * b[23] + a[23] * b[14]), fmaf(0.09932258725166321f, (a[12] * b[21] + a[21] * b[12]), fmaf(0.1332552284002304f, (a[9] * b[18] + a[18] * b[9]), fmaf(0.11516471952199936f, (a[7] * b[14] + a[14] * b[7]), fmaf(0.14567312598228455f, (a[4] * b[11] + a[11] * b[4]), fmaf(-0.05839917063713074f, (a[3] * b[8] + a[8] * b[3]), 0.16858388483524323f * (a[1] * b[18] + a[18] * b[1]))))))) + fmaf(0.1332552284002304f, (a[15] * b[22] + a[22] * b[15]), fmaf(0.025644980370998383f, (a[13] * b[20] + a[20] * b[13]), fmaf(0.06785023957490921f, (a[10] * b[17] + a[17] * b[10]), fmaf(0.14567312598228455f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.11516471952199936f, (a[5] * b[10] + a[10] * b[5]), fmaf(-0.15078601241111755f, (a[3] * b[20] + a[20] * b[3]), 0.23359668254852295f * (a[2] * b[7] + a[7] * b[2])))))))));
        o[14] = ((fmaf(0.06785023957490921f, (a[13] * b[23] + a[23] * b[13]), fmaf(0.06785023957490921f, (a[11] * b[17] + a[17] * b[11]), fmaf(0.1486770063638687f, (a[7] * b[15] + a[15] * b[7]), fmaf(0.1994711458683014f, (a[3] * b[23] + a[23] * b[3]), fmaf(0.18467439711093903f, (a[2] * b[8] + a[8] * b[2]), 0.282094806432724f * (a[0] * b[14] + a[14] * b[0])))))) + fmaf(-0.17951487004756927f, (a[14] * b[20] + a[20] * b[14]), fmaf(-0.10257992148399353f, (a[11] * b[19] + a[19] * b[11]), fmaf(-0.18806318938732147f, (a[8] * b[12] + a[12] * b[8]), fmaf(0.1486770063638687f, (a[5] * b[9] + a[9] * b[5]), fmaf(0.21324361860752106f, (a[2] * b[22] + a[22] * b[2]), -0.18467439711093903f * (a[1] * b[5] + a[5] * b[1]))))))) + (fmaf(0.15171775221824646f, (a[14] * b[24] + a[24] * b[14]), fmaf(-0.04441840946674347f, (a[12] * b[22] + a[22] * b[12]), fmaf(-0.09932258725166321f, (a[9] * b[19] + a[19] * b[9]), fmaf(-0.11516471952199936f, (a[5] * b[11] + a[11] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[7] + a[7] * b[3]), 0.1994711458683014f * (a[1] * b[17] + a[17] * b[1])))))) + fmaf(-0.09932258725166321f, (a[15] * b[21] + a[21] * b[15]), fmaf(0.10257992148399353f, (a[13] * b[21] + a[21] * b[13]), fmaf(0.15171775221824646f, (a[10] * b[16] + a[16] * b[10]), fmaf(0.11516471952199936f, (a[7] * b[13] + a[13] * b[7]), fmaf(-0.07539300620555878f, (a[3] * b[21] + a[21] * b[3]), 0.07539300620555878f * (a[1] * b[19] + a[19] * b[1]))))))));
        o[15] = ((fmaf(0.07693494111299515f, (a[15] * b[20] + a[20] * b[15]), fmaf(-0.20355072617530823f, (a[12] * b[23] + a[23] * b[12]), fmaf(-0.09403159469366074f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.09403159469366074f, (a[4] * b[11] + a[11] * b[4]), fmaf(0.1628675013780594f, (a[2] * b[23] + a[23] * b[2]), 0.282094806432724f * (a[0] * b[15] + a[15] * b[0])))))) + fmaf(0.1332552284002304f, (a[13] * b[22] + a[22] * b[13]), fmaf(0.09932258725166321f, (a[10] * b[19] + a[19] * b[10]), fmaf(-0.1486770063638687f, (a[5] * b[10] + a[10] * b[5]), fmaf(0.22617901861667633f, (a[3] * b[8] + a[8] * b[3]), -0.22617901861667633f * (a[1] * b[4] + a[4] * b[1])))))) + (fmaf(-0.11752006411552429f, (a[13] * b[24] + a[24] * b[13]), fmaf(-0.11752006411552429f, (a[11] * b[16] + a[16] * b[11]), fmaf(-0.2102610468864441f, (a[6] * b[15] + a[15] * b[6]), fmaf(-0.04352817311882973f, (a[3] * b[22] + a[22] * b[3]), 0.23032943904399872f * (a[1] * b[16] + a[16] * b[1]))))) + fmaf(-0.09932258725166321f, (a[14] * b[21] + a[21] * b[14]), fmaf(-0.1332552284002304f, (a[11] * b[18] + a[18] * b[11]), fmaf(0.1486770063638687f, (a[7] * b[14] + a[14] * b[7]), fmaf(0.23032943904399872f, (a[3] * b[24] + a[24] * b[3]), 0.04352817311882973f * (a[1] * b[18] + a[18] * b[1])))))));
        o[16] = ((fmaf(0.10652530938386917f, (a[16] * b[20] + a[20] * b[16]), fmaf(-0.07508081942796707f, (a[8] * b[18] + a[18] * b[8]), fmaf(-0.07508081942796707f, (a[4] * b[22] + a[22] * b[4]), 0.282094806432724f * (a[0] * b[16] + a[16] * b[0])))) + fmaf(-0.11909890919923782f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.11752006411552429f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.14046335220336914f, (a[5] * b[23] + a[23] * b[5]), 0.23032943904399872f * (a[1] * b[15] + a[15] * b[1]))))) + (fmaf(0.13504546880722046f, (a[18] * b[22] + a[22] * b[18]), fmaf(0.15171775221824646f, (a[10] * b[14] + a[14] * b[10]), fmaf(-0.2293756902217865f, (a[6] * b[16] + a[16] * b[6]), 0.23032943904399872f * (a[3] * b[9] + a[9] * b[3])))) + fmaf(-0.11909890919923782f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.11752006411552429f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.14046335220336914f, (a[7] * b[17] + a[17] * b[7]), 0.23841361701488495f * (a[4] * b[8] + a[8] * b[4]))))));
        o[17] = ((fmaf(0.11909890919923782f, (a[19] * b[24] + a[24] * b[19]), fmaf(-0.11909890919923782f, (a[16] * b[21] + a[21] * b[16]), fmaf(-0.11262122541666031f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[24] + a[24] * b[5]), fmaf(0.16858388483524323f, (a[4] * b[7] + a[7] * b[4]), 0.282094806432724f * (a[0] * b[17] + a[17] * b[0])))))) + fmaf(-0.15978795289993286f, (a[17] * b[20] + a[20] * b[17]), fmaf(-0.20355072617530823f, (a[9] * b[12] + a[12] * b[9]), fmaf(-0.057343922555446625f, (a[6] * b[17] + a[17] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[21] + a[21] * b[4]), 0.1994711458683014f * (a[1] * b[14] + a[14] * b[1])))))) + (fmaf(0.045015156269073486f, (a[18] * b[21] + a[21] * b[18]), fmaf(0.06785023957490921f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.14046335220336914f, (a[7] * b[16] + a[16] * b[7]), fmaf(0.16858388483524323f, (a[5] * b[8] + a[8] * b[5]), 0.1628675013780594f * (a[2] * b[9] + a[9] * b[2]))))) + fmaf(0.045015156269073486f, (a[19] * b[22] + a[22] * b[19]), fmaf(0.06785023957490921f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.13272538781166077f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.13272538781166077f, (a[5] * b[22] + a[22] * b[5]), 0.1994711458683014f * (a[3] * b[10] + a[10] * b[3])))))));
        o[18] = ((fmaf(0.10208478569984436f, (a[19] * b[21] + a[21] * b[19]), fmaf(0.13504546880722046f, (a[16] * b[22] + a[22] * b[16]), fmaf(0.1332552284002304f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.06553591042757034f, (a[6] * b[18] + a[18] * b[6]), fmaf(0.07508081942796707f, (a[4] * b[24] + a[24] * b[4]), fmaf(-0.04352817311882973f, (a[3] * b[9] + a[9] * b[3]), 0.282094806432724f * (a[0] * b[18] + a[18] * b[0]))))))) + fmaf(-0.045015156269073486f, (a[19] * b[23] + a[23] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.04441840946674347f, (a[10] * b[12] + a[12] * b[10]), fmaf(0.13272538781166077f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.180223748087883f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.16858388483524323f, (a[3] * b[11] + a[11] * b[3]), 0.16858388483524323f * (a[1] * b[13] + a[13] * b[1])))))))) + (fmaf(-0.08369845151901245f, (a[18] * b[20] + a[20] * b[18]), fmaf(0.11468784511089325f, (a[11] * b[13] + a[13] * b[11]), fmaf(0.09029786288738251f, (a[7] * b[19] + a[19] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[21] + a[21] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[6] + a[6] * b[4]), 0.04352817311882973f * (a[1] * b[15] + a[15] * b[1])))))) + fmaf(-0.13504546880722046f, (a[18] * b[24] + a[24] * b[18]), fmaf(-0.1332552284002304f, (a[11] * b[15] + a[15] * b[11]), fmaf(-0.07508081942796707f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.13272538781166077f, (a[5] * b[23] + a[23] * b[5]), fmaf(-0.19036461412906647f, (a[4] * b[20] + a[20] * b[4]), 0.21324361860752106f * (a[2] * b[10] + a[10] * b[2]))))))));
        o[19] = ((fmaf(0.10208478569984436f, (a[18] * b[21] + a[21] * b[18]), fmaf(-0.10257992148399353f, (a[11] * b[14] + a[14] * b[11]), fmaf(-0.09932258725166321f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.1392638087272644f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.22072811424732208f, (a[5] * b[6] + a[6] * b[5]), fmaf(-0.07539300620555878f, (a[3] * b[10] + a[10] * b[3]), 0.282094806432724f * (a[0] * b[19] + a[19] * b[0]))))))) + fmaf(-0.045015156269073486f, (a[18] * b[23] + a[23] * b[18]), fmaf(-0.11909890919923782f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.10257992148399353f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.09029786288738251f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[8] + a[8] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[7] + a[7] * b[4]), 0.1946638971567154f * (a[1] * b[12] + a[12] * b[1])))))))) + (fmaf(0.06848055124282837f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[22] + a[22] * b[17]), fmaf(0.09932258725166321f, (a[10] * b[15] + a[15] * b[10]), fmaf(-0.11262122541666031f, (a[8] * b[17] + a[17] * b[8]), fmaf(0.04486937075853348f, (a[5] * b[20] + a[20] * b[5]), fmaf(0.14188940823078156f, (a[4] * b[21] + a[21] * b[4]), 0.07539300620555878f * (a[1] * b[14] + a[14] * b[1]))))))) + fmaf(-0.10208478569984436f, (a[19] * b[22] + a[22] * b[19]), fmaf(0.11909890919923782f, (a[17] * b[24] + a[24] * b[17]), fmaf(0.09932258725166321f, (a[11] * b[12] + a[12] * b[11]), fmaf(-0.14188940823078156f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.09029786288738251f, (a[5] * b[22] + a[22] * b[5]), fmaf(0.11262122541666031f, (a[4] * b[23] + a[23] * b[4]), 0.23841361701488495f * (a[2] * b[11] + a[11] * b[2])))))))));
        o[20] = ((fmaf(-0.15978795289993286f, a[23] * b[23], fmaf(0.06848055124282837f, a[19] * b[19], fmaf(0.07693494111299515f, a[15] * b[15], fmaf(0.025644980370998383f, a[11] * b[11], fmaf(0.04029925540089607f, a[8] * b[8], fmaf(0.24179553985595703f, a[6] * b[6], fmaf(0.04029925540089607f, a[4] * b[4], 0.282094806432724f * (a[0] * b[20] + a[20] * b[0])))))))) + fmaf(0.10652530938386917f, a[24] * b[24], fmaf(0.13696110248565674f, a[20] * b[20], fmaf(0.10652530938386917f, a[16] * b[16], fmaf(0.1538698822259903f, a[12] * b[12], fmaf(-0.19036461412906647f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.16383977234363556f, (a[6] * b[20] + a[20] * b[6]), fmaf(-0.19036461412906647f, (a[4] * b[18] + a[18] * b[4]), -0.15078601241111755f * (a[1] * b[11] + a[11] * b[1]))))))))) + (fmaf(0.06848055124282837f, a[21] * b[21], fmaf(-0.15978795289993286f, a[17] * b[17], fmaf(0.025644980370998383f, a[13] * b[13], fmaf(0.07693494111299515f, a[9] * b[9], fmaf(-0.1611970216035843f, a[7] * b[7], fmaf(-0.1611970216035843f, a[5] * b[5], 0.2462325245141983f * (a[2] * b[12] + a[12] * b[2]))))))) + fmaf(-0.08369845151901245f, a[22] * b[22], fmaf(-0.08369845151901245f, a[18] * b[18], fmaf(-0.17951487004756927f, a[14] * b[14], fmaf(-0.17951487004756927f, a[10] * b[10], fmaf(0.04486937075853348f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.04486937075853348f, (a[5] * b[19] + a[19] * b[5]), -0.15078601241111755f * (a[3] * b[13] + a[13] * b[3])))))))));
        o[21] = ((fmaf(0.06848055124282837f, (a[20] * b[21] + a[21] * b[20]), fmaf(-0.09932258725166321f, (a[14] * b[15] + a[15] * b[14]), fmaf(-0.09932258725166321f, (a[9] * b[10] + a[10] * b[9]), fmaf(0.04486937075853348f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[18] + a[18] * b[5]), fmaf(-0.07539300620555878f, (a[3] * b[14] + a[14] * b[3]), 0.282094806432724f * (a[0] * b[21] + a[21] * b[0]))))))) + fmaf(0.10208478569984436f, (a[21] * b[22] + a[22] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[17] + a[17] * b[16]), fmaf(0.10257992148399353f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.09029786288738251f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.22072811424732208f, (a[6] * b[7] + a[7] * b[6]), fmaf(-0.06371872127056122f, (a[4] * b[5] + a[5] * b[4]), -0.07539300620555878f * (a[1] * b[10] + a[10] * b[1])))))))) + (fmaf(0.045015156269073486f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.045015156269073486f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.09932258725166321f, (a[12] * b[13] + a[13] * b[12]), fmaf(0.14188940823078156f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.1392638087272644f, (a[6] * b[21] + a[21] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[17] + a[17] * b[4]), 0.23841361701488495f * (a[2] * b[13] + a[13] * b[2]))))))) + fmaf(-0.11909890919923782f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.10208478569984436f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.10257992148399353f, (a[13] * b[14] + a[14] * b[13]), fmaf(-0.11262122541666031f, (a[8] * b[23] + a[23] * b[8]), fmaf(-0.06371872127056122f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.14188940823078156f, (a[4] * b[19] + a[19] * b[4]), 0.1946638971567154f * (a[3] * b[12] + a[12] * b[3])))))))));
        o[22] = ((fmaf(0.13504546880722046f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.10208478569984436f, a[19] * b[19], fmaf(0.11468784511089325f, a[13] * b[13], fmaf(-0.07508081942796707f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.180223748087883f, a[7] * b[7], fmaf(0.13272538781166077f, (a[5] * b[17] + a[17] * b[5]), fmaf(0.16858388483524323f, (a[3] * b[13] + a[13] * b[3]), 0.282094806432724f * (a[0] * b[22] + a[22] * b[0])))))))) + fmaf(-0.08369845151901245f, (a[20] * b[22] + a[22] * b[20]), fmaf(0.1332552284002304f, (a[13] * b[15] + a[15] * b[13]), fmaf(0.1332552284002304f, (a[9] * b[11] + a[11] * b[9]), fmaf(0.09029786288738251f, (a[7] * b[21] + a[21] * b[7]), fmaf(-0.09029786288738251f, (a[5] * b[19] + a[19] * b[5]), fmaf(-0.04352817311882973f, (a[3] * b[15] + a[15] * b[3]), -0.04352817311882973f * (a[1] * b[9] + a[9] * b[1])))))))) + (fmaf(0.10208478569984436f, a[21] * b[21], fmaf(0.13504546880722046f, (a[16] * b[18] + a[18] * b[16]), fmaf(-0.11468784511089325f, a[11] * b[11], fmaf(0.13272538781166077f, (a[7] * b[23] + a[23] * b[7]), fmaf(0.15607835352420807f, (a[6] * b[8] + a[8] * b[6]), fmaf(-0.07508081942796707f, (a[4] * b[16] + a[16] * b[4]), -0.16858388483524323f * (a[1] * b[11] + a[11] * b[1]))))))) + fmaf(0.045015156269073486f, (a[21] * b[23] + a[23] * b[21]), fmaf(0.045015156269073486f, (a[17] * b[19] + a[19] * b[17]), fmaf(-0.04441840946674347f, (a[12] * b[14] + a[14] * b[12]), fmaf(-0.19036461412906647f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.06553591042757034f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.180223748087883f, a[5] * b[5], 0.21324361860752106f * (a[2] * b[14] + a[14] * b[2])))))))));
        o[23] = ((fmaf(-0.11909890919923782f, (a[21] * b[24] + a[24] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[19] + a[19] * b[16]), fmaf(-0.11262122541666031f, (a[8] * b[21] + a[21] * b[8]), fmaf(-0.057343922555446625f, (a[6] * b[23] + a[23] * b[6]), fmaf(-0.16858388483524323f, (a[4] * b[5] + a[5] * b[4]), 0.282094806432724f * (a[0] * b[23] + a[23] * b[0])))))) + fmaf(-0.045015156269073486f, (a[18] * b[19] + a[19] * b[18]), fmaf(-0.06785023957490921f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.16858388483524323f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.11262122541666031f, (a[4] * b[19] + a[19] * b[4]), -0.1994711458683014f * (a[1] * b[10] + a[10] * b[1])))))) + (fmaf(-0.15978795289993286f, (a[20] * b[23] + a[23] * b[20]), fmaf(-0.20355072617530823f, (a[12] * b[15] + a[15] * b[12]), fmaf(0.13272538781166077f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.14046335220336914f, (a[5] * b[16] + a[16] * b[5]), 0.1628675013780594f * (a[2] * b[15] + a[15] * b[2]))))) + fmaf(0.045015156269073486f, (a[21] * b[22] + a[22] * b[21]), fmaf(0.06785023957490921f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.14046335220336914f, (a[7] * b[24] + a[24] * b[7]), fmaf(-0.13272538781166077f, (a[5] * b[18] + a[18] * b[5]), 0.1994711458683014f * (a[3] * b[14] + a[14] * b[3])))))));
        o[24] = ((fmaf(0.10652530938386917f, (a[20] * b[24] + a[24] * b[20]), fmaf(-0.11752006411552429f, (a[13] * b[15] + a[15] * b[13]), fmaf(0.23841361701488495f, a[8] * b[8], fmaf(0.07508081942796707f, (a[4] * b[18] + a[18] * b[4]), 0.282094806432724f * (a[0] * b[24] + a[24] * b[0]))))) + fmaf(-0.11909890919923782f, (a[21] * b[23] + a[23] * b[21]), fmaf(0.15171775221824646f, a[14] * b[14], fmaf(-0.07508081942796707f, (a[8] * b[22] + a[22] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[17] + a[17] * b[5]), -0.23032943904399872f * (a[1] * b[9] + a[9] * b[1])))))) + (fmaf(0.13504546880722046f, a[22] * b[22], fmaf(0.11909890919923782f, (a[17] * b[19] + a[19] * b[17]), fmaf(0.11752006411552429f, (a[9] * b[11] + a[11] * b[9]), fmaf(-0.2293756902217865f, (a[6] * b[24] + a[24] * b[6]), 0.23032943904399872f * (a[3] * b[15] + a[15] * b[3]))))) + fmaf(-0.13504546880722046f, a[18] * b[18], fmaf(-0.15171775221824646f, a[10] * b[10], fmaf(0.14046335220336914f, (a[7] * b[23] + a[23] * b[7]), -0.23841361701488495f * a[4] * b[4])))));
    }
    __device__ __forceinline__ static void mul_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[23] * b[23], fmaf(0.282094806432724f, a[19] * b[19], fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])))) + fmaf(0.282094806432724f, a[24] * b[24], fmaf(0.282094806432724f, a[20] * b[20], fmaf(0.282094806432724f, a[16] * b[16], fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1]))))) + (fmaf(0.282094806432724f, a[21] * b[21], fmaf(0.282094806432724f, a[17] * b[17], fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]))) + fmaf(0.282094806432724f, a[22] * b[22], fmaf(0.282094806432724f, a[18] * b[18], fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])))));
        o[1] = ((fmaf(0.04352817311882973f, a[15] * b[18], fmaf(0.16858388483524323f, a[13] * b[18], fmaf(-0.1994711458683014f, a[10] * b[23], fmaf(0.05839917063713074f, a[11] * b[8], fmaf(-0.18467439711093903f, a[14] * b[5], fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]))))))) + fmaf(0.1994711458683014f, a[14] * b[17], fmaf(-0.15078601241111755f, a[11] * b[20], fmaf(-0.04352817311882973f, a[9] * b[22], fmaf(0.20230065286159515f, a[11] * b[6], fmaf(-0.05839917063713074f, a[13] * b[4], -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1]))))))) + (fmaf(0.07539300620555878f, a[14] * b[19], fmaf(-0.16858388483524323f, a[11] * b[22], fmaf(-0.23032943904399872f, a[9] * b[24], fmaf(0.18467439711093903f, a[10] * b[7], fmaf(-0.22617901861667633f, a[15] * b[4], -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1])))))) + fmaf(0.23032943904399872f, a[15] * b[16], fmaf(0.1946638971567154f, a[12] * b[19], fmaf(-0.07539300620555878f, a[10] * b[21], fmaf(0.22617901861667633f, a[9] * b[8], fmaf(-0.14304816722869873f, a[12] * b[5], 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2]))))))));
        o[2] = ((fmaf(0.2462325245141983f, a[12] * b[20], fmaf(0.18467439711093903f, a[14] * b[8], fmaf(0.18467439711093903f, a[10] * b[4], 0.282094806432724f * (a[0] * b[2] + a[2] * b[0])))) + fmaf(0.23841361701488495f, a[13] * b[21], fmaf(0.1628675013780594f, a[9] * b[17], fmaf(0.23359668254852295f, a[11] * b[5], 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))))) + (fmaf(0.21324361860752106f, a[14] * b[22], fmaf(0.21324361860752106f, a[10] * b[18], fmaf(0.24776668846607208f, a[12] * b[6], 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])))) + fmaf(0.1628675013780594f, a[15] * b[23], fmaf(0.23841361701488495f, a[11] * b[19], fmaf(0.23359668254852295f, a[13] * b[7], 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))))));
        o[3] = ((fmaf(0.23032943904399872f, a[15] * b[24], fmaf(0.16858388483524323f, a[13] * b[22], fmaf(-0.07539300620555878f, a[10] * b[19], fmaf(0.22617901861667633f, a[15] * b[8], fmaf(0.20230065286159515f, a[13] * b[6], fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]))))))) + fmaf(-0.07539300620555878f, a[14] * b[21], fmaf(0.16858388483524323f, a[11] * b[18], fmaf(0.23032943904399872f, a[9] * b[16], fmaf(-0.14304816722869873f, a[12] * b[7], fmaf(0.22617901861667633f, a[9] * b[4], 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1]))))))) + (fmaf(0.1994711458683014f, a[14] * b[23], fmaf(0.1946638971567154f, a[12] * b[21], fmaf(-0.04352817311882973f, a[9] * b[18], fmaf(0.18467439711093903f, a[14] * b[7], fmaf(-0.05839917063713074f, a[11] * b[4], 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2])))))) + fmaf(-0.04352817311882973f, a[15] * b[22], fmaf(-0.15078601241111755f, a[13] * b[20], fmaf(0.1994711458683014f, a[10] * b[17], fmaf(-0.05839917063713074f, a[13] * b[8], fmaf(0.18467439711093903f, a[10] * b[5], -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3]))))))));
        o[4] = ((fmaf(0.07508081942796707f, (a[18] * b[24] + a[24] * b[18]), fmaf(0.23841361701488495f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.16858388483524323f, (a[5] * b[23] + a[23] * b[5]), fmaf(0.04029925540089607f, (a[4] * b[20] + a[20] * b[4]), fmaf(0.18467439711093903f, a[10] * b[2], 0.282094806432724f * (a[0] * b[4] + a[4] * b[0])))))) + fmaf(0.14188940823078156f, (a[19] * b[21] + a[21] * b[19]), fmaf(-0.07508081942796707f, (a[16] * b[22] + a[22] * b[16]), fmaf(0.15607835352420807f, (a[6] * b[18] + a[18] * b[6]), fmaf(-0.23841361701488495f, (a[4] * b[24] + a[24] * b[4]), fmaf(0.22617901861667633f, a[9] * b[3], 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1]))))))) + (fmaf(0.11262122541666031f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.11262122541666031f, (a[17] * b[21] + a[21] * b[17]), fmaf(0.16858388483524323f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(-0.05839917063713074f, a[11] * b[3], -0.05839917063713074f * a[13] * b[1]))))) + fmaf(-0.19036461412906647f, (a[18] * b[20] + a[20] * b[18]), fmaf(-0.06371872127056122f, (a[7] * b[19] + a[19] * b[7]), fmaf(-0.06371872127056122f, (a[5] * b[21] + a[21] * b[5]), fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * a[15] * b[1]))))));
        o[5] = ((fmaf(0.09029786288738251f, (a[18] * b[21] + a[21] * b[18]), fmaf(0.06371872127056122f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.180223748087883f, (a[5] * b[22] + a[22] * b[5]), fmaf(-0.16858388483524323f, (a[4] * b[23] + a[23] * b[4]), fmaf(0.23359668254852295f, a[11] * b[2], 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])))))) + fmaf(-0.13272538781166077f, (a[18] * b[23] + a[23] * b[18]), fmaf(0.14046335220336914f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.22072811424732208f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), fmaf(0.18467439711093903f, a[10] * b[3], 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1]))))))) + (fmaf(0.04486937075853348f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.13272538781166077f, (a[17] * b[22] + a[22] * b[17]), fmaf(0.180223748087883f, (a[7] * b[18] + a[18] * b[7]), fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * a[12] * b[1]))))) + fmaf(-0.09029786288738251f, (a[19] * b[22] + a[22] * b[19]), fmaf(-0.14046335220336914f, (a[17] * b[24] + a[24] * b[17]), fmaf(0.16858388483524323f, (a[8] * b[17] + a[17] * b[8]), fmaf(-0.1611970216035843f, (a[5] * b[20] + a[20] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[21] + a[21] * b[4]), -0.18467439711093903f * a[14] * b[1])))))));
        o[6] = ((fmaf(-0.057343922555446625f, a[23] * b[23], fmaf(0.1392638087272644f, a[19] * b[19], fmaf(0.15607835352420807f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.24179553985595703f, (a[6] * b[20] + a[20] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[18] + a[18] * b[4]), fmaf(0.24776668846607208f, a[12] * b[2], 0.282094806432724f * (a[0] * b[6] + a[6] * b[0]))))))) + fmaf(-0.2293756902217865f, a[24] * b[24], fmaf(0.16383977234363556f, a[20] * b[20], fmaf(-0.2293756902217865f, a[16] * b[16], fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.0901118740439415f, a[5] * b[5], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1]))))))) + (fmaf(0.1392638087272644f, a[21] * b[21], fmaf(-0.057343922555446625f, a[17] * b[17], fmaf(0.22072811424732208f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.22072811424732208f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.20230065286159515f, a[13] * b[3], 0.20230065286159515f * a[11] * b[1]))))) + fmaf(0.06553591042757034f, a[22] * b[22], fmaf(0.06553591042757034f, a[18] * b[18], fmaf(-0.180223748087883f, a[8] * b[8], fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2])))))));
        o[7] = ((fmaf(0.04486937075853348f, (a[20] * b[21] + a[21] * b[20]), fmaf(0.16858388483524323f, (a[8] * b[23] + a[23] * b[8]), fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.06371872127056122f, (a[4] * b[19] + a[19] * b[4]), fmaf(-0.14304816722869873f, a[12] * b[3], 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])))))) + fmaf(0.09029786288738251f, (a[21] * b[22] + a[22] * b[21]), fmaf(0.14046335220336914f, (a[16] * b[17] + a[17] * b[16]), fmaf(-0.1611970216035843f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.180223748087883f, (a[5] * b[18] + a[18] * b[5]), fmaf(0.18467439711093903f, a[14] * b[3], 0.18467439711093903f * a[10] * b[1])))))) + (fmaf(0.13272538781166077f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.13272538781166077f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.180223748087883f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2])))))) + fmaf(0.14046335220336914f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.09029786288738251f, (a[18] * b[19] + a[19] * b[18]), fmaf(-0.06371872127056122f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.22072811424732208f, (a[6] * b[21] + a[21] * b[6]), fmaf(0.16858388483524323f, (a[4] * b[17] + a[17] * b[4]), 0.23359668254852295f * a[13] * b[2])))))));
        o[8] = ((fmaf(-0.11262122541666031f, (a[21] * b[23] + a[23] * b[21]), fmaf(-0.11262122541666031f, (a[17] * b[19] + a[19] * b[17]), fmaf(0.16858388483524323f, (a[7] * b[23] + a[23] * b[7]), fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.23841361701488495f, (a[4] * b[16] + a[16] * b[4]), fmaf(0.18467439711093903f, a[14] * b[2], 0.282094806432724f * (a[0] * b[8] + a[8] * b[0]))))))) + fmaf(-0.07508081942796707f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.14188940823078156f, a[19] * b[19], fmaf(0.04029925540089607f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.15607835352420807f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1]))))))) + (fmaf(-0.19036461412906647f, (a[20] * b[22] + a[22] * b[20]), fmaf(0.23841361701488495f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.15607835352420807f, a[7] * b[7], fmaf(0.16858388483524323f, (a[5] * b[17] + a[17] * b[5]), fmaf(-0.05839917063713074f, a[13] * b[3], 0.22617901861667633f * a[9] * b[1]))))) + fmaf(0.14188940823078156f, a[21] * b[21], fmaf(-0.07508081942796707f, (a[16] * b[18] + a[18] * b[16]), fmaf(-0.06371872127056122f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.22617901861667633f, a[15] * b[3], 0.05839917063713074f * a[11] * b[1])))))));
        o[9] = ((fmaf(-0.09932258725166321f, a[14] * b[19], fmaf(0.11752006411552429f, a[11] * b[24], fmaf(-0.09403159469366074f, a[11] * b[8], fmaf(-0.09403159469366074f, a[13] * b[4], fmaf(0.1628675013780594f, (a[2] * b[17] + a[17] * b[2]), 0.282094806432724f * a[9] * b[0]))))) + fmaf(-0.20355072617530823f, a[12] * b[17], fmaf(0.07693494111299515f, a[9] * b[20], fmaf(0.1486770063638687f, a[14] * b[5], fmaf(0.22617901861667633f, (a[3] * b[4] + a[4] * b[3]), 0.22617901861667633f * (a[1] * b[8] + a[8] * b[1])))))) + (fmaf(-0.11752006411552429f, a[13] * b[16], fmaf(-0.09932258725166321f, a[10] * b[21], fmaf(-0.2102610468864441f, a[9] * b[6], fmaf(0.23032943904399872f, (a[3] * b[16] + a[16] * b[3]), -0.04352817311882973f * (a[1] * b[22] + a[22] * b[1]))))) + fmaf(0.1332552284002304f, a[13] * b[18], fmaf(0.1332552284002304f, a[11] * b[22], fmaf(0.1486770063638687f, a[10] * b[7], fmaf(-0.04352817311882973f, (a[3] * b[18] + a[18] * b[3]), -0.23032943904399872f * (a[1] * b[24] + a[24] * b[1])))))));
        o[10] = ((fmaf(0.06785023957490921f, a[13] * b[17], fmaf(-0.15171775221824646f, a[10] * b[24], fmaf(0.1486770063638687f, a[9] * b[7], fmaf(-0.07539300620555878f, (a[3] * b[19] + a[19] * b[3]), fmaf(0.18467439711093903f, (a[2] * b[4] + a[4] * b[2]), 0.282094806432724f * a[10] * b[0]))))) + fmaf(0.10257992148399353f, a[13] * b[19], fmaf(0.10257992148399353f, a[11] * b[21], fmaf(0.11516471952199936f, a[11] * b[7], fmaf(-0.18806318938732147f, a[12] * b[4], fmaf(0.21324361860752106f, (a[2] * b[18] + a[18] * b[2]), 0.18467439711093903f * (a[1] * b[7] + a[7] * b[1]))))))) + (fmaf(0.15171775221824646f, a[14] * b[16], fmaf(-0.06785023957490921f, a[11] * b[23], fmaf(-0.09932258725166321f, a[9] * b[21], fmaf(0.11516471952199936f, a[13] * b[5], fmaf(0.18467439711093903f, (a[3] * b[5] + a[5] * b[3]), -0.07539300620555878f * (a[1] * b[21] + a[21] * b[1])))))) + fmaf(0.09932258725166321f, a[15] * b[19], fmaf(-0.04441840946674347f, a[12] * b[18], fmaf(-0.17951487004756927f, a[10] * b[20], fmaf(-0.1486770063638687f, a[15] * b[5], fmaf(0.1994711458683014f, (a[3] * b[17] + a[17] * b[3]), -0.1994711458683014f * (a[1] * b[23] + a[23] * b[1]))))))));
        o[11] = ((fmaf(-0.1332552284002304f, a[15] * b[18], fmaf(0.11468784511089325f, a[13] * b[18], fmaf(-0.06785023957490921f, a[10] * b[23], fmaf(-0.14567312598228455f, a[11] * b[8], fmaf(-0.11516471952199936f, a[14] * b[5], fmaf(0.16858388483524323f, (a[3] * b[18] + a[18] * b[3]), fmaf(-0.16858388483524323f, (a[1] * b[22] + a[22] * b[1]), 0.282094806432724f * a[11] * b[0]))))))) + fmaf(0.06785023957490921f, a[14] * b[17], fmaf(0.025644980370998383f, a[11] * b[20], fmaf(0.1332552284002304f, a[9] * b[22], fmaf(0.12615662813186646f, a[11] * b[6], fmaf(0.14567312598228455f, a[13] * b[4], fmaf(0.23359668254852295f, (a[2] * b[5] + a[5] * b[2]), 0.20230065286159515f * (a[1] * b[6] + a[6] * b[1])))))))) + (fmaf(-0.10257992148399353f, a[14] * b[19], fmaf(-0.11468784511089325f, a[11] * b[22], fmaf(0.11752006411552429f, a[9] * b[24], fmaf(0.11516471952199936f, a[10] * b[7], fmaf(0.09403159469366074f, a[15] * b[4], fmaf(0.23841361701488495f, (a[2] * b[19] + a[19] * b[2]), 0.05839917063713074f * (a[1] * b[8] + a[8] * b[1]))))))) + fmaf(-0.11752006411552429f, a[15] * b[16], fmaf(0.09932258725166321f, a[12] * b[19], fmaf(0.10257992148399353f, a[10] * b[21], fmaf(-0.09403159469366074f, a[9] * b[8], fmaf(0.059470802545547485f, a[12] * b[5], fmaf(-0.05839917063713074f, (a[3] * b[4] + a[4] * b[3]), -0.15078601241111755f * (a[1] * b[20] + a[20] * b[1])))))))));
        o[12] = ((fmaf(0.09932258725166321f, a[13] * b[21], fmaf(-0.20355072617530823f, a[9] * b[17], fmaf(0.059470802545547485f, a[11] * b[5], fmaf(0.2462325245141983f, (a[2] * b[20] + a[20] * b[2]), 0.282094806432724f * a[12] * b[0])))) + fmaf(-0.04441840946674347f, a[14] * b[22], fmaf(-0.04441840946674347f, a[10] * b[18], fmaf(0.16820883750915527f, a[12] * b[6], fmaf(-0.14304816722869873f, (a[3] * b[7] + a[7] * b[3]), -0.14304816722869873f * (a[1] * b[5] + a[5] * b[1])))))) + (fmaf(-0.20355072617530823f, a[15] * b[23], fmaf(0.09932258725166321f, a[11] * b[19], fmaf(0.059470802545547485f, a[13] * b[7], fmaf(0.1946638971567154f, (a[3] * b[21] + a[21] * b[3]), 0.1946638971567154f * (a[1] * b[19] + a[19] * b[1]))))) + fmaf(0.1538698822259903f, a[12] * b[20], fmaf(-0.18806318938732147f, a[14] * b[8], fmaf(-0.18806318938732147f, a[10] * b[4], 0.24776668846607208f * (a[2] * b[6] + a[6] * b[2]))))));
        o[13] = ((fmaf(-0.11752006411552429f, a[15] * b[24], fmaf(0.11468784511089325f, a[13] * b[22], fmaf(0.10257992148399353f, a[10] * b[19], fmaf(-0.09403159469366074f, a[15] * b[8], fmaf(0.12615662813186646f, a[13] * b[6], fmaf(0.16858388483524323f, (a[3] * b[22] + a[22] * b[3]), fmaf(0.23841361701488495f, (a[2] * b[21] + a[21] * b[2]), 0.282094806432724f * a[13] * b[0]))))))) + fmaf(0.10257992148399353f, a[14] * b[21], fmaf(0.11468784511089325f, a[11] * b[18], fmaf(-0.11752006411552429f, a[9] * b[16], fmaf(0.059470802545547485f, a[12] * b[7], fmaf(-0.09403159469366074f, a[9] * b[4], fmaf(0.20230065286159515f, (a[3] * b[6] + a[6] * b[3]), -0.05839917063713074f * (a[1] * b[4] + a[4] * b[1])))))))) + (fmaf(0.06785023957490921f, a[14] * b[23], fmaf(0.09932258725166321f, a[12] * b[21], fmaf(0.1332552284002304f, a[9] * b[18], fmaf(0.11516471952199936f, a[14] * b[7], fmaf(0.14567312598228455f, a[11] * b[4], fmaf(-0.05839917063713074f, (a[3] * b[8] + a[8] * b[3]), 0.16858388483524323f * (a[1] * b[18] + a[18] * b[1]))))))) + fmaf(0.1332552284002304f, a[15] * b[22], fmaf(0.025644980370998383f, a[13] * b[20], fmaf(0.06785023957490921f, a[10] * b[17], fmaf(0.14567312598228455f, a[13] * b[8], fmaf(0.11516471952199936f, a[10] * b[5], fmaf(-0.15078601241111755f, (a[3] * b[20] + a[20] * b[3]), 0.23359668254852295f * (a[2] * b[7] + a[7] * b[2])))))))));
        o[14] = ((fmaf(0.06785023957490921f, a[13] * b[23], fmaf(0.06785023957490921f, a[11] * b[17], fmaf(0.1486770063638687f, a[15] * b[7], fmaf(0.1994711458683014f, (a[3] * b[23] + a[23] * b[3]), fmaf(0.18467439711093903f, (a[2] * b[8] + a[8] * b[2]), 0.282094806432724f * a[14] * b[0]))))) + fmaf(-0.17951487004756927f, a[14] * b[20], fmaf(-0.10257992148399353f, a[11] * b[19], fmaf(-0.18806318938732147f, a[12] * b[8], fmaf(0.1486770063638687f, a[9] * b[5], fmaf(0.21324361860752106f, (a[2] * b[22] + a[22] * b[2]), -0.18467439711093903f * (a[1] * b[5] + a[5] * b[1]))))))) + (fmaf(0.15171775221824646f, a[14] * b[24], fmaf(-0.04441840946674347f, a[12] * b[22], fmaf(-0.09932258725166321f, a[9] * b[19], fmaf(-0.11516471952199936f, a[11] * b[5], fmaf(0.18467439711093903f, (a[3] * b[7] + a[7] * b[3]), 0.1994711458683014f * (a[1] * b[17] + a[17] * b[1])))))) + fmaf(-0.09932258725166321f, a[15] * b[21], fmaf(0.10257992148399353f, a[13] * b[21], fmaf(0.15171775221824646f, a[10] * b[16], fmaf(0.11516471952199936f, a[13] * b[7], fmaf(-0.07539300620555878f, (a[3] * b[21] + a[21] * b[3]), 0.07539300620555878f * (a[1] * b[19] + a[19] * b[1]))))))));
        o[15] = ((fmaf(0.07693494111299515f, a[15] * b[20], fmaf(-0.20355072617530823f, a[12] * b[23], fmaf(-0.09403159469366074f, a[13] * b[8], fmaf(0.09403159469366074f, a[11] * b[4], fmaf(0.1628675013780594f, (a[2] * b[23] + a[23] * b[2]), 0.282094806432724f * a[15] * b[0]))))) + fmaf(0.1332552284002304f, a[13] * b[22], fmaf(0.09932258725166321f, a[10] * b[19], fmaf(-0.1486770063638687f, a[10] * b[5], fmaf(0.22617901861667633f, (a[3] * b[8] + a[8] * b[3]), -0.22617901861667633f * (a[1] * b[4] + a[4] * b[1])))))) + (fmaf(-0.11752006411552429f, a[13] * b[24], fmaf(-0.11752006411552429f, a[11] * b[16], fmaf(-0.2102610468864441f, a[15] * b[6], fmaf(-0.04352817311882973f, (a[3] * b[22] + a[22] * b[3]), 0.23032943904399872f * (a[1] * b[16] + a[16] * b[1]))))) + fmaf(-0.09932258725166321f, a[14] * b[21], fmaf(-0.1332552284002304f, a[11] * b[18], fmaf(0.1486770063638687f, a[14] * b[7], fmaf(0.23032943904399872f, (a[3] * b[24] + a[24] * b[3]), 0.04352817311882973f * (a[1] * b[18] + a[18] * b[1])))))));
        o[16] = ((fmaf(-0.11909890919923782f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.07508081942796707f, (a[8] * b[18] + a[18] * b[8]), fmaf(-0.07508081942796707f, (a[4] * b[22] + a[22] * b[4]), 0.282094806432724f * (a[0] * b[16] + a[16] * b[0])))) + fmaf(0.10652530938386917f, (a[16] * b[20] + a[20] * b[16]), fmaf(0.14046335220336914f, (a[5] * b[23] + a[23] * b[5]), 0.23032943904399872f * a[15] * b[1]))) + (fmaf(-0.11909890919923782f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.2293756902217865f, (a[6] * b[16] + a[16] * b[6]), 0.23032943904399872f * a[9] * b[3])) + fmaf(0.13504546880722046f, (a[18] * b[22] + a[22] * b[18]), fmaf(0.14046335220336914f, (a[7] * b[17] + a[17] * b[7]), 0.23841361701488495f * (a[4] * b[8] + a[8] * b[4])))));
        o[17] = ((fmaf(0.045015156269073486f, (a[19] * b[22] + a[22] * b[19]), fmaf(-0.11262122541666031f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[24] + a[24] * b[5]), fmaf(0.16858388483524323f, (a[4] * b[7] + a[7] * b[4]), 0.282094806432724f * (a[0] * b[17] + a[17] * b[0]))))) + fmaf(0.11909890919923782f, (a[19] * b[24] + a[24] * b[19]), fmaf(-0.11909890919923782f, (a[16] * b[21] + a[21] * b[16]), fmaf(-0.057343922555446625f, (a[6] * b[17] + a[17] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[21] + a[21] * b[4]), 0.1994711458683014f * a[14] * b[1]))))) + (fmaf(-0.15978795289993286f, (a[17] * b[20] + a[20] * b[17]), fmaf(0.14046335220336914f, (a[7] * b[16] + a[16] * b[7]), fmaf(0.16858388483524323f, (a[5] * b[8] + a[8] * b[5]), 0.1628675013780594f * a[9] * b[2]))) + fmaf(0.045015156269073486f, (a[18] * b[21] + a[21] * b[18]), fmaf(0.13272538781166077f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.13272538781166077f, (a[5] * b[22] + a[22] * b[5]), 0.1994711458683014f * a[10] * b[3])))));
        o[18] = ((fmaf(0.10208478569984436f, (a[19] * b[21] + a[21] * b[19]), fmaf(0.13504546880722046f, (a[16] * b[22] + a[22] * b[16]), fmaf(0.06553591042757034f, (a[6] * b[18] + a[18] * b[6]), fmaf(0.07508081942796707f, (a[4] * b[24] + a[24] * b[4]), fmaf(-0.04352817311882973f, a[9] * b[3], 0.282094806432724f * (a[0] * b[18] + a[18] * b[0])))))) + fmaf(-0.045015156269073486f, (a[19] * b[23] + a[23] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[21] + a[21] * b[17]), fmaf(0.13272538781166077f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.180223748087883f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.16858388483524323f, a[11] * b[3], 0.16858388483524323f * a[13] * b[1])))))) + (fmaf(-0.08369845151901245f, (a[18] * b[20] + a[20] * b[18]), fmaf(0.09029786288738251f, (a[7] * b[19] + a[19] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[21] + a[21] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[6] + a[6] * b[4]), 0.04352817311882973f * a[15] * b[1])))) + fmaf(-0.13504546880722046f, (a[18] * b[24] + a[24] * b[18]), fmaf(-0.07508081942796707f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.13272538781166077f, (a[5] * b[23] + a[23] * b[5]), fmaf(-0.19036461412906647f, (a[4] * b[20] + a[20] * b[4]), 0.21324361860752106f * a[10] * b[2]))))));
        o[19] = ((fmaf(-0.045015156269073486f, (a[18] * b[23] + a[23] * b[18]), fmaf(-0.11909890919923782f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.1392638087272644f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.22072811424732208f, (a[5] * b[6] + a[6] * b[5]), fmaf(-0.07539300620555878f, a[10] * b[3], 0.282094806432724f * (a[0] * b[19] + a[19] * b[0])))))) + fmaf(0.06848055124282837f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[22] + a[22] * b[17]), fmaf(0.09029786288738251f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[8] + a[8] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[7] + a[7] * b[4]), 0.1946638971567154f * a[12] * b[1])))))) + (fmaf(-0.10208478569984436f, (a[19] * b[22] + a[22] * b[19]), fmaf(0.11909890919923782f, (a[17] * b[24] + a[24] * b[17]), fmaf(-0.11262122541666031f, (a[8] * b[17] + a[17] * b[8]), fmaf(0.04486937075853348f, (a[5] * b[20] + a[20] * b[5]), fmaf(0.14188940823078156f, (a[4] * b[21] + a[21] * b[4]), 0.07539300620555878f * a[14] * b[1]))))) + fmaf(0.10208478569984436f, (a[18] * b[21] + a[21] * b[18]), fmaf(-0.14188940823078156f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.09029786288738251f, (a[5] * b[22] + a[22] * b[5]), fmaf(0.11262122541666031f, (a[4] * b[23] + a[23] * b[4]), 0.23841361701488495f * a[11] * b[2]))))));
        o[20] = ((fmaf(-0.08369845151901245f, a[22] * b[22], fmaf(-0.08369845151901245f, a[18] * b[18], fmaf(0.04029925540089607f, a[8] * b[8], fmaf(0.24179553985595703f, a[6] * b[6], fmaf(0.04029925540089607f, a[4] * b[4], 0.282094806432724f * (a[0] * b[20] + a[20] * b[0])))))) + fmaf(-0.15978795289993286f, a[23] * b[23], fmaf(0.06848055124282837f, a[19] * b[19], fmaf(-0.19036461412906647f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.16383977234363556f, (a[6] * b[20] + a[20] * b[6]), fmaf(-0.19036461412906647f, (a[4] * b[18] + a[18] * b[4]), -0.15078601241111755f * a[11] * b[1])))))) + (fmaf(0.10652530938386917f, a[24] * b[24], fmaf(0.13696110248565674f, a[20] * b[20], fmaf(0.10652530938386917f, a[16] * b[16], fmaf(-0.1611970216035843f, a[7] * b[7], fmaf(-0.1611970216035843f, a[5] * b[5], 0.2462325245141983f * a[12] * b[2]))))) + fmaf(0.06848055124282837f, a[21] * b[21], fmaf(-0.15978795289993286f, a[17] * b[17], fmaf(0.04486937075853348f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.04486937075853348f, (a[5] * b[19] + a[19] * b[5]), -0.15078601241111755f * a[13] * b[3]))))));
        o[21] = ((fmaf(0.10208478569984436f, (a[21] * b[22] + a[22] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[17] + a[17] * b[16]), fmaf(0.04486937075853348f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[18] + a[18] * b[5]), fmaf(-0.07539300620555878f, a[14] * b[3], 0.282094806432724f * (a[0] * b[21] + a[21] * b[0])))))) + fmaf(0.045015156269073486f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.045015156269073486f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.09029786288738251f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.22072811424732208f, (a[6] * b[7] + a[7] * b[6]), fmaf(-0.06371872127056122f, (a[4] * b[5] + a[5] * b[4]), -0.07539300620555878f * a[10] * b[1])))))) + (fmaf(-0.11909890919923782f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.10208478569984436f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.14188940823078156f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.1392638087272644f, (a[6] * b[21] + a[21] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[17] + a[17] * b[4]), 0.23841361701488495f * a[13] * b[2]))))) + fmaf(0.06848055124282837f, (a[20] * b[21] + a[21] * b[20]), fmaf(-0.11262122541666031f, (a[8] * b[23] + a[23] * b[8]), fmaf(-0.06371872127056122f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.14188940823078156f, (a[4] * b[19] + a[19] * b[4]), 0.1946638971567154f * a[12] * b[3]))))));
        o[22] = ((fmaf(-0.08369845151901245f, (a[20] * b[22] + a[22] * b[20]), fmaf(-0.07508081942796707f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.180223748087883f, a[7] * b[7], fmaf(0.13272538781166077f, (a[5] * b[17] + a[17] * b[5]), fmaf(0.16858388483524323f, a[13] * b[3], 0.282094806432724f * (a[0] * b[22] + a[22] * b[0])))))) + fmaf(0.10208478569984436f, a[21] * b[21], fmaf(0.13504546880722046f, (a[16] * b[18] + a[18] * b[16]), fmaf(0.09029786288738251f, (a[7] * b[21] + a[21] * b[7]), fmaf(-0.09029786288738251f, (a[5] * b[19] + a[19] * b[5]), fmaf(-0.04352817311882973f, a[15] * b[3], -0.04352817311882973f * a[9] * b[1])))))) + (fmaf(0.045015156269073486f, (a[21] * b[23] + a[23] * b[21]), fmaf(0.045015156269073486f, (a[17] * b[19] + a[19] * b[17]), fmaf(0.13272538781166077f, (a[7] * b[23] + a[23] * b[7]), fmaf(0.15607835352420807f, (a[6] * b[8] + a[8] * b[6]), fmaf(-0.07508081942796707f, (a[4] * b[16] + a[16] * b[4]), -0.16858388483524323f * a[11] * b[1]))))) + fmaf(0.13504546880722046f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.10208478569984436f, a[19] * b[19], fmaf(-0.19036461412906647f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.06553591042757034f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.180223748087883f, a[5] * b[5], 0.21324361860752106f * a[14] * b[2])))))));
        o[23] = ((fmaf(0.045015156269073486f, (a[21] * b[22] + a[22] * b[21]), fmaf(-0.11262122541666031f, (a[8] * b[21] + a[21] * b[8]), fmaf(-0.057343922555446625f, (a[6] * b[23] + a[23] * b[6]), fmaf(-0.16858388483524323f, (a[4] * b[5] + a[5] * b[4]), 0.282094806432724f * (a[0] * b[23] + a[23] * b[0]))))) + fmaf(-0.11909890919923782f, (a[21] * b[24] + a[24] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[19] + a[19] * b[16]), fmaf(0.16858388483524323f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.11262122541666031f, (a[4] * b[19] + a[19] * b[4]), -0.1994711458683014f * a[10] * b[1]))))) + (fmaf(-0.045015156269073486f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.13272538781166077f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.14046335220336914f, (a[5] * b[16] + a[16] * b[5]), 0.1628675013780594f * a[15] * b[2]))) + fmaf(-0.15978795289993286f, (a[20] * b[23] + a[23] * b[20]), fmaf(0.14046335220336914f, (a[7] * b[24] + a[24] * b[7]), fmaf(-0.13272538781166077f, (a[5] * b[18] + a[18] * b[5]), 0.1994711458683014f * a[14] * b[3])))));
        o[24] = ((fmaf(0.10652530938386917f, (a[20] * b[24] + a[24] * b[20]), fmaf(0.23841361701488495f, a[8] * b[8], fmaf(0.07508081942796707f, (a[4] * b[18] + a[18] * b[4]), 0.282094806432724f * (a[0] * b[24] + a[24] * b[0])))) + fmaf(-0.11909890919923782f, (a[21] * b[23] + a[23] * b[21]), fmaf(-0.07508081942796707f, (a[8] * b[22] + a[22] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[17] + a[17] * b[5]), -0.23032943904399872f * a[9] * b[1])))) + (fmaf(0.13504546880722046f, a[22] * b[22], fmaf(0.11909890919923782f, (a[17] * b[19] + a[19] * b[17]), fmaf(-0.2293756902217865f, (a[6] * b[24] + a[24] * b[6]), 0.23032943904399872f * a[15] * b[3]))) + fmaf(-0.13504546880722046f, a[18] * b[18], fmaf(0.14046335220336914f, (a[7] * b[23] + a[23] * b[7]), -0.23841361701488495f * a[4] * b[4]))));
    }
    __device__ __forceinline__ static void mul_onto_lobe(const float* __restrict__ a, const float* __restrict__ b,
                                               float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[24] * b[24], fmaf(0.282094806432724f, a[20] * b[20], fmaf(0.282094806432724f, a[16] * b[16], fmaf(0.282094806432724f, a[12] * b[12], fmaf(0.282094806432724f, a[8] * b[8], fmaf(0.282094806432724f, a[4] * b[4], 0.282094806432724f * a[0] * b[0])))))) + fmaf(0.282094806432724f, a[21] * b[21], fmaf(0.282094806432724f, a[17] * b[17], fmaf(0.282094806432724f, a[13] * b[13], fmaf(0.282094806432724f, a[9] * b[9], fmaf(0.282094806432724f, a[5] * b[5], 0.282094806432724f * a[1] * b[1])))))) + (fmaf(0.282094806432724f, a[22] * b[22], fmaf(0.282094806432724f, a[18] * b[18], fmaf(0.282094806432724f, a[14] * b[14], fmaf(0.282094806432724f, a[10] * b[10], fmaf(0.282094806432724f, a[6] * b[6], 0.282094806432724f * a[2] * b[2]))))) + fmaf(0.282094806432724f, a[23] * b[23], fmaf(0.282094806432724f, a[19] * b[19], fmaf(0.282094806432724f, a[15] * b[15], fmaf(0.282094806432724f, a[11] * b[11], fmaf(0.282094806432724f, a[7] * b[7], 0.282094806432724f * a[3] * b[3])))))));
        o[1] = ((fmaf(0.04352817311882973f, (a[15] * b[18] + a[18] * b[15]), fmaf(0.16858388483524323f, (a[13] * b[18] + a[18] * b[13]), fmaf(-0.1994711458683014f, (a[10] * b[23] + a[23] * b[10]), fmaf(0.05839917063713074f, (a[8] * b[11] + a[11] * b[8]), fmaf(-0.18467439711093903f, (a[5] * b[14] + a[14] * b[5]), fmaf(0.21850968897342682f, (a[3] * b[4] + a[4] * b[3]), 0.282094806432724f * (a[0] * b[1] + a[1] * b[0]))))))) + fmaf(0.1994711458683014f, (a[14] * b[17] + a[17] * b[14]), fmaf(-0.15078601241111755f, (a[11] * b[20] + a[20] * b[11]), fmaf(-0.04352817311882973f, (a[9] * b[22] + a[22] * b[9]), fmaf(0.20230065286159515f, (a[6] * b[11] + a[11] * b[6]), fmaf(-0.05839917063713074f, (a[4] * b[13] + a[13] * b[4]), -0.12615662813186646f * (a[1] * b[6] + a[6] * b[1]))))))) + (fmaf(0.07539300620555878f, (a[14] * b[19] + a[19] * b[14]), fmaf(-0.16858388483524323f, (a[11] * b[22] + a[22] * b[11]), fmaf(-0.23032943904399872f, (a[9] * b[24] + a[24] * b[9]), fmaf(0.18467439711093903f, (a[7] * b[10] + a[10] * b[7]), fmaf(-0.22617901861667633f, (a[4] * b[15] + a[15] * b[4]), -0.21850968897342682f * (a[1] * b[8] + a[8] * b[1])))))) + fmaf(0.23032943904399872f, (a[15] * b[16] + a[16] * b[15]), fmaf(0.1946638971567154f, (a[12] * b[19] + a[19] * b[12]), fmaf(-0.07539300620555878f, (a[10] * b[21] + a[21] * b[10]), fmaf(0.22617901861667633f, (a[8] * b[9] + a[9] * b[8]), fmaf(-0.14304816722869873f, (a[5] * b[12] + a[12] * b[5]), 0.21850968897342682f * (a[2] * b[5] + a[5] * b[2]))))))));
        o[2] = ((fmaf(0.2462325245141983f, (a[12] * b[20] + a[20] * b[12]), fmaf(0.18467439711093903f, (a[8] * b[14] + a[14] * b[8]), fmaf(0.18467439711093903f, (a[4] * b[10] + a[10] * b[4]), 0.282094806432724f * (a[0] * b[2] + a[2] * b[0])))) + fmaf(0.23841361701488495f, (a[13] * b[21] + a[21] * b[13]), fmaf(0.1628675013780594f, (a[9] * b[17] + a[17] * b[9]), fmaf(0.23359668254852295f, (a[5] * b[11] + a[11] * b[5]), 0.21850968897342682f * (a[1] * b[5] + a[5] * b[1]))))) + (fmaf(0.21324361860752106f, (a[14] * b[22] + a[22] * b[14]), fmaf(0.21324361860752106f, (a[10] * b[18] + a[18] * b[10]), fmaf(0.24776668846607208f, (a[6] * b[12] + a[12] * b[6]), 0.2523132562637329f * (a[2] * b[6] + a[6] * b[2])))) + fmaf(0.1628675013780594f, (a[15] * b[23] + a[23] * b[15]), fmaf(0.23841361701488495f, (a[11] * b[19] + a[19] * b[11]), fmaf(0.23359668254852295f, (a[7] * b[13] + a[13] * b[7]), 0.21850968897342682f * (a[3] * b[7] + a[7] * b[3]))))));
        o[3] = ((fmaf(0.23032943904399872f, (a[15] * b[24] + a[24] * b[15]), fmaf(0.16858388483524323f, (a[13] * b[22] + a[22] * b[13]), fmaf(-0.07539300620555878f, (a[10] * b[19] + a[19] * b[10]), fmaf(0.22617901861667633f, (a[8] * b[15] + a[15] * b[8]), fmaf(0.20230065286159515f, (a[6] * b[13] + a[13] * b[6]), fmaf(0.21850968897342682f, (a[3] * b[8] + a[8] * b[3]), 0.282094806432724f * (a[0] * b[3] + a[3] * b[0]))))))) + fmaf(-0.07539300620555878f, (a[14] * b[21] + a[21] * b[14]), fmaf(0.16858388483524323f, (a[11] * b[18] + a[18] * b[11]), fmaf(0.23032943904399872f, (a[9] * b[16] + a[16] * b[9]), fmaf(-0.14304816722869873f, (a[7] * b[12] + a[12] * b[7]), fmaf(0.22617901861667633f, (a[4] * b[9] + a[9] * b[4]), 0.21850968897342682f * (a[1] * b[4] + a[4] * b[1]))))))) + (fmaf(0.1994711458683014f, (a[14] * b[23] + a[23] * b[14]), fmaf(0.1946638971567154f, (a[12] * b[21] + a[21] * b[12]), fmaf(-0.04352817311882973f, (a[9] * b[18] + a[18] * b[9]), fmaf(0.18467439711093903f, (a[7] * b[14] + a[14] * b[7]), fmaf(-0.05839917063713074f, (a[4] * b[11] + a[11] * b[4]), 0.21850968897342682f * (a[2] * b[7] + a[7] * b[2])))))) + fmaf(-0.04352817311882973f, (a[15] * b[22] + a[22] * b[15]), fmaf(-0.15078601241111755f, (a[13] * b[20] + a[20] * b[13]), fmaf(0.1994711458683014f, (a[10] * b[17] + a[17] * b[10]), fmaf(-0.05839917063713074f, (a[8] * b[13] + a[13] * b[8]), fmaf(0.18467439711093903f, (a[5] * b[10] + a[10] * b[5]), -0.12615662813186646f * (a[3] * b[6] + a[6] * b[3]))))))));
        o[4] = ((fmaf(0.07508081942796707f, (a[18] * b[24] + a[24] * b[18]), fmaf(0.09403159469366074f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.23841361701488495f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.16858388483524323f, (a[5] * b[23] + a[23] * b[5]), fmaf(0.04029925540089607f, (a[4] * b[20] + a[20] * b[4]), fmaf(0.18467439711093903f, (a[2] * b[10] + a[10] * b[2]), 0.282094806432724f * (a[0] * b[4] + a[4] * b[0]))))))) + fmaf(0.14188940823078156f, (a[19] * b[21] + a[21] * b[19]), fmaf(-0.07508081942796707f, (a[16] * b[22] + a[22] * b[16]), fmaf(-0.09403159469366074f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.15607835352420807f, (a[6] * b[18] + a[18] * b[6]), fmaf(-0.23841361701488495f, (a[4] * b[24] + a[24] * b[4]), fmaf(0.22617901861667633f, (a[3] * b[9] + a[9] * b[3]), 0.21850968897342682f * (a[1] * b[3] + a[3] * b[1])))))))) + (fmaf(0.11262122541666031f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.11262122541666031f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.18806318938732147f, (a[10] * b[12] + a[12] * b[10]), fmaf(0.16858388483524323f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.15607835352420807f, (a[5] * b[7] + a[7] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[11] + a[11] * b[3]), -0.05839917063713074f * (a[1] * b[13] + a[13] * b[1]))))))) + fmaf(-0.19036461412906647f, (a[18] * b[20] + a[20] * b[18]), fmaf(0.14567312598228455f, (a[11] * b[13] + a[13] * b[11]), fmaf(-0.06371872127056122f, (a[7] * b[19] + a[19] * b[7]), fmaf(-0.06371872127056122f, (a[5] * b[21] + a[21] * b[5]), fmaf(-0.180223748087883f, (a[4] * b[6] + a[6] * b[4]), -0.22617901861667633f * (a[1] * b[15] + a[15] * b[1]))))))));
        o[5] = ((fmaf(-0.09029786288738251f, (a[19] * b[22] + a[22] * b[19]), fmaf(-0.14046335220336914f, (a[17] * b[24] + a[24] * b[17]), fmaf(0.059470802545547485f, (a[11] * b[12] + a[12] * b[11]), fmaf(0.06371872127056122f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.180223748087883f, (a[5] * b[22] + a[22] * b[5]), fmaf(-0.16858388483524323f, (a[4] * b[23] + a[23] * b[4]), fmaf(0.23359668254852295f, (a[2] * b[11] + a[11] * b[2]), 0.282094806432724f * (a[0] * b[5] + a[5] * b[0])))))))) + fmaf(0.09029786288738251f, (a[18] * b[21] + a[21] * b[18]), fmaf(-0.11516471952199936f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.1486770063638687f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.22072811424732208f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.0901118740439415f, (a[5] * b[6] + a[6] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[10] + a[10] * b[3]), 0.21850968897342682f * (a[1] * b[2] + a[2] * b[1])))))))) + (fmaf(-0.13272538781166077f, (a[18] * b[23] + a[23] * b[18]), fmaf(0.14046335220336914f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.11516471952199936f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.180223748087883f, (a[7] * b[18] + a[18] * b[7]), fmaf(-0.15607835352420807f, (a[5] * b[8] + a[8] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[7] + a[7] * b[4]), -0.14304816722869873f * (a[1] * b[12] + a[12] * b[1]))))))) + fmaf(0.04486937075853348f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.13272538781166077f, (a[17] * b[22] + a[22] * b[17]), fmaf(-0.1486770063638687f, (a[10] * b[15] + a[15] * b[10]), fmaf(0.16858388483524323f, (a[8] * b[17] + a[17] * b[8]), fmaf(-0.1611970216035843f, (a[5] * b[20] + a[20] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[21] + a[21] * b[4]), -0.18467439711093903f * (a[1] * b[14] + a[14] * b[1])))))))));
        o[6] = ((fmaf(0.06553591042757034f, a[22] * b[22], fmaf(0.06553591042757034f, a[18] * b[18], fmaf(0.12615662813186646f, a[13] * b[13], fmaf(0.15607835352420807f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.24179553985595703f, (a[6] * b[20] + a[20] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[18] + a[18] * b[4]), fmaf(0.24776668846607208f, (a[2] * b[12] + a[12] * b[2]), 0.282094806432724f * (a[0] * b[6] + a[6] * b[0])))))))) + fmaf(-0.057343922555446625f, a[23] * b[23], fmaf(0.1392638087272644f, a[19] * b[19], fmaf(-0.2102610468864441f, a[15] * b[15], fmaf(-0.2102610468864441f, a[9] * b[9], fmaf(0.0901118740439415f, a[7] * b[7], fmaf(0.0901118740439415f, a[5] * b[5], fmaf(-0.12615662813186646f, a[3] * b[3], -0.12615662813186646f * a[1] * b[1])))))))) + (fmaf(-0.2293756902217865f, a[24] * b[24], fmaf(0.16383977234363556f, a[20] * b[20], fmaf(-0.2293756902217865f, a[16] * b[16], fmaf(0.12615662813186646f, a[11] * b[11], fmaf(0.22072811424732208f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.22072811424732208f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.20230065286159515f, (a[3] * b[13] + a[13] * b[3]), 0.20230065286159515f * (a[1] * b[11] + a[11] * b[1])))))))) + fmaf(0.1392638087272644f, a[21] * b[21], fmaf(-0.057343922555446625f, a[17] * b[17], fmaf(0.16820883750915527f, a[12] * b[12], fmaf(-0.180223748087883f, a[8] * b[8], fmaf(0.180223748087883f, a[6] * b[6], fmaf(-0.180223748087883f, a[4] * b[4], 0.2523132562637329f * a[2] * b[2]))))))));
        o[7] = ((fmaf(0.14046335220336914f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.09029786288738251f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.11516471952199936f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.16858388483524323f, (a[8] * b[23] + a[23] * b[8]), fmaf(0.15607835352420807f, (a[7] * b[8] + a[8] * b[7]), fmaf(-0.06371872127056122f, (a[4] * b[19] + a[19] * b[4]), fmaf(-0.14304816722869873f, (a[3] * b[12] + a[12] * b[3]), 0.282094806432724f * (a[0] * b[7] + a[7] * b[0])))))))) + fmaf(0.04486937075853348f, (a[20] * b[21] + a[21] * b[20]), fmaf(0.1486770063638687f, (a[14] * b[15] + a[15] * b[14]), fmaf(0.1486770063638687f, (a[9] * b[10] + a[10] * b[9]), fmaf(-0.1611970216035843f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.180223748087883f, (a[5] * b[18] + a[18] * b[5]), fmaf(0.18467439711093903f, (a[3] * b[14] + a[14] * b[3]), 0.18467439711093903f * (a[1] * b[10] + a[10] * b[1])))))))) + (fmaf(0.09029786288738251f, (a[21] * b[22] + a[22] * b[21]), fmaf(0.14046335220336914f, (a[16] * b[17] + a[17] * b[16]), fmaf(0.11516471952199936f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.180223748087883f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.0901118740439415f, (a[6] * b[7] + a[7] * b[6]), fmaf(0.15607835352420807f, (a[4] * b[5] + a[5] * b[4]), 0.21850968897342682f * (a[2] * b[3] + a[3] * b[2]))))))) + fmaf(0.13272538781166077f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.13272538781166077f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.059470802545547485f, (a[12] * b[13] + a[13] * b[12]), fmaf(-0.06371872127056122f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.22072811424732208f, (a[6] * b[21] + a[21] * b[6]), fmaf(0.16858388483524323f, (a[4] * b[17] + a[17] * b[4]), 0.23359668254852295f * (a[2] * b[13] + a[13] * b[2])))))))));
        o[8] = ((fmaf(0.14188940823078156f, a[21] * b[21], fmaf(-0.07508081942796707f, (a[16] * b[18] + a[18] * b[16]), fmaf(-0.14567312598228455f, a[11] * b[11], fmaf(0.16858388483524323f, (a[7] * b[23] + a[23] * b[7]), fmaf(-0.180223748087883f, (a[6] * b[8] + a[8] * b[6]), fmaf(0.23841361701488495f, (a[4] * b[16] + a[16] * b[4]), fmaf(0.18467439711093903f, (a[2] * b[14] + a[14] * b[2]), 0.282094806432724f * (a[0] * b[8] + a[8] * b[0])))))))) + fmaf(-0.11262122541666031f, (a[21] * b[23] + a[23] * b[21]), fmaf(-0.11262122541666031f, (a[17] * b[19] + a[19] * b[17]), fmaf(-0.18806318938732147f, (a[12] * b[14] + a[14] * b[12]), fmaf(0.04029925540089607f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.15607835352420807f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.15607835352420807f, a[5] * b[5], fmaf(0.21850968897342682f, a[3] * b[3], -0.21850968897342682f * a[1] * b[1])))))))) + (fmaf(-0.07508081942796707f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.14188940823078156f, a[19] * b[19], fmaf(0.14567312598228455f, a[13] * b[13], fmaf(0.23841361701488495f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.15607835352420807f, a[7] * b[7], fmaf(0.16858388483524323f, (a[5] * b[17] + a[17] * b[5]), fmaf(-0.05839917063713074f, (a[3] * b[13] + a[13] * b[3]), 0.22617901861667633f * (a[1] * b[9] + a[9] * b[1])))))))) + fmaf(-0.19036461412906647f, (a[20] * b[22] + a[22] * b[20]), fmaf(-0.09403159469366074f, (a[13] * b[15] + a[15] * b[13]), fmaf(-0.09403159469366074f, (a[9] * b[11] + a[11] * b[9]), fmaf(-0.06371872127056122f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[19] + a[19] * b[5]), fmaf(0.22617901861667633f, (a[3] * b[15] + a[15] * b[3]), 0.05839917063713074f * (a[1] * b[11] + a[11] * b[1])))))))));
        o[9] = 0.0f;
        o[10] = 0.0f;
        o[11] = 0.0f;
        o[12] = 0.0f;
        o[13] = 0.0f;
        o[14] = 0.0f;
        o[15] = 0.0f;
        o[16] = ((fmaf(0.10652530938386917f, (a[16] * b[20] + a[20] * b[16]), fmaf(-0.07508081942796707f, (a[8] * b[18] + a[18] * b[8]), fmaf(-0.07508081942796707f, (a[4] * b[22] + a[22] * b[4]), 0.282094806432724f * (a[0] * b[16] + a[16] * b[0])))) + fmaf(-0.11909890919923782f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.11752006411552429f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.14046335220336914f, (a[5] * b[23] + a[23] * b[5]), 0.23032943904399872f * (a[1] * b[15] + a[15] * b[1]))))) + (fmaf(0.13504546880722046f, (a[18] * b[22] + a[22] * b[18]), fmaf(0.15171775221824646f, (a[10] * b[14] + a[14] * b[10]), fmaf(-0.2293756902217865f, (a[6] * b[16] + a[16] * b[6]), 0.23032943904399872f * (a[3] * b[9] + a[9] * b[3])))) + fmaf(-0.11909890919923782f, (a[19] * b[23] + a[23] * b[19]), fmaf(-0.11752006411552429f, (a[11] * b[15] + a[15] * b[11]), fmaf(0.14046335220336914f, (a[7] * b[17] + a[17] * b[7]), 0.23841361701488495f * (a[4] * b[8] + a[8] * b[4]))))));
        o[17] = ((fmaf(0.11909890919923782f, (a[19] * b[24] + a[24] * b[19]), fmaf(-0.11909890919923782f, (a[16] * b[21] + a[21] * b[16]), fmaf(-0.11262122541666031f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[24] + a[24] * b[5]), fmaf(0.16858388483524323f, (a[4] * b[7] + a[7] * b[4]), 0.282094806432724f * (a[0] * b[17] + a[17] * b[0])))))) + fmaf(-0.15978795289993286f, (a[17] * b[20] + a[20] * b[17]), fmaf(-0.20355072617530823f, (a[9] * b[12] + a[12] * b[9]), fmaf(-0.057343922555446625f, (a[6] * b[17] + a[17] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[21] + a[21] * b[4]), 0.1994711458683014f * (a[1] * b[14] + a[14] * b[1])))))) + (fmaf(0.045015156269073486f, (a[18] * b[21] + a[21] * b[18]), fmaf(0.06785023957490921f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.14046335220336914f, (a[7] * b[16] + a[16] * b[7]), fmaf(0.16858388483524323f, (a[5] * b[8] + a[8] * b[5]), 0.1628675013780594f * (a[2] * b[9] + a[9] * b[2]))))) + fmaf(0.045015156269073486f, (a[19] * b[22] + a[22] * b[19]), fmaf(0.06785023957490921f, (a[11] * b[14] + a[14] * b[11]), fmaf(0.13272538781166077f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.13272538781166077f, (a[5] * b[22] + a[22] * b[5]), 0.1994711458683014f * (a[3] * b[10] + a[10] * b[3])))))));
        o[18] = ((fmaf(0.10208478569984436f, (a[19] * b[21] + a[21] * b[19]), fmaf(0.13504546880722046f, (a[16] * b[22] + a[22] * b[16]), fmaf(0.1332552284002304f, (a[9] * b[13] + a[13] * b[9]), fmaf(0.06553591042757034f, (a[6] * b[18] + a[18] * b[6]), fmaf(0.07508081942796707f, (a[4] * b[24] + a[24] * b[4]), fmaf(-0.04352817311882973f, (a[3] * b[9] + a[9] * b[3]), 0.282094806432724f * (a[0] * b[18] + a[18] * b[0]))))))) + fmaf(-0.045015156269073486f, (a[19] * b[23] + a[23] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[21] + a[21] * b[17]), fmaf(-0.04441840946674347f, (a[10] * b[12] + a[12] * b[10]), fmaf(0.13272538781166077f, (a[7] * b[17] + a[17] * b[7]), fmaf(0.180223748087883f, (a[5] * b[7] + a[7] * b[5]), fmaf(0.16858388483524323f, (a[3] * b[11] + a[11] * b[3]), 0.16858388483524323f * (a[1] * b[13] + a[13] * b[1])))))))) + (fmaf(-0.08369845151901245f, (a[18] * b[20] + a[20] * b[18]), fmaf(0.11468784511089325f, (a[11] * b[13] + a[13] * b[11]), fmaf(0.09029786288738251f, (a[7] * b[19] + a[19] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[21] + a[21] * b[5]), fmaf(0.15607835352420807f, (a[4] * b[6] + a[6] * b[4]), 0.04352817311882973f * (a[1] * b[15] + a[15] * b[1])))))) + fmaf(-0.13504546880722046f, (a[18] * b[24] + a[24] * b[18]), fmaf(-0.1332552284002304f, (a[11] * b[15] + a[15] * b[11]), fmaf(-0.07508081942796707f, (a[8] * b[16] + a[16] * b[8]), fmaf(-0.13272538781166077f, (a[5] * b[23] + a[23] * b[5]), fmaf(-0.19036461412906647f, (a[4] * b[20] + a[20] * b[4]), 0.21324361860752106f * (a[2] * b[10] + a[10] * b[2]))))))));
        o[19] = ((fmaf(0.10208478569984436f, (a[18] * b[21] + a[21] * b[18]), fmaf(-0.10257992148399353f, (a[11] * b[14] + a[14] * b[11]), fmaf(-0.09932258725166321f, (a[9] * b[14] + a[14] * b[9]), fmaf(0.1392638087272644f, (a[6] * b[19] + a[19] * b[6]), fmaf(0.22072811424732208f, (a[5] * b[6] + a[6] * b[5]), fmaf(-0.07539300620555878f, (a[3] * b[10] + a[10] * b[3]), 0.282094806432724f * (a[0] * b[19] + a[19] * b[0]))))))) + fmaf(-0.045015156269073486f, (a[18] * b[23] + a[23] * b[18]), fmaf(-0.11909890919923782f, (a[16] * b[23] + a[23] * b[16]), fmaf(0.10257992148399353f, (a[10] * b[13] + a[13] * b[10]), fmaf(0.09029786288738251f, (a[7] * b[18] + a[18] * b[7]), fmaf(0.06371872127056122f, (a[5] * b[8] + a[8] * b[5]), fmaf(-0.06371872127056122f, (a[4] * b[7] + a[7] * b[4]), 0.1946638971567154f * (a[1] * b[12] + a[12] * b[1])))))))) + (fmaf(0.06848055124282837f, (a[19] * b[20] + a[20] * b[19]), fmaf(0.045015156269073486f, (a[17] * b[22] + a[22] * b[17]), fmaf(0.09932258725166321f, (a[10] * b[15] + a[15] * b[10]), fmaf(-0.11262122541666031f, (a[8] * b[17] + a[17] * b[8]), fmaf(0.04486937075853348f, (a[5] * b[20] + a[20] * b[5]), fmaf(0.14188940823078156f, (a[4] * b[21] + a[21] * b[4]), 0.07539300620555878f * (a[1] * b[14] + a[14] * b[1]))))))) + fmaf(-0.10208478569984436f, (a[19] * b[22] + a[22] * b[19]), fmaf(0.11909890919923782f, (a[17] * b[24] + a[24] * b[17]), fmaf(0.09932258725166321f, (a[11] * b[12] + a[12] * b[11]), fmaf(-0.14188940823078156f, (a[8] * b[19] + a[19] * b[8]), fmaf(-0.09029786288738251f, (a[5] * b[22] + a[22] * b[5]), fmaf(0.11262122541666031f, (a[4] * b[23] + a[23] * b[4]), 0.23841361701488495f * (a[2] * b[11] + a[11] * b[2])))))))));
        o[20] = ((fmaf(-0.15978795289993286f, a[23] * b[23], fmaf(0.06848055124282837f, a[19] * b[19], fmaf(0.07693494111299515f, a[15] * b[15], fmaf(0.025644980370998383f, a[11] * b[11], fmaf(0.04029925540089607f, a[8] * b[8], fmaf(0.24179553985595703f, a[6] * b[6], fmaf(0.04029925540089607f, a[4] * b[4], 0.282094806432724f * (a[0] * b[20] + a[20] * b[0])))))))) + fmaf(0.10652530938386917f, a[24] * b[24], fmaf(0.13696110248565674f, a[20] * b[20], fmaf(0.10652530938386917f, a[16] * b[16], fmaf(0.1538698822259903f, a[12] * b[12], fmaf(-0.19036461412906647f, (a[8] * b[22] + a[22] * b[8]), fmaf(0.16383977234363556f, (a[6] * b[20] + a[20] * b[6]), fmaf(-0.19036461412906647f, (a[4] * b[18] + a[18] * b[4]), -0.15078601241111755f * (a[1] * b[11] + a[11] * b[1]))))))))) + (fmaf(0.06848055124282837f, a[21] * b[21], fmaf(-0.15978795289993286f, a[17] * b[17], fmaf(0.025644980370998383f, a[13] * b[13], fmaf(0.07693494111299515f, a[9] * b[9], fmaf(-0.1611970216035843f, a[7] * b[7], fmaf(-0.1611970216035843f, a[5] * b[5], 0.2462325245141983f * (a[2] * b[12] + a[12] * b[2]))))))) + fmaf(-0.08369845151901245f, a[22] * b[22], fmaf(-0.08369845151901245f, a[18] * b[18], fmaf(-0.17951487004756927f, a[14] * b[14], fmaf(-0.17951487004756927f, a[10] * b[10], fmaf(0.04486937075853348f, (a[7] * b[21] + a[21] * b[7]), fmaf(0.04486937075853348f, (a[5] * b[19] + a[19] * b[5]), -0.15078601241111755f * (a[3] * b[13] + a[13] * b[3])))))))));
        o[21] = ((fmaf(0.06848055124282837f, (a[20] * b[21] + a[21] * b[20]), fmaf(-0.09932258725166321f, (a[14] * b[15] + a[15] * b[14]), fmaf(-0.09932258725166321f, (a[9] * b[10] + a[10] * b[9]), fmaf(0.04486937075853348f, (a[7] * b[20] + a[20] * b[7]), fmaf(0.09029786288738251f, (a[5] * b[18] + a[18] * b[5]), fmaf(-0.07539300620555878f, (a[3] * b[14] + a[14] * b[3]), 0.282094806432724f * (a[0] * b[21] + a[21] * b[0]))))))) + fmaf(0.10208478569984436f, (a[21] * b[22] + a[22] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[17] + a[17] * b[16]), fmaf(0.10257992148399353f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.09029786288738251f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.22072811424732208f, (a[6] * b[7] + a[7] * b[6]), fmaf(-0.06371872127056122f, (a[4] * b[5] + a[5] * b[4]), -0.07539300620555878f * (a[1] * b[10] + a[10] * b[1])))))))) + (fmaf(0.045015156269073486f, (a[22] * b[23] + a[23] * b[22]), fmaf(0.045015156269073486f, (a[17] * b[18] + a[18] * b[17]), fmaf(0.09932258725166321f, (a[12] * b[13] + a[13] * b[12]), fmaf(0.14188940823078156f, (a[8] * b[21] + a[21] * b[8]), fmaf(0.1392638087272644f, (a[6] * b[21] + a[21] * b[6]), fmaf(-0.11262122541666031f, (a[4] * b[17] + a[17] * b[4]), 0.23841361701488495f * (a[2] * b[13] + a[13] * b[2]))))))) + fmaf(-0.11909890919923782f, (a[23] * b[24] + a[24] * b[23]), fmaf(0.10208478569984436f, (a[18] * b[19] + a[19] * b[18]), fmaf(0.10257992148399353f, (a[13] * b[14] + a[14] * b[13]), fmaf(-0.11262122541666031f, (a[8] * b[23] + a[23] * b[8]), fmaf(-0.06371872127056122f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.14188940823078156f, (a[4] * b[19] + a[19] * b[4]), 0.1946638971567154f * (a[3] * b[12] + a[12] * b[3])))))))));
        o[22] = ((fmaf(0.13504546880722046f, (a[22] * b[24] + a[24] * b[22]), fmaf(-0.10208478569984436f, a[19] * b[19], fmaf(0.11468784511089325f, a[13] * b[13], fmaf(-0.07508081942796707f, (a[8] * b[24] + a[24] * b[8]), fmaf(0.180223748087883f, a[7] * b[7], fmaf(0.13272538781166077f, (a[5] * b[17] + a[17] * b[5]), fmaf(0.16858388483524323f, (a[3] * b[13] + a[13] * b[3]), 0.282094806432724f * (a[0] * b[22] + a[22] * b[0])))))))) + fmaf(-0.08369845151901245f, (a[20] * b[22] + a[22] * b[20]), fmaf(0.1332552284002304f, (a[13] * b[15] + a[15] * b[13]), fmaf(0.1332552284002304f, (a[9] * b[11] + a[11] * b[9]), fmaf(0.09029786288738251f, (a[7] * b[21] + a[21] * b[7]), fmaf(-0.09029786288738251f, (a[5] * b[19] + a[19] * b[5]), fmaf(-0.04352817311882973f, (a[3] * b[15] + a[15] * b[3]), -0.04352817311882973f * (a[1] * b[9] + a[9] * b[1])))))))) + (fmaf(0.10208478569984436f, a[21] * b[21], fmaf(0.13504546880722046f, (a[16] * b[18] + a[18] * b[16]), fmaf(-0.11468784511089325f, a[11] * b[11], fmaf(0.13272538781166077f, (a[7] * b[23] + a[23] * b[7]), fmaf(0.15607835352420807f, (a[6] * b[8] + a[8] * b[6]), fmaf(-0.07508081942796707f, (a[4] * b[16] + a[16] * b[4]), -0.16858388483524323f * (a[1] * b[11] + a[11] * b[1]))))))) + fmaf(0.045015156269073486f, (a[21] * b[23] + a[23] * b[21]), fmaf(0.045015156269073486f, (a[17] * b[19] + a[19] * b[17]), fmaf(-0.04441840946674347f, (a[12] * b[14] + a[14] * b[12]), fmaf(-0.19036461412906647f, (a[8] * b[20] + a[20] * b[8]), fmaf(0.06553591042757034f, (a[6] * b[22] + a[22] * b[6]), fmaf(-0.180223748087883f, a[5] * b[5], 0.21324361860752106f * (a[2] * b[14] + a[14] * b[2])))))))));
        o[23] = ((fmaf(-0.11909890919923782f, (a[21] * b[24] + a[24] * b[21]), fmaf(-0.11909890919923782f, (a[16] * b[19] + a[19] * b[16]), fmaf(-0.11262122541666031f, (a[8] * b[21] + a[21] * b[8]), fmaf(-0.057343922555446625f, (a[6] * b[23] + a[23] * b[6]), fmaf(-0.16858388483524323f, (a[4] * b[5] + a[5] * b[4]), 0.282094806432724f * (a[0] * b[23] + a[23] * b[0])))))) + fmaf(-0.045015156269073486f, (a[18] * b[19] + a[19] * b[18]), fmaf(-0.06785023957490921f, (a[10] * b[11] + a[11] * b[10]), fmaf(0.16858388483524323f, (a[7] * b[8] + a[8] * b[7]), fmaf(0.11262122541666031f, (a[4] * b[19] + a[19] * b[4]), -0.1994711458683014f * (a[1] * b[10] + a[10] * b[1])))))) + (fmaf(-0.15978795289993286f, (a[20] * b[23] + a[23] * b[20]), fmaf(-0.20355072617530823f, (a[12] * b[15] + a[15] * b[12]), fmaf(0.13272538781166077f, (a[7] * b[22] + a[22] * b[7]), fmaf(0.14046335220336914f, (a[5] * b[16] + a[16] * b[5]), 0.1628675013780594f * (a[2] * b[15] + a[15] * b[2]))))) + fmaf(0.045015156269073486f, (a[21] * b[22] + a[22] * b[21]), fmaf(0.06785023957490921f, (a[13] * b[14] + a[14] * b[13]), fmaf(0.14046335220336914f, (a[7] * b[24] + a[24] * b[7]), fmaf(-0.13272538781166077f, (a[5] * b[18] + a[18] * b[5]), 0.1994711458683014f * (a[3] * b[14] + a[14] * b[3])))))));
        o[24] = ((fmaf(0.10652530938386917f, (a[20] * b[24] + a[24] * b[20]), fmaf(-0.11752006411552429f, (a[13] * b[15] + a[15] * b[13]), fmaf(0.23841361701488495f, a[8] * b[8], fmaf(0.07508081942796707f, (a[4] * b[18] + a[18] * b[4]), 0.282094806432724f * (a[0] * b[24] + a[24] * b[0]))))) + fmaf(-0.11909890919923782f, (a[21] * b[23] + a[23] * b[21]), fmaf(0.15171775221824646f, a[14] * b[14], fmaf(-0.07508081942796707f, (a[8] * b[22] + a[22] * b[8]), fmaf(-0.14046335220336914f, (a[5] * b[17] + a[17] * b[5]), -0.23032943904399872f * (a[1] * b[9] + a[9] * b[1])))))) + (fmaf(0.13504546880722046f, a[22] * b[22], fmaf(0.11909890919923782f, (a[17] * b[19] + a[19] * b[17]), fmaf(0.11752006411552429f, (a[9] * b[11] + a[11] * b[9]), fmaf(-0.2293756902217865f, (a[6] * b[24] + a[24] * b[6]), 0.23032943904399872f * (a[3] * b[15] + a[15] * b[3]))))) + fmaf(-0.13504546880722046f, a[18] * b[18], fmaf(-0.15171775221824646f, a[10] * b[10], fmaf(0.14046335220336914f, (a[7] * b[23] + a[23] * b[7]), -0.23841361701488495f * a[4] * b[4])))));
    }
    __device__ __forceinline__ static void sqr(const float* __restrict__ a, float* __restrict__ o) {
        o[0] = ((fmaf(0.282094806432724f, a[24] * a[24], fmaf(0.282094806432724f, a[20] * a[20], fmaf(0.282094806432724f, a[16] * a[16], fmaf(0.282094806432724f, a[12] * a[12], fmaf(0.282094806432724f, a[8] * a[8], fmaf(0.282094806432724f, a[4] * a[4], 0.282094806432724f * a[0] * a[0])))))) + fmaf(0.282094806432724f, a[21] * a[21], fmaf(0.282094806432724f, a[17] * a[17], fmaf(0.282094806432724f, a[13] * a[13], fmaf(0.282094806432724f, a[9] * a[9], fmaf(0.282094806432724f, a[5] * a[5], 0.282094806432724f * a[1] * a[1])))))) + (fmaf(0.282094806432724f, a[22] * a[22], fmaf(0.282094806432724f, a[18] * a[18], fmaf(0.282094806432724f, a[14] * a[14], fmaf(0.282094806432724f, a[10] * a[10], fmaf(0.282094806432724f, a[6] * a[6], 0.282094806432724f * a[2] * a[2]))))) + fmaf(0.282094806432724f, a[23] * a[23], fmaf(0.282094806432724f, a[19] * a[19], fmaf(0.282094806432724f, a[15] * a[15], fmaf(0.282094806432724f, a[11] * a[11], fmaf(0.282094806432724f, a[7] * a[7], 0.282094806432724f * a[3] * a[3])))))));
        o[1] = ((fmaf(0.08705634623765945f, a[15] * a[18], fmaf(0.33716776967048645f, a[13] * a[18], fmaf(-0.3989422917366028f, a[10] * a[23], fmaf(0.11679834127426147f, a[8] * a[11], fmaf(-0.36934879422187805f, a[5] * a[14], fmaf(0.43701937794685364f, a[3] * a[4], 0.564189612865448f * a[0] * a[1])))))) + fmaf(0.3989422917366028f, a[14] * a[17], fmaf(-0.3015720248222351f, a[11] * a[20], fmaf(-0.08705634623765945f, a[9] * a[22], fmaf(0.4046013057231903f, a[6] * a[11], fmaf(-0.11679834127426147f, a[4] * a[13], -0.2523132562637329f * a[1] * a[6])))))) + (fmaf(0.15078601241111755f, a[14] * a[19], fmaf(-0.33716776967048645f, a[11] * a[22], fmaf(-0.46065887808799744f, a[9] * a[24], fmaf(0.36934879422187805f, a[7] * a[10], fmaf(-0.45235803723335266f, a[4] * a[15], -0.43701937794685364f * a[1] * a[8]))))) + fmaf(0.46065887808799744f, a[15] * a[16], fmaf(0.3893277943134308f, a[12] * a[19], fmaf(-0.15078601241111755f, a[10] * a[21], fmaf(0.45235803723335266f, a[8] * a[9], fmaf(-0.28609633445739746f, a[5] * a[12], 0.43701937794685364f * a[2] * a[5])))))));
        o[2] = ((fmaf(0.4924650490283966f, a[12] * a[20], fmaf(0.36934879422187805f, a[8] * a[14], fmaf(0.36934879422187805f, a[4] * a[10], 0.564189612865448f * a[0] * a[2]))) + fmaf(0.4768272340297699f, a[13] * a[21], fmaf(0.3257350027561188f, a[9] * a[17], fmaf(0.4671933650970459f, a[5] * a[11], 0.43701937794685364f * a[1] * a[5])))) + (fmaf(0.4264872372150421f, a[14] * a[22], fmaf(0.4264872372150421f, a[10] * a[18], fmaf(0.49553337693214417f, a[6] * a[12], 0.5046265125274658f * a[2] * a[6]))) + fmaf(0.3257350027561188f, a[15] * a[23], fmaf(0.4768272340297699f, a[11] * a[19], fmaf(0.4671933650970459f, a[7] * a[13], 0.43701937794685364f * a[3] * a[7])))));
        o[3] = ((fmaf(0.46065887808799744f, a[15] * a[24], fmaf(0.33716776967048645f, a[13] * a[22], fmaf(-0.15078601241111755f, a[10] * a[19], fmaf(0.45235803723335266f, a[8] * a[15], fmaf(0.4046013057231903f, a[6] * a[13], fmaf(0.43701937794685364f, a[3] * a[8], 0.564189612865448f * a[0] * a[3])))))) + fmaf(-0.15078601241111755f, a[14] * a[21], fmaf(0.33716776967048645f, a[11] * a[18], fmaf(0.46065887808799744f, a[9] * a[16], fmaf(-0.28609633445739746f, a[7] * a[12], fmaf(0.45235803723335266f, a[4] * a[9], 0.43701937794685364f * a[1] * a[4])))))) + (fmaf(0.3989422917366028f, a[14] * a[23], fmaf(0.3893277943134308f, a[12] * a[21], fmaf(-0.08705634623765945f, a[9] * a[18], fmaf(0.36934879422187805f, a[7] * a[14], fmaf(-0.11679834127426147f, a[4] * a[11], 0.43701937794685364f * a[2] * a[7]))))) + fmaf(-0.08705634623765945f, a[15] * a[22], fmaf(-0.3015720248222351f, a[13] * a[20], fmaf(0.3989422917366028f, a[10] * a[17], fmaf(-0.11679834127426147f, a[8] * a[13], fmaf(0.36934879422187805f, a[5] * a[10], -0.2523132562637329f * a[3] * a[6])))))));
        o[4] = ((fmaf(0.15016163885593414f, a[18] * a[24], fmaf(0.18806318938732147f, a[11] * a[15], fmaf(0.4768272340297699f, a[8] * a[16], fmaf(-0.33716776967048645f, a[5] * a[23], fmaf(0.08059851080179214f, a[4] * a[20], fmaf(0.36934879422187805f, a[2] * a[10], 0.564189612865448f * a[0] * a[4])))))) + fmaf(0.2837788164615631f, a[19] * a[21], fmaf(-0.15016163885593414f, a[16] * a[22], fmaf(-0.18806318938732147f, a[9] * a[13], fmaf(0.31215670704841614f, a[6] * a[18], fmaf(-0.4768272340297699f, a[4] * a[24], fmaf(0.45235803723335266f, a[3] * a[9], 0.43701937794685364f * a[1] * a[3]))))))) + (fmaf(0.22524245083332062f, a[19] * a[23], fmaf(-0.22524245083332062f, a[17] * a[21], fmaf(-0.37612637877464294f, a[10] * a[12], fmaf(0.33716776967048645f, a[7] * a[17], fmaf(0.31215670704841614f, a[5] * a[7], fmaf(-0.11679834127426147f, a[3] * a[11], -0.11679834127426147f * a[1] * a[13])))))) + fmaf(-0.38072922825813293f, a[18] * a[20], fmaf(0.2913462519645691f, a[11] * a[13], fmaf(-0.12743744254112244f, a[7] * a[19], fmaf(-0.12743744254112244f, a[5] * a[21], fmaf(-0.360447496175766f, a[4] * a[6], -0.45235803723335266f * a[1] * a[15])))))));
        o[5] = ((fmaf(-0.18059572577476501f, a[19] * a[22], fmaf(-0.2809267044067383f, a[17] * a[24], fmaf(0.11894160509109497f, a[11] * a[12], fmaf(0.12743744254112244f, a[8] * a[19], fmaf(-0.360447496175766f, a[5] * a[22], fmaf(-0.33716776967048645f, a[4] * a[23], fmaf(0.4671933650970459f, a[2] * a[11], 0.564189612865448f * a[0] * a[5]))))))) + fmaf(0.18059572577476501f, a[18] * a[21], fmaf(-0.23032943904399872f, a[11] * a[14], fmaf(0.2973540127277374f, a[9] * a[14], fmaf(0.44145622849464417f, a[6] * a[19], fmaf(0.180223748087883f, a[5] * a[6], fmaf(0.36934879422187805f, a[3] * a[10], 0.43701937794685364f * a[1] * a[2]))))))) + (fmaf(-0.26545077562332153f, a[18] * a[23], fmaf(0.2809267044067383f, a[16] * a[23], fmaf(0.23032943904399872f, a[10] * a[13], fmaf(0.360447496175766f, a[7] * a[18], fmaf(-0.31215670704841614f, a[5] * a[8], fmaf(0.31215670704841614f, a[4] * a[7], -0.28609633445739746f * a[1] * a[12])))))) + fmaf(0.08973874151706696f, a[19] * a[20], fmaf(0.26545077562332153f, a[17] * a[22], fmaf(-0.2973540127277374f, a[10] * a[15], fmaf(0.33716776967048645f, a[8] * a[17], fmaf(-0.3223940432071686f, a[5] * a[20], fmaf(-0.12743744254112244f, a[4] * a[21], -0.36934879422187805f * a[1] * a[14]))))))));
        o[6] = ((fmaf(0.06553591042757034f, a[22] * a[22], fmaf(0.06553591042757034f, a[18] * a[18], fmaf(0.12615662813186646f, a[13] * a[13], fmaf(0.31215670704841614f, a[8] * a[22], fmaf(0.48359107971191406f, a[6] * a[20], fmaf(0.31215670704841614f, a[4] * a[18], fmaf(0.49553337693214417f, a[2] * a[12], 0.564189612865448f * a[0] * a[6]))))))) + fmaf(-0.057343922555446625f, a[23] * a[23], fmaf(0.1392638087272644f, a[19] * a[19], fmaf(-0.2102610468864441f, a[15] * a[15], fmaf(-0.2102610468864441f, a[9] * a[9], fmaf(0.0901118740439415f, a[7] * a[7], fmaf(0.0901118740439415f, a[5] * a[5], fmaf(-0.12615662813186646f, a[3] * a[3], -0.12615662813186646f * a[1] * a[1])))))))) + (fmaf(-0.2293756902217865f, a[24] * a[24], fmaf(0.16383977234363556f, a[20] * a[20], fmaf(-0.2293756902217865f, a[16] * a[16], fmaf(0.12615662813186646f, a[11] * a[11], fmaf(0.44145622849464417f, a[7] * a[21], fmaf(0.44145622849464417f, a[5] * a[19], fmaf(0.4046013057231903f, a[3] * a[13], 0.4046013057231903f * a[1] * a[11]))))))) + fmaf(0.1392638087272644f, a[21] * a[21], fmaf(-0.057343922555446625f, a[17] * a[17], fmaf(0.16820883750915527f, a[12] * a[12], fmaf(-0.180223748087883f, a[8] * a[8], fmaf(0.180223748087883f, a[6] * a[6], fmaf(-0.180223748087883f, a[4] * a[4], 0.2523132562637329f * a[2] * a[2]))))))));
        o[7] = ((fmaf(0.2809267044067383f, a[23] * a[24], fmaf(0.18059572577476501f, a[18] * a[19], fmaf(0.23032943904399872f, a[13] * a[14], fmaf(0.33716776967048645f, a[8] * a[23], fmaf(0.31215670704841614f, a[7] * a[8], fmaf(-0.12743744254112244f, a[4] * a[19], fmaf(-0.28609633445739746f, a[3] * a[12], 0.564189612865448f * a[0] * a[7]))))))) + fmaf(0.08973874151706696f, a[20] * a[21], fmaf(0.2973540127277374f, a[14] * a[15], fmaf(0.2973540127277374f, a[9] * a[10], fmaf(-0.3223940432071686f, a[7] * a[20], fmaf(0.360447496175766f, a[5] * a[18], fmaf(0.36934879422187805f, a[3] * a[14], 0.36934879422187805f * a[1] * a[10]))))))) + (fmaf(0.18059572577476501f, a[21] * a[22], fmaf(0.2809267044067383f, a[16] * a[17], fmaf(0.23032943904399872f, a[10] * a[11], fmaf(0.360447496175766f, a[7] * a[22], fmaf(0.180223748087883f, a[6] * a[7], fmaf(0.31215670704841614f, a[4] * a[5], 0.43701937794685364f * a[2] * a[3])))))) + fmaf(0.26545077562332153f, a[22] * a[23], fmaf(0.26545077562332153f, a[17] * a[18], fmaf(0.11894160509109497f, a[12] * a[13], fmaf(-0.12743744254112244f, a[8] * a[21], fmaf(0.44145622849464417f, a[6] * a[21], fmaf(0.33716776967048645f, a[4] * a[17], 0.4671933650970459f * a[2] * a[13]))))))));
        o[8] = ((fmaf(0.14188940823078156f, a[21] * a[21], fmaf(-0.15016163885593414f, a[16] * a[18], fmaf(-0.14567312598228455f, a[11] * a[11], fmaf(0.33716776967048645f, a[7] * a[23], fmaf(-0.360447496175766f, a[6] * a[8], fmaf(0.4768272340297699f, a[4] * a[16], fmaf(0.36934879422187805f, a[2] * a[14], 0.564189612865448f * a[0] * a[8]))))))) + fmaf(-0.22524245083332062f, a[21] * a[23], fmaf(-0.22524245083332062f, a[17] * a[19], fmaf(-0.37612637877464294f, a[12] * a[14], fmaf(0.08059851080179214f, a[8] * a[20], fmaf(0.31215670704841614f, a[6] * a[22], fmaf(-0.15607835352420807f, a[5] * a[5], fmaf(0.21850968897342682f, a[3] * a[3], -0.21850968897342682f * a[1] * a[1])))))))) + (fmaf(-0.15016163885593414f, a[22] * a[24], fmaf(-0.14188940823078156f, a[19] * a[19], fmaf(0.14567312598228455f, a[13] * a[13], fmaf(0.4768272340297699f, a[8] * a[24], fmaf(0.15607835352420807f, a[7] * a[7], fmaf(0.33716776967048645f, a[5] * a[17], fmaf(-0.11679834127426147f, a[3] * a[13], 0.45235803723335266f * a[1] * a[9]))))))) + fmaf(-0.38072922825813293f, a[20] * a[22], fmaf(-0.18806318938732147f, a[13] * a[15], fmaf(-0.18806318938732147f, a[9] * a[11], fmaf(-0.12743744254112244f, a[7] * a[21], fmaf(0.12743744254112244f, a[5] * a[19], fmaf(0.45235803723335266f, a[3] * a[15], 0.11679834127426147f * a[1] * a[11]))))))));
        o[9] = ((fmaf(-0.19864517450332642f, a[14] * a[19], fmaf(0.23504012823104858f, a[11] * a[24], fmaf(-0.18806318938732147f, a[8] * a[11], fmaf(-0.18806318938732147f, a[4] * a[13], fmaf(0.3257350027561188f, a[2] * a[17], 0.564189612865448f * a[0] * a[9]))))) + fmaf(-0.40710145235061646f, a[12] * a[17], fmaf(0.1538698822259903f, a[9] * a[20], fmaf(0.2973540127277374f, a[5] * a[14], fmaf(0.45235803723335266f, a[3] * a[4], 0.45235803723335266f * a[1] * a[8]))))) + (fmaf(-0.23504012823104858f, a[13] * a[16], fmaf(-0.19864517450332642f, a[10] * a[21], fmaf(-0.4205220937728882f, a[6] * a[9], fmaf(0.46065887808799744f, a[3] * a[16], -0.08705634623765945f * a[1] * a[22])))) + fmaf(0.2665104568004608f, a[13] * a[18], fmaf(0.2665104568004608f, a[11] * a[22], fmaf(0.2973540127277374f, a[7] * a[10], fmaf(-0.08705634623765945f, a[3] * a[18], -0.46065887808799744f * a[1] * a[24]))))));
        o[10] = ((fmaf(0.13570047914981842f, a[13] * a[17], fmaf(-0.3034355044364929f, a[10] * a[24], fmaf(0.2973540127277374f, a[7] * a[9], fmaf(-0.15078601241111755f, a[3] * a[19], fmaf(0.36934879422187805f, a[2] * a[4], 0.564189612865448f * a[0] * a[10]))))) + fmaf(0.20515984296798706f, a[13] * a[19], fmaf(0.20515984296798706f, a[11] * a[21], fmaf(0.23032943904399872f, a[7] * a[11], fmaf(-0.37612637877464294f, a[4] * a[12], fmaf(0.4264872372150421f, a[2] * a[18], 0.36934879422187805f * a[1] * a[7])))))) + (fmaf(0.3034355044364929f, a[14] * a[16], fmaf(-0.13570047914981842f, a[11] * a[23], fmaf(-0.19864517450332642f, a[9] * a[21], fmaf(0.23032943904399872f, a[5] * a[13], fmaf(0.36934879422187805f, a[3] * a[5], -0.15078601241111755f * a[1] * a[21]))))) + fmaf(0.19864517450332642f, a[15] * a[19], fmaf(-0.08883681893348694f, a[12] * a[18], fmaf(-0.35902974009513855f, a[10] * a[20], fmaf(-0.2973540127277374f, a[5] * a[15], fmaf(0.3989422917366028f, a[3] * a[17], -0.3989422917366028f * a[1] * a[23])))))));
        o[11] = ((fmaf(-0.2665104568004608f, a[15] * a[18], fmaf(0.2293756902217865f, a[13] * a[18], fmaf(-0.13570047914981842f, a[10] * a[23], fmaf(-0.2913462519645691f, a[8] * a[11], fmaf(-0.23032943904399872f, a[5] * a[14], fmaf(0.33716776967048645f, a[3] * a[18], fmaf(-0.33716776967048645f, a[1] * a[22], 0.564189612865448f * a[0] * a[11]))))))) + fmaf(0.13570047914981842f, a[14] * a[17], fmaf(0.051289960741996765f, a[11] * a[20], fmaf(0.2665104568004608f, a[9] * a[22], fmaf(0.2523132562637329f, a[6] * a[11], fmaf(0.2913462519645691f, a[4] * a[13], fmaf(0.4671933650970459f, a[2] * a[5], 0.4046013057231903f * a[1] * a[6]))))))) + (fmaf(-0.20515984296798706f, a[14] * a[19], fmaf(-0.2293756902217865f, a[11] * a[22], fmaf(0.23504012823104858f, a[9] * a[24], fmaf(0.23032943904399872f, a[7] * a[10], fmaf(0.18806318938732147f, a[4] * a[15], fmaf(0.4768272340297699f, a[2] * a[19], 0.11679834127426147f * a[1] * a[8])))))) + fmaf(-0.23504012823104858f, a[15] * a[16], fmaf(0.19864517450332642f, a[12] * a[19], fmaf(0.20515984296798706f, a[10] * a[21], fmaf(-0.18806318938732147f, a[8] * a[9], fmaf(0.11894160509109497f, a[5] * a[12], fmaf(-0.11679834127426147f, a[3] * a[4], -0.3015720248222351f * a[1] * a[20]))))))));
        o[12] = ((fmaf(0.19864517450332642f, a[13] * a[21], fmaf(-0.40710145235061646f, a[9] * a[17], fmaf(0.11894160509109497f, a[5] * a[11], fmaf(0.4924650490283966f, a[2] * a[20], 0.564189612865448f * a[0] * a[12])))) + fmaf(-0.08883681893348694f, a[14] * a[22], fmaf(-0.08883681893348694f, a[10] * a[18], fmaf(0.33641767501831055f, a[6] * a[12], fmaf(-0.28609633445739746f, a[3] * a[7], -0.28609633445739746f * a[1] * a[5]))))) + (fmaf(-0.40710145235061646f, a[15] * a[23], fmaf(0.19864517450332642f, a[11] * a[19], fmaf(0.11894160509109497f, a[7] * a[13], fmaf(0.3893277943134308f, a[3] * a[21], 0.3893277943134308f * a[1] * a[19])))) + fmaf(0.3077397644519806f, a[12] * a[20], fmaf(-0.37612637877464294f, a[8] * a[14], fmaf(-0.37612637877464294f, a[4] * a[10], 0.49553337693214417f * a[2] * a[6])))));
        o[13] = ((fmaf(-0.23504012823104858f, a[15] * a[24], fmaf(0.2293756902217865f, a[13] * a[22], fmaf(0.20515984296798706f, a[10] * a[19], fmaf(-0.18806318938732147f, a[8] * a[15], fmaf(0.2523132562637329f, a[6] * a[13], fmaf(0.33716776967048645f, a[3] * a[22], fmaf(0.4768272340297699f, a[2] * a[21], 0.564189612865448f * a[0] * a[13]))))))) + fmaf(0.20515984296798706f, a[14] * a[21], fmaf(0.2293756902217865f, a[11] * a[18], fmaf(-0.23504012823104858f, a[9] * a[16], fmaf(0.11894160509109497f, a[7] * a[12], fmaf(-0.18806318938732147f, a[4] * a[9], fmaf(0.4046013057231903f, a[3] * a[6], -0.11679834127426147f * a[1] * a[4]))))))) + (fmaf(0.13570047914981842f, a[14] * a[23], fmaf(0.19864517450332642f, a[12] * a[21], fmaf(0.2665104568004608f, a[9] * a[18], fmaf(0.23032943904399872f, a[7] * a[14], fmaf(0.2913462519645691f, a[4] * a[11], fmaf(-0.11679834127426147f, a[3] * a[8], 0.33716776967048645f * a[1] * a[18])))))) + fmaf(0.2665104568004608f, a[15] * a[22], fmaf(0.051289960741996765f, a[13] * a[20], fmaf(0.13570047914981842f, a[10] * a[17], fmaf(0.2913462519645691f, a[8] * a[13], fmaf(0.23032943904399872f, a[5] * a[10], fmaf(-0.3015720248222351f, a[3] * a[20], 0.4671933650970459f * a[2] * a[7]))))))));
        o[14] = ((fmaf(0.13570047914981842f, a[13] * a[23], fmaf(0.13570047914981842f, a[11] * a[17], fmaf(0.2973540127277374f, a[7] * a[15], fmaf(0.3989422917366028f, a[3] * a[23], fmaf(0.36934879422187805f, a[2] * a[8], 0.564189612865448f * a[0] * a[14]))))) + fmaf(-0.35902974009513855f, a[14] * a[20], fmaf(-0.20515984296798706f, a[11] * a[19], fmaf(-0.37612637877464294f, a[8] * a[12], fmaf(0.2973540127277374f, a[5] * a[9], fmaf(0.4264872372150421f, a[2] * a[22], -0.36934879422187805f * a[1] * a[5])))))) + (fmaf(0.3034355044364929f, a[14] * a[24], fmaf(-0.08883681893348694f, a[12] * a[22], fmaf(-0.19864517450332642f, a[9] * a[19], fmaf(-0.23032943904399872f, a[5] * a[11], fmaf(0.36934879422187805f, a[3] * a[7], 0.3989422917366028f * a[1] * a[17]))))) + fmaf(-0.19864517450332642f, a[15] * a[21], fmaf(0.20515984296798706f, a[13] * a[21], fmaf(0.3034355044364929f, a[10] * a[16], fmaf(0.23032943904399872f, a[7] * a[13], fmaf(-0.15078601241111755f, a[3] * a[21], 0.15078601241111755f * a[1] * a[19])))))));
        o[15] = ((fmaf(0.1538698822259903f, a[15] * a[20], fmaf(-0.40710145235061646f, a[12] * a[23], fmaf(-0.18806318938732147f, a[8] * a[13], fmaf(0.18806318938732147f, a[4] * a[11], fmaf(0.3257350027561188f, a[2] * a[23], 0.564189612865448f * a[0] * a[15]))))) + fmaf(0.2665104568004608f, a[13] * a[22], fmaf(0.19864517450332642f, a[10] * a[19], fmaf(-0.2973540127277374f, a[5] * a[10], fmaf(0.45235803723335266f, a[3] * a[8], -0.45235803723335266f * a[1] * a[4]))))) + (fmaf(-0.23504012823104858f, a[13] * a[24], fmaf(-0.23504012823104858f, a[11] * a[16], fmaf(-0.4205220937728882f, a[6] * a[15], fmaf(-0.08705634623765945f, a[3] * a[22], 0.46065887808799744f * a[1] * a[16])))) + fmaf(-0.19864517450332642f, a[14] * a[21], fmaf(-0.2665104568004608f, a[11] * a[18], fmaf(0.2973540127277374f, a[7] * a[14], fmaf(0.46065887808799744f, a[3] * a[24], 0.08705634623765945f * a[1] * a[18]))))));
        o[16] = ((fmaf(0.21305061876773834f, a[16] * a[20], fmaf(-0.15016163885593414f, a[8] * a[18], fmaf(-0.15016163885593414f, a[4] * a[22], 0.564189612865448f * a[0] * a[16]))) + fmaf(-0.23819781839847565f, a[17] * a[21], fmaf(-0.23504012823104858f, a[9] * a[13], fmaf(0.2809267044067383f, a[5] * a[23], 0.46065887808799744f * a[1] * a[15])))) + (fmaf(0.2700909376144409f, a[18] * a[22], fmaf(0.3034355044364929f, a[10] * a[14], fmaf(-0.458751380443573f, a[6] * a[16], 0.46065887808799744f * a[3] * a[9]))) + fmaf(-0.23819781839847565f, a[19] * a[23], fmaf(-0.23504012823104858f, a[11] * a[15], fmaf(0.2809267044067383f, a[7] * a[17], 0.4768272340297699f * a[4] * a[8])))));
        o[17] = ((fmaf(0.23819781839847565f, a[19] * a[24], fmaf(-0.23819781839847565f, a[16] * a[21], fmaf(-0.22524245083332062f, a[8] * a[19], fmaf(-0.2809267044067383f, a[5] * a[24], fmaf(0.33716776967048645f, a[4] * a[7], 0.564189612865448f * a[0] * a[17]))))) + fmaf(-0.3195759057998657f, a[17] * a[20], fmaf(-0.40710145235061646f, a[9] * a[12], fmaf(-0.11468784511089325f, a[6] * a[17], fmaf(-0.22524245083332062f, a[4] * a[21], 0.3989422917366028f * a[1] * a[14]))))) + (fmaf(0.09003031253814697f, a[18] * a[21], fmaf(0.13570047914981842f, a[10] * a[13], fmaf(0.2809267044067383f, a[7] * a[16], fmaf(0.33716776967048645f, a[5] * a[8], 0.3257350027561188f * a[2] * a[9])))) + fmaf(0.09003031253814697f, a[19] * a[22], fmaf(0.13570047914981842f, a[11] * a[14], fmaf(0.26545077562332153f, a[7] * a[18], fmaf(0.26545077562332153f, a[5] * a[22], 0.3989422917366028f * a[3] * a[10]))))));
        o[18] = ((fmaf(0.20416957139968872f, a[19] * a[21], fmaf(0.2700909376144409f, a[16] * a[22], fmaf(0.2665104568004608f, a[9] * a[13], fmaf(0.13107182085514069f, a[6] * a[18], fmaf(0.15016163885593414f, a[4] * a[24], fmaf(-0.08705634623765945f, a[3] * a[9], 0.564189612865448f * a[0] * a[18])))))) + fmaf(-0.09003031253814697f, a[19] * a[23], fmaf(0.09003031253814697f, a[17] * a[21], fmaf(-0.08883681893348694f, a[10] * a[12], fmaf(0.26545077562332153f, a[7] * a[17], fmaf(0.360447496175766f, a[5] * a[7], fmaf(0.33716776967048645f, a[3] * a[11], 0.33716776967048645f * a[1] * a[13]))))))) + (fmaf(-0.1673969030380249f, a[18] * a[20], fmaf(0.2293756902217865f, a[11] * a[13], fmaf(0.18059572577476501f, a[7] * a[19], fmaf(0.18059572577476501f, a[5] * a[21], fmaf(0.31215670704841614f, a[4] * a[6], 0.08705634623765945f * a[1] * a[15]))))) + fmaf(-0.2700909376144409f, a[18] * a[24], fmaf(-0.2665104568004608f, a[11] * a[15], fmaf(-0.15016163885593414f, a[8] * a[16], fmaf(-0.26545077562332153f, a[5] * a[23], fmaf(-0.38072922825813293f, a[4] * a[20], 0.4264872372150421f * a[2] * a[10])))))));
        o[19] = ((fmaf(0.20416957139968872f, a[18] * a[21], fmaf(-0.20515984296798706f, a[11] * a[14], fmaf(-0.19864517450332642f, a[9] * a[14], fmaf(0.2785276174545288f, a[6] * a[19], fmaf(0.44145622849464417f, a[5] * a[6], fmaf(-0.15078601241111755f, a[3] * a[10], 0.564189612865448f * a[0] * a[19])))))) + fmaf(-0.09003031253814697f, a[18] * a[23], fmaf(-0.23819781839847565f, a[16] * a[23], fmaf(0.20515984296798706f, a[10] * a[13], fmaf(0.18059572577476501f, a[7] * a[18], fmaf(0.12743744254112244f, a[5] * a[8], fmaf(-0.12743744254112244f, a[4] * a[7], 0.3893277943134308f * a[1] * a[12]))))))) + (fmaf(0.13696110248565674f, a[19] * a[20], fmaf(0.09003031253814697f, a[17] * a[22], fmaf(0.19864517450332642f, a[10] * a[15], fmaf(-0.22524245083332062f, a[8] * a[17], fmaf(0.08973874151706696f, a[5] * a[20], fmaf(0.2837788164615631f, a[4] * a[21], 0.15078601241111755f * a[1] * a[14])))))) + fmaf(-0.20416957139968872f, a[19] * a[22], fmaf(0.23819781839847565f, a[17] * a[24], fmaf(0.19864517450332642f, a[11] * a[12], fmaf(-0.2837788164615631f, a[8] * a[19], fmaf(-0.18059572577476501f, a[5] * a[22], fmaf(0.22524245083332062f, a[4] * a[23], 0.4768272340297699f * a[2] * a[11]))))))));
        o[20] = ((fmaf(-0.15978795289993286f, a[23] * a[23], fmaf(0.06848055124282837f, a[19] * a[19], fmaf(0.07693494111299515f, a[15] * a[15], fmaf(0.025644980370998383f, a[11] * a[11], fmaf(0.04029925540089607f, a[8] * a[8], fmaf(0.24179553985595703f, a[6] * a[6], fmaf(0.04029925540089607f, a[4] * a[4], 0.564189612865448f * a[0] * a[20]))))))) + fmaf(0.10652530938386917f, a[24] * a[24], fmaf(0.13696110248565674f, a[20] * a[20], fmaf(0.10652530938386917f, a[16] * a[16], fmaf(0.1538698822259903f, a[12] * a[12], fmaf(-0.38072922825813293f, a[8] * a[22], fmaf(0.3276795446872711f, a[6] * a[20], fmaf(-0.38072922825813293f, a[4] * a[18], -0.3015720248222351f * a[1] * a[11])))))))) + (fmaf(0.06848055124282837f, a[21] * a[21], fmaf(-0.15978795289993286f, a[17] * a[17], fmaf(0.025644980370998383f, a[13] * a[13], fmaf(0.07693494111299515f, a[9] * a[9], fmaf(-0.1611970216035843f, a[7] * a[7], fmaf(-0.1611970216035843f, a[5] * a[5], 0.4924650490283966f * a[2] * a[12])))))) + fmaf(-0.08369845151901245f, a[22] * a[22], fmaf(-0.08369845151901245f, a[18] * a[18], fmaf(-0.17951487004756927f, a[14] * a[14], fmaf(-0.17951487004756927f, a[10] * a[10], fmaf(0.08973874151706696f, a[7] * a[21], fmaf(0.08973874151706696f, a[5] * a[19], -0.3015720248222351f * a[3] * a[13]))))))));
        o[21] = ((fmaf(0.13696110248565674f, a[20] * a[21], fmaf(-0.19864517450332642f, a[14] * a[15], fmaf(-0.19864517450332642f, a[9] * a[10], fmaf(0.08973874151706696f, a[7] * a[20], fmaf(0.18059572577476501f, a[5] * a[18], fmaf(-0.15078601241111755f, a[3] * a[14], 0.564189612865448f * a[0] * a[21])))))) + fmaf(0.20416957139968872f, a[21] * a[22], fmaf(-0.23819781839847565f, a[16] * a[17], fmaf(0.20515984296798706f, a[10] * a[11], fmaf(0.18059572577476501f, a[7] * a[22], fmaf(0.44145622849464417f, a[6] * a[7], fmaf(-0.12743744254112244f, a[4] * a[5], -0.15078601241111755f * a[1] * a[10]))))))) + (fmaf(0.09003031253814697f, a[22] * a[23], fmaf(0.09003031253814697f, a[17] * a[18], fmaf(0.19864517450332642f, a[12] * a[13], fmaf(0.2837788164615631f, a[8] * a[21], fmaf(0.2785276174545288f, a[6] * a[21], fmaf(-0.22524245083332062f, a[4] * a[17], 0.4768272340297699f * a[2] * a[13])))))) + fmaf(-0.23819781839847565f, a[23] * a[24], fmaf(0.20416957139968872f, a[18] * a[19], fmaf(0.20515984296798706f, a[13] * a[14], fmaf(-0.22524245083332062f, a[8] * a[23], fmaf(-0.12743744254112244f, a[7] * a[8], fmaf(0.2837788164615631f, a[4] * a[19], 0.3893277943134308f * a[3] * a[12]))))))));
        o[22] = ((fmaf(0.2700909376144409f, a[22] * a[24], fmaf(-0.10208478569984436f, a[19] * a[19], fmaf(0.11468784511089325f, a[13] * a[13], fmaf(-0.15016163885593414f, a[8] * a[24], fmaf(0.180223748087883f, a[7] * a[7], fmaf(0.26545077562332153f, a[5] * a[17], fmaf(0.33716776967048645f, a[3] * a[13], 0.564189612865448f * a[0] * a[22]))))))) + fmaf(-0.1673969030380249f, a[20] * a[22], fmaf(0.2665104568004608f, a[13] * a[15], fmaf(0.2665104568004608f, a[9] * a[11], fmaf(0.18059572577476501f, a[7] * a[21], fmaf(-0.18059572577476501f, a[5] * a[19], fmaf(-0.08705634623765945f, a[3] * a[15], -0.08705634623765945f * a[1] * a[9]))))))) + (fmaf(0.10208478569984436f, a[21] * a[21], fmaf(0.2700909376144409f, a[16] * a[18], fmaf(-0.11468784511089325f, a[11] * a[11], fmaf(0.26545077562332153f, a[7] * a[23], fmaf(0.31215670704841614f, a[6] * a[8], fmaf(-0.15016163885593414f, a[4] * a[16], -0.33716776967048645f * a[1] * a[11])))))) + fmaf(0.09003031253814697f, a[21] * a[23], fmaf(0.09003031253814697f, a[17] * a[19], fmaf(-0.08883681893348694f, a[12] * a[14], fmaf(-0.38072922825813293f, a[8] * a[20], fmaf(0.13107182085514069f, a[6] * a[22], fmaf(-0.180223748087883f, a[5] * a[5], 0.4264872372150421f * a[2] * a[14]))))))));
        o[23] = ((fmaf(-0.23819781839847565f, a[21] * a[24], fmaf(-0.23819781839847565f, a[16] * a[19], fmaf(-0.22524245083332062f, a[8] * a[21], fmaf(-0.11468784511089325f, a[6] * a[23], fmaf(-0.33716776967048645f, a[4] * a[5], 0.564189612865448f * a[0] * a[23]))))) + fmaf(-0.09003031253814697f, a[18] * a[19], fmaf(-0.13570047914981842f, a[10] * a[11], fmaf(0.33716776967048645f, a[7] * a[8], fmaf(0.22524245083332062f, a[4] * a[19], -0.3989422917366028f * a[1] * a[10]))))) + (fmaf(-0.3195759057998657f, a[20] * a[23], fmaf(-0.40710145235061646f, a[12] * a[15], fmaf(0.26545077562332153f, a[7] * a[22], fmaf(0.2809267044067383f, a[5] * a[16], 0.3257350027561188f * a[2] * a[15])))) + fmaf(0.09003031253814697f, a[21] * a[22], fmaf(0.13570047914981842f, a[13] * a[14], fmaf(0.2809267044067383f, a[7] * a[24], fmaf(-0.26545077562332153f, a[5] * a[18], 0.3989422917366028f * a[3] * a[14]))))));
        o[24] = ((fmaf(0.21305061876773834f, a[20] * a[24], fmaf(-0.23504012823104858f, a[13] * a[15], fmaf(0.23841361701488495f, a[8] * a[8], fmaf(0.15016163885593414f, a[4] * a[18], 0.564189612865448f * a[0] * a[24])))) + fmaf(-0.23819781839847565f, a[21] * a[23], fmaf(0.15171775221824646f, a[14] * a[14], fmaf(-0.15016163885593414f, a[8] * a[22], fmaf(-0.2809267044067383f, a[5] * a[17], -0.46065887808799744f * a[1] * a[9]))))) + (fmaf(0.13504546880722046f, a[22] * a[22], fmaf(0.23819781839847565f, a[17] * a[19], fmaf(0.23504012823104858f, a[9] * a[11], fmaf(-0.458751380443573f, a[6] * a[24], 0.46065887808799744f * a[3] * a[15])))) + fmaf(-0.13504546880722046f, a[18] * a[18], fmaf(-0.15171775221824646f, a[10] * a[10], fmaf(0.2809267044067383f, a[7] * a[23], -0.23841361701488495f * a[4] * a[4])))));
    }
};

#if defined(SHS_NB) && SHS_NB == 6
// lane-pair rules: product, then projected exponential (plain, weighted)
static __device__ const float kLpLeg6[96] = {0.09627555310726166f, 0.19014164805412292f, 0.18406742811203003f, 0.04652512073516846f, 0.15714223682880402f, 0.25652122497558594f, 0.014512873254716396f, 0.06856247037649155f, 0.004373585805296898f, 0.026470474898815155f, 0.0012942698085680604f, 0.00037873201654292643f, 0.16013231873512268f, 0.19700372219085693f, 0.15417835116386414f, 0.09990215301513672f, 0.21137355268001556f, 0.0f, 0.036872684955596924f, 0.1080133244395256f, 0.012599730864167213f, 0.0f, 0.004122147336602211f, 0.0f, 0.12515482306480408f, 0.12649886310100555f, -0.09113376587629318f, 0.13102267682552338f, 0.2663714289665222f, 0.06967514008283615f, 0.08854003250598907f, 0.2639823257923126f, 0.05780312418937683f, 0.22584053874015808f, 0.03705662116408348f, 0.023490939289331436f, 0.17269699275493622f, 0.022869709879159927f, -0.16741353273391724f, 0.23340384662151337f, 0.20621128380298615f, 0.0f, 0.18662303686141968f, 0.279779314994812f, 0.1381494402885437f, 0.0f, 0.09791262447834015f, 0.0f, 0.1403641700744629f, -0.026905516162514687f, -0.1376871019601822f, 0.20683826506137848f, 0.07370050996541977f, -0.2425079345703125f, 0.19674327969551086f, 0.1590183526277542f, 0.180795356631279f, 0.22271154820919037f, 0.16314642131328583f, 0.1455753594636917f, 0.12776632606983185f, -0.15799476206302643f, 0.014452863484621048f, 0.24306106567382812f, -0.1587732434272766f, 0.0f, 0.2735573649406433f, -0.07777585834264755f, 0.2850414514541626f, 0.0f, 0.2843632102012634f, 0.0f, 0.14731866121292114f, -0.14808091521263123f, 0.1121562197804451f, 0.25083374977111816f, -0.1951584368944168f, 0.1285189688205719f, 0.27568212151527405f, -0.18251359462738037f, 0.2927181124687195f, -0.16920839250087738f, 0.305206298828125f, 0.31467151641845703f, 0.04680580645799637f, -0.10123119503259659f, 0.142460435628891f, 0.10288506746292114f, -0.17417211830615997f, 0.0f, 0.13379472494125366f, -0.1994764804840088f, 0.16108393669128418f, 0.0f, 0.18568259477615356f, 0.0f};
static __device__ const float kLeLeg6[288] = {0.282094806432724f, 0.5962111353874207f, 0.6966167688369751f, 0.0933968797326088f, 0.33349815011024475f, 0.6064973473548889f, 0.019960161298513412f, 0.09929478168487549f, 0.004121108911931515f, 0.026212655007839203f, 0.0008355395984835923f, 0.0001675097446423024f, 0.4795929789543152f, 0.66567063331604f, 0.6931184530258179f, 0.20499086380004883f, 0.47001588344573975f, 0.0f, 0.05183584615588188f, 0.16249744594097137f, 0.012135355733335018f, 0.0f, 0.002720072865486145f, 0.0f, 0.282094806432724f, 0.4580381512641907f, 0.19715876877307892f, 0.20877224206924438f, 0.6028831005096436f, 0.694404661655426f, 0.099734365940094f, 0.40785059332847595f, 0.04602940008044243f, 0.2426128387451172f, 0.020860688760876656f, 0.00934850238263607f, 0.44175395369529724f, 0.3667958080768585f, -0.013120017945766449f, 0.4220680892467499f, 0.7035349011421204f, 0.0f, 0.23857153952121735f, 0.5745615363121033f, 0.12484792619943619f, 0.0f, 0.06255322694778442f, 0.0f, 0.282094806432724f, 0.2454536110162735f, -0.2628938853740692f, 0.31180721521377563f, 0.5727651119232178f, 0.02309684082865715f, 0.22247010469436646f, 0.6067496538162231f, 0.15334708988666534f, 0.5511578917503357f, 0.10379639267921448f, 0.06947188824415207f, 0.3761763870716095f, -0.010414783842861652f, -0.3923318088054657f, 0.5367931723594666f, 0.37777870893478394f, 0.0f, 0.4531651437282562f, 0.5848469138145447f, 0.35418701171875f, 0.0f, 0.2650418281555176f, 0.0f, 0.282094806432724f, 0.010984186083078384f, -0.3367987275123596f, 0.3954535126686096f, 0.2680802643299103f, -0.4877561032772064f, 0.3578410744667053f, 0.43838274478912354f, 0.31282636523246765f, 0.5458644032478333f, 0.2685464322566986f, 0.2279583215713501f, 0.2869650423526764f, -0.27950891852378845f, -0.11332645267248154f, 0.5193423628807068f, -0.1861763745546341f, 0.0f, 0.5560482740402222f, 0.032114166766405106f, 0.5511856079101562f, 0.0f, 0.5231051445007324f, 0.0f, 0.282094806432724f, -0.18737411499023438f, -0.044248729944229126f, 0.45434778928756714f, -0.13748858869075775f, -0.21471181511878967f, 0.47236329317092896f, -0.021640226244926453f, 0.4744410812854767f, 0.08564011752605438f, 0.46794116497039795f, 0.4563734233379364f, 0.17972339689731598f, -0.3189375698566437f, 0.28745853900909424f, 0.3736993372440338f, -0.4697921574115753f, 0.0f, 0.4596995711326599f, -0.4528975486755371f, 0.523543119430542f, 0.0f, 0.5708690881729126f, 0.0f, 0.282094806432724f, -0.3005523085594177f, 0.26849499344825745f, 0.48475590348243713f, -0.4178895950317383f, 0.3530324697494507f, 0.5377067923545837f, -0.414544939994812f, 0.5762172937393188f, -0.4103360176086426f, 0.6063591837882996f, 0.6309481859207153f, 0.061189357191324234f, -0.13653768599033356f, 0.2038392275571823f, 0.13574638962745667f, -0.24025601148605347f, 0.0f, 0.1781618595123291f, -0.2815471291542053f, 0.21648497879505157f, 0.0f, 0.2518526315689087f, 0.0f, 0.003484004409983754f, 0.007363489829003811f, 0.008603546768426895f, 0.0011534957448020577f, 0.004118860233575106f, 0.007490530144423246f, 0.00024651744752191007f, 0.0012263376265764236f, 5.08976518176496e-05f, 0.000323738728184253f, 1.0319310604245402e-05f, 2.068824642265099e-06f, 0.005923200864344835f, 0.008221347816288471f, 0.008560341782867908f, 0.0025317342951893806f, 0.005804919172078371f, 0.0f, 0.0006401973078027368f, 0.0020069205202162266f, 0.00014987739268690348f, 0.0f, 3.3594187698327005e-05f, 0.0f, 0.007897709496319294f, 0.01282353326678276f, 0.005519785452634096f, 0.005844923667609692f, 0.016878707334399223f, 0.01944100484251976f, 0.0027922282461076975f, 0.011418450623750687f, 0.0012886689510196447f, 0.006792346481233835f, 0.00058402941795066f, 0.0002617267600726336f, 0.012367631308734417f, 0.010269053280353546f, -0.00036731656291522086f, 0.011816493235528469f, 0.019696621224284172f, 0.0f, 0.006679203826934099f, 0.016085797920823097f, 0.0034953237045556307f, 0.0f, 0.0017512808553874493f, 0.0f, 0.011822143569588661f, 0.010286569595336914f, -0.011017464101314545f, 0.013067344203591347f, 0.02400367334485054f, 0.0009679518989287317f, 0.009323367848992348f, 0.025427913293242455f, 0.006426532287150621f, 0.02309815213084221f, 0.004349941853433847f, 0.002911456162109971f, 0.015764953568577766f, -0.0004364670312497765f, -0.01644200086593628f, 0.022496148943901062f, 0.01583210565149784f, 0.0f, 0.01899143122136593f, 0.024510003626346588f, 0.014843413606286049f, 0.0f, 0.011107482016086578f, 0.0f, 0.015004370361566544f, 0.0005842390237376094f, -0.017914025112986565f, 0.021033819764852524f, 0.01425895094871521f, -0.025943312793970108f, 0.019033247604966164f, 0.023317188024520874f, 0.01663895510137081f, 0.029034042730927467f, 0.014283744618296623f, 0.01212489977478981f, 0.01526341401040554f, -0.014866829849779606f, -0.006027732975780964f, 0.027623355388641357f, -0.009902555495500565f, 0.0f, 0.029575711116194725f, 0.0017081238329410553f, 0.02931707166135311f, 0.0f, 0.027823494747281075f, 0.0f, 0.017243947833776474f, -0.011453842744231224f, -0.0027048452757298946f, 0.02777346409857273f, -0.008404430001974106f, -0.013124947436153889f, 0.028874719515442848f, -0.001322828116826713f, 0.02900172956287861f, 0.005235026590526104f, 0.028604403138160706f, 0.027897287160158157f, 0.010986167937517166f, -0.01949607953429222f, 0.01757182367146015f, 0.02284356951713562f, -0.02871754951775074f, 0.0f, 0.02810060791671276f, -0.027684813365340233f, 0.0320032499730587f, 0.0f, 0.03489620238542557f, 0.0f, 0.01840006746351719f, -0.019603990018367767f, 0.017513001337647438f, 0.03161895275115967f, -0.027257494628429413f, 0.0230270866304636f, 0.03507275506854057f, -0.027039334177970886f, 0.037584662437438965f, -0.026764800772070885f, 0.03955071419477463f, 0.04115457087755203f, 0.003991170320659876f, -0.008905881084501743f, 0.013295728713274002f, 0.008854268118739128f, -0.01567106880247593f, 0.0f, 0.011620881967246532f, -0.018364345654845238f, 0.01412056665867567f, 0.0f, 0.016427477821707726f, 0.0f};
static __constant__ float kLpTrig6[44] = {1.0f, 0.9807852506637573f, 0.19509032368659973f, 0.9238795042037964f, 0.3826834261417389f, 0.8314695954322815f, 0.5555702447891235f, 0.7071067690849304f, 0.7071067690849304f, 0.5555702447891235f, 0.8314695954322815f, 1.0f, 0.8314695954322815f, 0.5555702447891235f, 0.3826834261417389f, 0.9238795042037964f, -0.19509032368659973f, 0.9807852506637573f, -0.7071067690849304f, 0.7071067690849304f, -0.9807852506637573f, 0.19509032368659973f, 1.0f, 0.5555702447891235f, 0.8314695954322815f, -0.3826834261417389f, 0.9238795042037964f, -0.9807852506637573f, 0.19509032368659973f, -0.7071067690849304f, -0.7071067690849304f, 0.19509032368659973f, -0.9807852506637573f, 1.0f, 0.19509032368659973f, 0.9807852506637573f, -0.9238795042037964f, 0.3826834261417389f, -0.5555702447891235f, -0.8314695954322815f, 0.7071067690849304f, -0.7071067690849304f, 0.8314695954322815f, 0.5555702447891235f};
#endif
template <> struct SH<6> {
    static constexpr int K = 36;
    static constexpr int NNZ_SYM = 1517;   // entries (i, j <= k)
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            case 9: return 0.03933623805642128f;
            case 10: return 0.09635371714830399f;
            case 11: return 0.304697185754776f;
            case 12: return 0.7463526725769043f;
            case 13: return 0.304697185754776f;
            case 14: return 0.09635371714830399f;
            case 15: return 0.03933623805642128f;
            case 16: return 0.005960340145975351f;
            case 17: return 0.016858387738466263f;
            case 18: return 0.06307831406593323f;
            case 19: return 0.2676186263561249f;
            case 20: return 0.8462843894958496f;
            case 21: return 0.2676186263561249f;
            case 22: return 0.06307831406593323f;
            case 23: return 0.016858387738466263f;
            case 24: return 0.005960340145975351f;
            case 25: return 0.0006945841596461833f;
            case 26: return 0.002196467947214842f;
            case 27: return 0.009318824857473373f;
            case 28: return 0.045652732253074646f;
            case 29: return 0.2415715456008911f;
            case 30: return 0.935602605342865f;
            case 31: return 0.2415715456008911f;
            case 32: return 0.045652732253074646f;
            case 33: return 0.009318824857473373f;
            case 34: return 0.002196467947214842f;
            case 35: return 0.0006945841596461833f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            case 3: return 0.0f;
            case 4: return -0.13089969754219055f;
            case 5: return 0.0f;
            default: return 0.0f;
        }
    }
    static constexpr int LPS = 4;   // lane-pair product rule: node pairs
    static constexpr int LPQ = 4;   // ... and azimuth quads
    static constexpr int LES = 6;   // lane-pair projected-exponential rule: node pairs
    static constexpr int LEQ = 6;   // ... and azimuth quads
#if defined(SHS_NB) && SHS_NB == 6
    __device__ __forceinline__ static const float* lp_leg() { return kLpLeg6; }
    __device__ __forceinline__ static const float* le_leg() { return kLeLeg6; }
    __device__ __forceinline__ static const float* lp_trig_row(int b) { return kLpTrig6 + b * 11; }
#endif
    __device__ __forceinline__ static float lp_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 11 + h) {
            case 1: return 0.9807852506637573f;
            case 2: return 0.19509032368659973f;
            case 3: return 0.9238795042037964f;
            case 4: return 0.3826834261417389f;
            case 5: return 0.8314695954322815f;
            case 6: return 0.5555702447891235f;
            case 7: return 0.7071067690849304f;
            case 8: return 0.7071067690849304f;
            case 9: return 0.5555702447891235f;
            case 10: return 0.8314695954322815f;
            case 12: return 0.8314695954322815f;
            case 13: return 0.5555702447891235f;
            case 14: return 0.3826834261417389f;
            case 15: return 0.9238795042037964f;
            case 16: return -0.19509032368659973f;
            case 17: return 0.9807852506637573f;
            case 18: return -0.7071067690849304f;
            case 19: return 0.7071067690849304f;
            case 20: return -0.9807852506637573f;
            case 21: return 0.19509032368659973f;
            case 23: return 0.5555702447891235f;
            case 24: return 0.8314695954322815f;
            case 25: return -0.3826834261417389f;
            case 26: return 0.9238795042037964f;
            case 27: return -0.9807852506637573f;
            case 28: return 0.19509032368659973f;
            case 29: return -0.7071067690849304f;
            case 30: return -0.7071067690849304f;
            case 31: return 0.19509032368659973f;
            case 32: return -0.9807852506637573f;
            case 34: return 0.19509032368659973f;
            case 35: return 0.9807852506637573f;
            case 36: return -0.9238795042037964f;
            case 37: return 0.3826834261417389f;
            case 38: return -0.5555702447891235f;
            case 39: return -0.8314695954322815f;
            case 40: return 0.7071067690849304f;
            case 41: return -0.7071067690849304f;
            case 42: return 0.8314695954322815f;
            case 43: return 0.5555702447891235f;
            default: return 1.0f;
        }
    }
    __device__ __forceinline__ static float le_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 11 + h) {
            case 1: return 0.9914448857307434f;
            case 2: return 0.13052618503570557f;
            case 3: return 0.9659258127212524f;
            case 4: return 0.258819043636322f;
            case 5: return 0.9238795042037964f;
            case 6: return 0.3826834261417389f;
            case 7: return 0.8660253882408142f;
            case 8: return 0.5f;
            case 9: return 0.7933533191680908f;
            case 10: return 0.6087614297866821f;
            case 12: return 0.9238795042037964f;
            case 13: return 0.3826834261417389f;
            case 14: return 0.7071067690849304f;
            case 15: return 0.7071067690849304f;
            case 16: return 0.3826834261417389f;
            case 17: return 0.9238795042037964f;
            case 18: return 6.123234262925839e-17f;
            case 19: return 1.0f;
            case 20: return -0.3826834261417389f;
            case 21: return 0.9238795042037964f;
            case 23: return 0.7933533191680908f;
            case 24: return 0.6087614297866821f;
            case 25: return 0.258819043636322f;
            case 26: return 0.9659258127212524f;
            case 27: return -0.3826834261417389f;
            case 28: return 0.9238795042037964f;
            case 29: return -0.8660253882408142f;
            case 30: return 0.5f;
            case 31: return -0.9914448857307434f;
            case 32: return -0.13052618503570557f;
            case 34: return 0.6087614297866821f;
            case 35: return 0.7933533191680908f;
            case 36: return -0.258819043636322f;
            case 37: return 0.9659258127212524f;
            case 38: return -0.9238795042037964f;
            case 39: return 0.3826834261417389f;
            case 40: return -0.8660253882408142f;
            case 41: return -0.5f;
            case 42: return -0.13052618503570557f;
            case 43: return -0.9914448857307434f;
            case 45: return 0.3826834261417389f;
            case 46: return 0.9238795042037964f;
            case 47: return -0.7071067690849304f;
            case 48: return 0.7071067690849304f;
            case 49: return -0.9238795042037964f;
            case 50: return -0.3826834261417389f;
            case 51: return -1.8369701465288538e-16f;
            case 52: return -1.0f;
            case 53: return 0.9238795042037964f;
            case 54: return -0.3826834261417389f;
            case 56: return 0.13052618503570557f;
            case 57: return 0.9914448857307434f;
            case 58: return -0.9659258127212524f;
            case 59: return 0.258819043636322f;
            case 60: return -0.3826834261417389f;
            case 61: return -0.9238795042037964f;
            case 62: return 0.8660253882408142f;
            case 63: return -0.5f;
            case 64: return 0.6087614297866821f;
            case 65: return 0.7933533191680908f;
            default: return 1.0f;
        }
    }
};

#if defined(SHS_NB) && SHS_NB == 7
// lane-pair rules: product, then projected exponential (plain, weighted)
static __device__ const float kLpLeg7[160] = {0.07776033133268356f, 0.1604437679052353f, 0.17591159045696259f, 0.14576031267642975f, 0.030566656962037086f, 0.10700652748346329f, 0.18740160763263702f, 0.007755899336189032f, 0.03787914291024208f, 0.08903763443231583f, 0.0019012305419892073f, 0.011880581267178059f, 0.0004576571809593588f, 0.003480701008811593f, 0.00010893459693761542f, 2.5732151698321104e-05f, 0.13117045164108276f, 0.17456598579883575f, 0.1658613383769989f, 0.0f, 0.06656565517187119f, 0.14835511147975922f, 0.22126656770706177f, 0.019984738901257515f, 0.06116100028157234f, 0.0f, 0.0055548627860844135f, 0.02148888260126114f, 0.0014782703947275877f, 0.0f, 0.0003825205785688013f, 0.0f, 0.10176809132099152f, 0.1416567713022232f, 0.0057292720302939415f, -0.13807961344718933f, 0.08842682093381882f, 0.22677944600582123f, 0.1871802657842636f, 0.04959646612405777f, 0.18204443156719208f, 0.2513335645198822f, 0.026874219998717308f, 0.1277928352355957f, 0.014299598522484303f, 0.08337191492319107f, 0.0075237080454826355f, 0.003928481601178646f, 0.15248256921768188f, 0.08637560904026031f, -0.07675936818122864f, 0.0f, 0.17104756832122803f, 0.23445476591587067f, 0.09396131336688995f, 0.11351354420185089f, 0.23436066508293152f, 0.0f, 0.06974370777606964f, 0.18988792598247528f, 0.04102684557437897f, 0.0f, 0.023466672748327255f, 0.0f, 0.11560682207345963f, 0.049735285341739655f, -0.1469823718070984f, -0.024236643686890602f, 0.1469256728887558f, 0.17976497113704681f, -0.13454866409301758f, 0.12053308635950089f, 0.23290126025676727f, -0.028189362958073616f, 0.09552856534719467f, 0.24985216557979584f, 0.07434694468975067f, 0.24441133439540863f, 0.05721541494131088f, 0.043696604669094086f, 0.13604286313056946f, -0.07190325111150742f, -0.12661293148994446f, 0.0f, 0.22321036458015442f, 0.03159971162676811f, -0.21622465550899506f, 0.21666410565376282f, 0.1382545530796051f, 0.0f, 0.19470907747745514f, 0.21051988005638123f, 0.16752943396568298f, 0.0f, 0.1401575207710266f, 0.0f, 0.12383381277322769f, -0.060434337705373764f, -0.06501844525337219f, 0.1434260606765747f, 0.19329603016376495f, -0.011000985279679298f, -0.15925481915473938f, 0.1947605460882187f, 0.0531000941991806f, -0.19980302453041077f, 0.18958215415477753f, 0.10853941738605499f, 0.18121609091758728f, 0.15576526522636414f, 0.17128373682498932f, 0.1606646180152893f, 0.09295744448900223f, -0.14631447196006775f, 0.09065702557563782f, 0.0f, 0.18732348084449768f, -0.19330981373786926f, 0.05287531390786171f, 0.22332343459129333f, -0.16165538132190704f, 0.0f, 0.24649208784103394f, -0.11979328095912933f, 0.2604818046092987f, 0.0f, 0.2676529884338379f, 0.0f, 0.12773483991622925f, -0.13331623375415802f, 0.11267582327127457f, -0.0813179761171341f, 0.21877773106098175f, -0.18196919560432434f, 0.14197389781475067f, 0.24187514185905457f, -0.17697179317474365f, 0.12588657438755035f, 0.2583436071872711f, -0.17147885262966156f, 0.270961195230484f, -0.1651965230703354f, 0.28101956844329834f, 0.2892349064350128f, 0.032937441021203995f, -0.07268138229846954f, 0.10626965761184692f, 0.0f, 0.07282960414886475f, -0.12687724828720093f, 0.16899468004703522f, 0.09527086466550827f, -0.14748406410217285f, 0.0f, 0.11538220942020416f, -0.16550104320049286f, 0.13378988206386566f, 0.0f, 0.150844007730484f, 0.0f};
static __device__ const float kLeLeg7[448] = {0.282094806432724f, 0.6050053238868713f, 0.7337506413459778f, 0.7436875104904175f, 0.08064790815114975f, 0.2914804220199585f, 0.5422344207763672f, 0.014882830902934074f, 0.07487541437149048f, 0.18467740714550018f, 0.00265336106531322f, 0.017060957849025726f, 0.000464526005089283f, 0.003632891923189163f, 8.041624823817983e-05f, 1.3815361853630748e-05f, 0.48190075159072876f, 0.6859782338142395f, 0.7521823048591614f, 0.0f, 0.17786070704460144f, 0.4148964583873749f, 0.6680772304534912f, 0.03883617743849754f, 0.12354122847318649f, 0.0f, 0.00785090122371912f, 0.03146146610379219f, 0.0015195264713838696f, 0.0f, 0.0002859679516404867f, 0.0f, 0.282094806432724f, 0.5002028346061707f, 0.33283063769340515f, -0.037704091519117355f, 0.1815134733915329f, 0.5619985461235046f, 0.7632161974906921f, 0.07539057731628418f, 0.32866668701171875f, 0.6359331011772156f, 0.03025127202272415f, 0.169509157538414f, 0.01191991288214922f, 0.08151230216026306f, 0.004644325003027916f, 0.0017957952804863453f, 0.4536356031894684f, 0.4538605809211731f, 0.15976978838443756f, 0.0f, 0.3768298625946045f, 0.700112521648407f, 0.7355261445045471f, 0.18519000709056854f, 0.4870571792125702f, 0.0f, 0.08425901085138321f, 0.2842300832271576f, 0.03670463338494301f, 0.0f, 0.015546969138085842f, 0.0f, 0.282094806432724f, 0.33203983306884766f, -0.1206328421831131f, -0.4215880334377289f, 0.2745485305786133f, 0.6218326687812805f, 0.31886351108551025f, 0.1724795252084732f, 0.5660937428474426f, 0.6012592911720276f, 0.1046825647354126f, 0.4477361738681793f, 0.062389861792325974f, 0.3283042311668396f, 0.03676832094788551f, 0.021503949537873268f, 0.4041726291179657f, 0.1300550252199173f, -0.32900097966194153f, 0.0f, 0.5078264474868774f, 0.5566006898880005f, -0.020793095231056213f, 0.3774833381175995f, 0.6590285897254944f, 0.0f, 0.2597806453704834f, 0.6120079755783081f, 0.17116761207580566f, 0.0f, 0.10966213047504425f, 0.0f, 0.282094806432724f, 0.13155442476272583f, -0.35559025406837463f, -0.08521328866481781f, 0.35491126775741577f, 0.45212191343307495f, -0.3051152229309082f, 0.2882298231124878f, 0.5757606625556946f, -0.03383835777640343f, 0.22613950073719025f, 0.6096431016921997f, 0.1742275357246399f, 0.5894106030464172f, 0.13273249566555023f, 0.10035116225481033f, 0.335813045501709f, -0.16367165744304657f, -0.32220059633255005f, 0.0f, 0.545439600944519f, 0.10240838676691055f, -0.5257964134216309f, 0.5241189002990723f, 0.36253634095191956f, 0.0f, 0.4662722051143646f, 0.5328931212425232f, 0.3971503973007202f, 0.0f, 0.3289203643798828f, 0.0f, 0.282094806432724f, -0.0642000138759613f, -0.2642127573490143f, 0.3176251947879791f, 0.4187522530555725f, 0.12824709713459015f, -0.4800601899623871f, 0.4012486934661865f, 0.2982756793498993f, -0.4915175139904022f, 0.3714398741722107f, 0.42788830399513245f, 0.3376496136188507f, 0.5227455496788025f, 0.30350375175476074f, 0.27073636651039124f, 0.25175178050994873f, -0.32160407304763794f, 0.0516158863902092f, 0.0f, 0.4824574589729309f, -0.33728790283203125f, -0.16429507732391357f, 0.546990156173706f, -0.18464216589927673f, 0.0f, 0.5741516351699829f, -0.023816371336579323f, 0.5770047903060913f, 0.0f, 0.5638357400894165f, 0.0f, 0.282094806432724f, -0.21904003620147705f, 0.03257828578352928f, 0.16972026228904724f, 0.46305686235427856f, -0.21260583400726318f, -0.0892399251461029f, 0.4906456470489502f, -0.12202231585979462f, -0.2030356377363205f, 0.5022500157356262f, -0.03477540984749794f, 0.504864513874054f, 0.04890919476747513f, 0.5018221139907837f, 0.4950048625469208f, 0.15591910481452942f, -0.296621710062027f, 0.31815603375434875f, 0.0f, 0.3304174244403839f, -0.4627828299999237f, 0.4030117094516754f, 0.41424816846847534f, -0.477090060710907f, 0.0f, 0.4808225631713867f, -0.47038865089416504f, 0.5343364477157593f, 0.0f, 0.5773844718933105f, 0.0f, 0.282094806432724f, -0.30434414744377136f, 0.280807226896286f, -0.24261875450611115f, 0.4857417047023773f, -0.42784395813941956f, 0.377977579832077f, 0.5398960113525391f, -0.4293491542339325f, 0.36160001158714294f, 0.5797399282455444f, -0.4301821291446686f, 0.6113067269325256f, -0.4295520782470703f, 0.6373898983001709f, 0.6595321297645569f, 0.05279592052102089f, -0.11861658841371536f, 0.1793360412120819f, 0.0f, 0.11736404150724411f, -0.20973744988441467f, 0.29129156470298767f, 0.15434898436069489f, -0.24699321389198303f, 0.0f, 0.18793129920959473f, -0.28084641695022583f, 0.21907870471477509f, 0.0f, 0.24832561612129211f, 0.0f, 0.0022231293842196465f, 0.004767918959259987f, 0.005782533437013626f, 0.005860844161361456f, 0.0006355691002681851f, 0.002297095488756895f, 0.0042732348665595055f, 0.00011728843674063683f, 0.0005900773103348911f, 0.001455403515137732f, 2.091057649522554e-05f, 0.00013445380318444222f, 3.6608312257158104e-06f, 2.8630052838707343e-05f, 6.33743411526666e-07f, 1.0887594470432305e-07f, 0.0037977579049766064f, 0.00540604954585433f, 0.005927789490669966f, 0.0f, 0.0014016826171427965f, 0.0032697112765163183f, 0.005264975130558014f, 0.00030605969368480146f, 0.0009736022911965847f, 0.0f, 6.187129474710673e-05f, 0.00024794114870019257f, 1.1975066627201159e-05f, 0.0f, 2.2536530650540954e-06f, 0.0f, 0.005074161104857922f, 0.008997364901006222f, 0.005986768752336502f, -0.0006781998090445995f, 0.0032649615313857794f, 0.01010891143232584f, 0.013728300109505653f, 0.0013560829684138298f, 0.005911869928240776f, 0.011438804678618908f, 0.0005441427347250283f, 0.0030490346252918243f, 0.00021440863201860338f, 0.0014661969617009163f, 8.353948214789852e-05f, 3.230174843338318e-05f, 0.008159739896655083f, 0.008163786493241787f, 0.0028738481923937798f, 0.0f, 0.006778202019631863f, 0.012593227438628674f, 0.013230226933956146f, 0.0033310926519334316f, 0.0087609076872468f, 0.0f, 0.001515603275038302f, 0.005112569313496351f, 0.0006602220819331706f, 0.0f, 0.0002796500630211085f, 0.0f, 0.007692359387874603f, 0.009054295718669891f, -0.0032895011827349663f, -0.011496159248054028f, 0.007486582268029451f, 0.016956571489572525f, 0.008694995194673538f, 0.004703293088823557f, 0.015436642803251743f, 0.016395561397075653f, 0.0028545577079057693f, 0.012209185399115086f, 0.0017012906027957797f, 0.008952430449426174f, 0.001002624398097396f, 0.0005863848491571844f, 0.011021263897418976f, 0.003546432126313448f, -0.008971430361270905f, 0.0f, 0.013847769238054752f, 0.015177778899669647f, -0.0005670007667504251f, 0.010293480940163136f, 0.0179708544164896f, 0.0f, 0.00708388164639473f, 0.016688663512468338f, 0.00466751866042614f, 0.0f, 0.002990344073623419f, 0.0f, 0.00995126273483038f, 0.0046407547779381275f, -0.01254391111433506f, -0.003006010316312313f, 0.0125199593603611f, 0.0159491915255785f, -0.010763337835669518f, 0.010167684406042099f, 0.02031070925295353f, -0.0011936923256143928f, 0.00797736644744873f, 0.02150595746934414f, 0.006146104075014591f, 0.02079222910106182f, 0.004682312253862619f, 0.0035400185734033585f, 0.01184624433517456f, -0.0057737319730222225f, -0.011366047896444798f, 0.0f, 0.0192410945892334f, 0.0036125897895544767f, -0.018548157066106796f, 0.01848897896707058f, 0.012788943946361542f, 0.0f, 0.016448361799120903f, 0.018798502162098885f, 0.014009999111294746f, 0.0f, 0.0116030965000391f, 0.0f, 0.011744937859475613f, -0.0026729495730251074f, -0.011000423692166805f, 0.013224235735833645f, 0.017434632405638695f, 0.005339531693607569f, -0.01998717151582241f, 0.01670587621629238f, 0.012418624013662338f, -0.02046419307589531f, 0.015464793890714645f, 0.017815008759498596f, 0.014057946391403675f, 0.0217643640935421f, 0.012636292725801468f, 0.01127203181385994f, 0.010481614619493484f, -0.013389894738793373f, 0.0021490128710865974f, 0.0f, 0.02008698135614395f, -0.014042886905372143f, -0.0068403794430196285f, 0.022773781791329384f, -0.007687524892389774f, 0.0f, 0.023904642090201378f, -0.0009915879927575588f, 0.024023432284593582f, 0.0f, 0.02347514219582081f, 0.0f, 0.012989457696676254f, -0.01008601114153862f, 0.0015001136343926191f, 0.007815011776983738f, 0.021322114393115044f, -0.009789738804101944f, -0.004109179601073265f, 0.02259247936308384f, -0.00561869191005826f, -0.009349065832793713f, 0.023126818239688873f, -0.0016012833220884204f, 0.023247206583619118f, 0.0022520937491208315f, 0.023107115179300308f, 0.022793205454945564f, 0.007179517764598131f, -0.013658370822668076f, 0.014649949036538601f, 0.0f, 0.015214542858302593f, -0.021309496834874153f, 0.018557248637080193f, 0.01907464861869812f, -0.0219682939350605f, 0.0f, 0.02214016206562519f, -0.021659716963768005f, 0.02460428513586521f, 0.0f, 0.026586493477225304f, 0.0f, 0.013626615516841412f, -0.01470137294381857f, 0.01356441993266344f, -0.011719722300767899f, 0.02346380054950714f, -0.020667042583227158f, 0.018258243799209595f, 0.026079727336764336f, -0.020739750936627388f, 0.01746712438762188f, 0.028004391118884087f, -0.020779989659786224f, 0.029529228806495667f, -0.02074955403804779f, 0.03078918159008026f, 0.03185876086354256f, 0.002550311852246523f, -0.005729785654693842f, 0.008662845008075237f, 0.0f, 0.005669281352311373f, -0.01013138797134161f, 0.01407086756080389f, 0.007455842569470406f, -0.011931031011044979f, 0.0f, 0.009078038856387138f, -0.01356631238013506f, 0.010582617484033108f, 0.0f, 0.011995392851531506f, 0.0f};
static __constant__ float kLpTrig7[65] = {1.0f, 0.9876883625984192f, 0.15643446147441864f, 0.9510565400123596f, 0.30901700258255005f, 0.8910065293312073f, 0.45399048924446106f, 0.80901700258255f, 0.5877852439880371f, 0.7071067690849304f, 0.7071067690849304f, 0.5877852439880371f, 0.80901700258255f, 1.0f, 0.8910065293312073f, 0.45399048924446106f, 0.5877852439880371f, 0.80901700258255f, 0.15643446147441864f, 0.9876883625984192f, -0.30901700258255005f, 0.9510565400123596f, -0.7071067690849304f, 0.7071067690849304f, -0.9510565400123596f, 0.30901700258255005f, 1.0f, 0.7071067690849304f, 0.7071067690849304f, 6.123234262925839e-17f, 1.0f, -0.7071067690849304f, 0.7071067690849304f, -1.0f, 1.2246468525851679e-16f, -0.7071067690849304f, -0.7071067690849304f, -1.8369701465288538e-16f, -1.0f, 1.0f, 0.45399048924446106f, 0.8910065293312073f, -0.5877852439880371f, 0.80901700258255f, -0.9876883625984192f, -0.15643446147441864f, -0.30901700258255005f, -0.9510565400123596f, 0.7071067690849304f, -0.7071067690849304f, 0.9510565400123596f, 0.30901700258255005f, 1.0f, 0.15643446147441864f, 0.9876883625984192f, -0.9510565400123596f, 0.30901700258255005f, -0.45399048924446106f, -0.8910065293312073f, 0.80901700258255f, -0.5877852439880371f, 0.7071067690849304f, 0.7071067690849304f, -0.5877852439880371f, 0.80901700258255f};
#endif
template <> struct SH<7> {
    static constexpr int K = 49;
    static constexpr int NNZ_SYM = 3348;   // entries (i, j <= k)
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            case 9: return 0.03933623805642128f;
            case 10: return 0.09635371714830399f;
            case 11: return 0.304697185754776f;
            case 12: return 0.7463526725769043f;
            case 13: return 0.304697185754776f;
            case 14: return 0.09635371714830399f;
            case 15: return 0.03933623805642128f;
            case 16: return 0.005960340145975351f;
            case 17: return 0.016858387738466263f;
            case 18: return 0.06307831406593323f;
            case 19: return 0.2676186263561249f;
            case 20: return 0.8462843894958496f;
            case 21: return 0.2676186263561249f;
            case 22: return 0.06307831406593323f;
            case 23: return 0.016858387738466263f;
            case 24: return 0.005960340145975351f;
            case 25: return 0.0006945841596461833f;
            case 26: return 0.002196467947214842f;
            case 27: return 0.009318824857473373f;
            case 28: return 0.045652732253074646f;
            case 29: return 0.2415715456008911f;
            case 30: return 0.935602605342865f;
            case 31: return 0.2415715456008911f;
            case 32: return 0.045652732253074646f;
            case 33: return 0.009318824857473373f;
            case 34: return 0.002196467947214842f;
            case 35: return 0.0006945841596461833f;
            case 36: return 6.572237907676026e-05f;
            case 37: return 0.00022766899201087654f;
            case 38: return 0.00106786226388067f;
            case 39: return 0.005848922301083803f;
            case 40: return 0.035093534737825394f;
            case 41: return 0.22195099294185638f;
            case 42: return 1.0171072483062744f;
            case 43: return 0.22195099294185638f;
            case 44: return 0.035093534737825394f;
            case 45: return 0.005848922301083803f;
            case 46: return 0.00106786226388067f;
            case 47: return 0.00022766899201087654f;
            case 48: return 6.572237907676026e-05f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            case 3: return 0.0f;
            case 4: return -0.13089969754219055f;
            case 5: return 0.0f;
            case 6: return 0.04908738657832146f;
            default: return 0.0f;
        }
    }
    static constexpr int LPS = 5;   // lane-pair product rule: node pairs
    static constexpr int LPQ = 5;   // ... and azimuth quads
    static constexpr int LES = 7;   // lane-pair projected-exponential rule: node pairs
    static constexpr int LEQ = 7;   // ... and azimuth quads
#if defined(SHS_NB) && SHS_NB == 7
    __device__ __forceinline__ static const float* lp_leg() { return kLpLeg7; }
    __device__ __forceinline__ static const float* le_leg() { return kLeLeg7; }
    __device__ __forceinline__ static const float* lp_trig_row(int b) { return kLpTrig7 + b * 13; }
#endif
    __device__ __forceinline__ static float lp_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 13 + h) {
            case 1: return 0.9876883625984192f;
            case 2: return 0.15643446147441864f;
            case 3: return 0.9510565400123596f;
            case 4: return 0.30901700258255005f;
            case 5: return 0.8910065293312073f;
            case 6: return 0.45399048924446106f;
            case 7: return 0.80901700258255f;
            case 8: return 0.5877852439880371f;
            case 9: return 0.7071067690849304f;
            case 10: return 0.7071067690849304f;
            case 11: return 0.5877852439880371f;
            case 12: return 0.80901700258255f;
            case 14: return 0.8910065293312073f;
            case 15: return 0.45399048924446106f;
            case 16: return 0.5877852439880371f;
            case 17: return 0.80901700258255f;
            case 18: return 0.15643446147441864f;
            case 19: return 0.9876883625984192f;
            case 20: return -0.30901700258255005f;
            case 21: return 0.9510565400123596f;
            case 22: return -0.7071067690849304f;
            case 23: return 0.7071067690849304f;
            case 24: return -0.9510565400123596f;
            case 25: return 0.30901700258255005f;
            case 27: return 0.7071067690849304f;
            case 28: return 0.7071067690849304f;
            case 29: return 6.123234262925839e-17f;
            case 30: return 1.0f;
            case 31: return -0.7071067690849304f;
            case 32: return 0.7071067690849304f;
            case 33: return -1.0f;
            case 34: return 1.2246468525851679e-16f;
            case 35: return -0.7071067690849304f;
            case 36: return -0.7071067690849304f;
            case 37: return -1.8369701465288538e-16f;
            case 38: return -1.0f;
            case 40: return 0.45399048924446106f;
            case 41: return 0.8910065293312073f;
            case 42: return -0.5877852439880371f;
            case 43: return 0.80901700258255f;
            case 44: return -0.9876883625984192f;
            case 45: return -0.15643446147441864f;
            case 46: return -0.30901700258255005f;
            case 47: return -0.9510565400123596f;
            case 48: return 0.7071067690849304f;
            case 49: return -0.7071067690849304f;
            case 50: return 0.9510565400123596f;
            case 51: return 0.30901700258255005f;
            case 53: return 0.15643446147441864f;
            case 54: return 0.9876883625984192f;
            case 55: return -0.9510565400123596f;
            case 56: return 0.30901700258255005f;
            case 57: return -0.45399048924446106f;
            case 58: return -0.8910065293312073f;
            case 59: return 0.80901700258255f;
            case 60: return -0.5877852439880371f;
            case 61: return 0.7071067690849304f;
            case 62: return 0.7071067690849304f;
            case 63: return -0.5877852439880371f;
            case 64: return 0.80901700258255f;
            default: return 1.0f;
        }
    }
    __device__ __forceinline__ static float le_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 13 + h) {
            case 1: return 0.9937121868133545f;
            case 2: return 0.11196447908878326f;
            case 3: return 0.9749279022216797f;
            case 4: return 0.22252093255519867f;
            case 5: return 0.9438833594322205f;
            case 6: return 0.33027905225753784f;
            case 7: return 0.9009688496589661f;
            case 8: return 0.4338837265968323f;
            case 9: return 0.8467242121696472f;
            case 10: return 0.5320320725440979f;
            case 11: return 0.7818315029144287f;
            case 12: return 0.6234897971153259f;
            case 14: return 0.9438833594322205f;
            case 15: return 0.33027905225753784f;
            case 16: return 0.7818315029144287f;
            case 17: return 0.6234897971153259f;
            case 18: return 0.5320320725440979f;
            case 19: return 0.8467242121696472f;
            case 20: return 0.22252093255519867f;
            case 21: return 0.9749279022216797f;
            case 22: return -0.11196447908878326f;
            case 23: return 0.9937121868133545f;
            case 24: return -0.4338837265968323f;
            case 25: return 0.9009688496589661f;
            case 27: return 0.8467242121696472f;
            case 28: return 0.5320320725440979f;
            case 29: return 0.4338837265968323f;
            case 30: return 0.9009688496589661f;
            case 31: return -0.11196447908878326f;
            case 32: return 0.9937121868133545f;
            case 33: return -0.6234897971153259f;
            case 34: return 0.7818315029144287f;
            case 35: return -0.9438833594322205f;
            case 36: return 0.33027905225753784f;
            case 37: return -0.9749279022216797f;
            case 38: return -0.22252093255519867f;
            case 40: return 0.7071067690849304f;
            case 41: return 0.7071067690849304f;
            case 42: return 6.123234262925839e-17f;
            case 43: return 1.0f;
            case 44: return -0.7071067690849304f;
            case 45: return 0.7071067690849304f;
            case 46: return -1.0f;
            case 47: return 1.2246468525851679e-16f;
            case 48: return -0.7071067690849304f;
            case 49: return -0.7071067690849304f;
            case 50: return -1.8369701465288538e-16f;
            case 51: return -1.0f;
            case 53: return 0.5320320725440979f;
            case 54: return 0.8467242121696472f;
            case 55: return -0.4338837265968323f;
            case 56: return 0.9009688496589661f;
            case 57: return -0.9937121868133545f;
            case 58: return 0.11196447908878326f;
            case 59: return -0.6234897971153259f;
            case 60: return -0.7818315029144287f;
            case 61: return 0.33027905225753784f;
            case 62: return -0.9438833594322205f;
            case 63: return 0.9749279022216797f;
            case 64: return -0.22252093255519867f;
            case 66: return 0.33027905225753784f;
            case 67: return 0.9438833594322205f;
            case 68: return -0.7818315029144287f;
            case 69: return 0.6234897971153259f;
            case 70: return -0.8467242121696472f;
            case 71: return -0.5320320725440979f;
            case 72: return 0.22252093255519867f;
            case 73: return -0.9749279022216797f;
            case 74: return 0.9937121868133545f;
            case 75: return -0.11196447908878326f;
            case 76: return 0.4338837265968323f;
            case 77: return 0.9009688496589661f;
            case 79: return 0.11196447908878326f;
            case 80: return 0.9937121868133545f;
            case 81: return -0.9749279022216797f;
            case 82: return 0.22252093255519867f;
            case 83: return -0.33027905225753784f;
            case 84: return -0.9438833594322205f;
            case 85: return 0.9009688496589661f;
            case 86: return -0.4338837265968323f;
            case 87: return 0.5320320725440979f;
            case 88: return 0.8467242121696472f;
            case 89: return -0.7818315029144287f;
            case 90: return 0.6234897971153259f;
            default: return 1.0f;
        }
    }
};

#if defined(SHS_NB) && SHS_NB == 8
// lane-pair rules: product, then projected exponential (plain, weighted)
static __device__ const float kLpLeg8[240] = {0.06520631164312363f, 0.13781440258026123f, 0.16102319955825806f, 0.15215513110160828f, 0.021588720381259918f, 0.07708820700645447f, 0.14019207656383514f, 0.19657686352729797f, 0.00461379811167717f, 0.022952022030949593f, 0.05559203401207924f, 0.0009525957866571844f, 0.006059064529836178f, 0.01822534203529358f, 0.00019313527445774525f, 0.0014945222064852715f, 3.87199324904941e-05f, 0.0003527893277350813f, 7.703575647610705e-06f, 1.5242303561535664e-06f, 0.11085808277130127f, 0.15386998653411865f, 0.16021457314491272f, 0.13757289946079254f, 0.04738370701670647f, 0.10864433646202087f, 0.1700213998556137f, 0.0f, 0.011981873773038387f, 0.03756134212017059f, 0.07660231739282608f, 0.0028050916735082865f, 0.011091789230704308f, 0.0f, 0.0006287457654252648f, 0.0029944006819278f, 0.0001370324462186545f, 0.0f, 2.9285665732459165e-05f, 0.0f, 0.08565717935562134f, 0.13908180594444275f, 0.05986662954092026f, -0.06713762134313583f, 0.0633930191397667f, 0.18306352198123932f, 0.21085374057292938f, 0.10451316833496094f, 0.03028402104973793f, 0.1238425225019455f, 0.21286974847316742f, 0.013976679183542728f, 0.07366860657930374f, 0.16529589891433716f, 0.00633428106084466f, 0.04081254079937935f, 0.0028386428020894527f, 0.021603398025035858f, 0.0012624345254153013f, 0.0005583513411693275f, 0.13413716852664948f, 0.11137636750936508f, -0.003983851056545973f, -0.11710293591022491f, 0.12815962731838226f, 0.21362611651420593f, 0.17273001372814178f, 0.0f, 0.0724414810538292f, 0.17446376383304596f, 0.22883576154708862f, 0.037909671664237976f, 0.11820931732654572f, 0.0f, 0.018994087353348732f, 0.07242981344461441f, 0.009253524243831635f, 0.0f, 0.004420579876750708f, 0.0f, 0.09798557311296463f, 0.08525826036930084f, -0.09131614118814468f, -0.11765225976705551f, 0.10830617696046829f, 0.19894984364509583f, 0.008022683672606945f, -0.19128155708312988f, 0.07727494835853577f, 0.2107543796300888f, 0.1254342496395111f, 0.053265079855918884f, 0.19144459068775177f, 0.19945865869522095f, 0.03605365753173828f, 0.16045929491519928f, 0.0241310466080904f, 0.12792740762233734f, 0.016028307378292084f, 0.010587655007839203f, 0.13066479563713074f, -0.003617573296651244f, -0.13627637922763824f, -0.04429611191153526f, 0.18645501136779785f, 0.13122136890888214f, -0.11810997873544693f, 0.0f, 0.15740682184696198f, 0.20314645767211914f, 0.0009861834114417434f, 0.1230267807841301f, 0.2253846824169159f, 0.0f, 0.09206223487854004f, 0.21661099791526794f, 0.06698594242334366f, 0.0f, 0.04779353365302086f, 0.0f, 0.10608874261379242f, 0.00413087522611022f, -0.1266615241765976f, 0.07696889340877533f, 0.14872010052204132f, 0.10081823915243149f, -0.18343278765678406f, 0.007615973707288504f, 0.1345750093460083f, 0.1648647040128708f, -0.14551927149295807f, 0.11764611303806305f, 0.20528586208820343f, -0.08582877367734909f, 0.10099354386329651f, 0.22752733528614044f, 0.08572938293218613f, 0.23614519834518433f, 0.07221883535385132f, 0.060502298176288605f, 0.1079203188419342f, -0.10511626303195953f, -0.04261922463774681f, 0.13283823430538177f, 0.1953115612268448f, -0.07001624256372452f, -0.14808103442192078f, 0.0f, 0.20911574363708496f, 0.012077328749001026f, -0.18980476260185242f, 0.2072870284318924f, 0.08569271862506866f, 0.0f, 0.19672666490077972f, 0.1459958702325821f, 0.18154096603393555f, 0.0f, 0.1642742156982422f, 0.0f, 0.11112427711486816f, -0.07381140440702438f, -0.01743069291114807f, 0.10047222673892975f, 0.1789790838956833f, -0.054160233587026596f, -0.08458041399717331f, 0.17426559329032898f, 0.1860758513212204f, -0.008524632081389427f, -0.13042566180229187f, 0.18689434230327606f, 0.033735811710357666f, -0.16413705050945282f, 0.18433387577533722f, 0.07256858795881271f, 0.17977702617645264f, 0.10785961151123047f, 0.17399948835372925f, 0.1674797534942627f, 0.07079759240150452f, -0.12563757598400116f, 0.11323718726634979f, -0.039617281407117844f, 0.14720962941646576f, -0.18506301939487457f, 0.12129383534193039f, 0.0f, 0.18108728528022766f, -0.17840780317783356f, 0.07581662386655807f, 0.20623688399791718f, -0.1622493416070938f, 0.0f, 0.22487977147102356f, -0.139549121260643f, 0.23842665553092957f, 0.0f, 0.24788059294223785f, 0.0f, 0.11355419456958771f, -0.12098407745361328f, 0.10807975381612778f, -0.08776627480983734f, 0.19513322412967682f, -0.16821692883968353f, 0.14210937917232513f, -0.10832967609167099f, 0.21644802391529083f, -0.16687056422233582f, 0.13246333599090576f, 0.23195002973079681f, -0.16517631709575653f, 0.12301430851221085f, 0.24408331513404846f, -0.1628371924161911f, 0.253981351852417f, -0.15985198318958282f, 0.2622710168361664f, 0.26933905482292175f, 0.024631112813949585f, -0.054961759597063065f, 0.0820532739162445f, -0.1040557399392128f, 0.054643236100673676f, -0.09671244770288467f, 0.13222384452819824f, 0.0f, 0.07171712070703506f, -0.11333373934030533f, 0.14613576233386993f, 0.087143674492836f, -0.12822918593883514f, 0.0f, 0.10138054937124252f, -0.14173586666584015f, 0.11468159407377243f, 0.0f, 0.12720850110054016f, 0.0f};
static __device__ const float kLeLeg8[640] = {0.282094806432724f, 0.6108322739601135f, 0.7587076425552368f, 0.8024648427963257f, 0.07094971090555191f, 0.2584724724292755f, 0.48795923590660095f, 0.7245708703994751f, 0.011518623679876328f, 0.05838014557957649f, 0.14570735394954681f, 0.0018066286575049162f, 0.011699545197188854f, 0.0361325666308403f, 0.00027825316647067666f, 0.0021913156379014254f, 4.237711618770845e-05f, 0.000392841175198555f, 6.4048267631733324e-06f, 9.626843393562012e-07f, 0.48342376947402954f, 0.6995154619216919f, 0.7922953963279724f, 0.7908328771591187f, 0.15696685016155243f, 0.3703010082244873f, 0.6073318123817444f, 0.0f, 0.030152400955557823f, 0.09684120118618011f, 0.204736590385437f, 0.00536244036629796f, 0.02167833410203457f, 0.0f, 0.0009130798862315714f, 0.004440254531800747f, 0.00015117340080905706f, 0.0f, 2.454286914144177e-05f, 0.0f, 0.282094806432724f, 0.5288062691688538f, 0.4332386255264282f, 0.12681901454925537f, 0.16040606796741486f, 0.5193262100219727f, 0.7771311402320862f, 0.774089515209198f, 0.05887635797262192f, 0.26746249198913574f, 0.5564955472946167f, 0.020877545699477196f, 0.12169450521469116f, 0.32081058621406555f, 0.007269772235304117f, 0.051662128418684006f, 0.002503123367205262f, 0.020974058657884598f, 0.0008553196093998849f, 0.000290653231786564f, 0.461521714925766f, 0.5150310397148132f, 0.29784974455833435f, -0.05915773659944534f, 0.3387991189956665f, 0.6733590960502625f, 0.8136188983917236f, 0.0f, 0.14713852107524872f, 0.4091092348098755f, 0.691368579864502f, 0.0591612234711647f, 0.20980627834796906f, 0.0f, 0.022774748504161835f, 0.09791873395442963f, 0.008524921722710133f, 0.0f, 0.0031290357001125813f, 0.0f, 0.282094806432724f, 0.39359357953071594f, 0.018211757764220238f, -0.38138410449028015f, 0.24463455379009247f, 0.6285143494606018f, 0.5217272043228149f, -0.0579991415143013f, 0.13694144785404205f, 0.5034611225128174f, 0.6975259780883789f, 0.07405773550271988f, 0.3527039885520935f, 0.6644591093063354f, 0.03932863101363182f, 0.22964313626289368f, 0.020652245730161667f, 0.1427166610956192f, 0.010762432590126991f, 0.005577687174081802f, 0.42294958233833313f, 0.24117226898670197f, -0.21048904955387115f, -0.44790521264076233f, 0.47351714968681335f, 0.6510443687438965f, 0.26493629813194275f, 0.0f, 0.3136294484138489f, 0.6490544676780701f, 0.6177658438682556f, 0.1923200637102127f, 0.524702787399292f, 0.0f, 0.11291147023439407f, 0.3805752098560333f, 0.06445726007223129f, 0.0f, 0.036081865429878235f, 0.0f, 0.282094806432724f, 0.22452960908412933f, -0.2879684865474701f, -0.3008277714252472f, 0.3201611340045929f, 0.5549961924552917f, -0.044748563319444656f, -0.5584453344345093f, 0.2345505803823471f, 0.6082530617713928f, 0.29154467582702637f, 0.16600562632083893f, 0.5692598223686218f, 0.5239323973655701f, 0.11537507176399231f, 0.4908573031425476f, 0.07929050922393799f, 0.402326762676239f, 0.05407732352614403f, 0.03667834401130676f, 0.36909249424934387f, -0.04138867184519768f, -0.3913777768611908f, -0.06159166991710663f, 0.5407955646514893f, 0.32933056354522705f, -0.39608559012413025f, 0.0f, 0.4687756597995758f, 0.5534201264381409f, -0.08651652932167053f, 0.37620416283607483f, 0.6415792107582092f, 0.0f, 0.2890598773956299f, 0.6385716795921326f, 0.2159595489501953f, 0.0f, 0.1582123339176178f, 0.0f, 0.282094806432724f, 0.04583054408431053f, -0.35458382964134216f, 0.12894819676876068f, 0.384176105260849f, 0.32660973072052f, -0.4573071599006653f, -0.12329808622598648f, 0.3377225399017334f, 0.48913657665252686f, -0.30245769023895264f, 0.28681913018226624f, 0.57930988073349f, -0.10303568840026855f, 0.23919881880283356f, 0.6170144081115723f, 0.1972559243440628f, 0.6180117130279541f, 0.16143056750297546f, 0.13138386607170105f, 0.3018958866596222f, -0.25159263610839844f, -0.1836709827184677f, 0.34278231859207153f, 0.5307828187942505f, -0.10648290067911148f, -0.4651665985584259f, 0.0f, 0.5520908832550049f, 0.13303987681865692f, -0.5200333595275879f, 0.5316561460494995f, 0.331875741481781f, 0.0f, 0.49018144607543945f, 0.4811188876628876f, 0.4394436776638031f, 0.0f, 0.3863072693347931f, 0.0f, 0.282094806432724f, -0.1169036328792572f, -0.18545503914356232f, 0.33673009276390076f, 0.43434005975723267f, 0.01986619643867016f, -0.40778017044067383f, 0.44140905141830444f, 0.4316771626472473f, 0.1751290261745453f, -0.4818282127380371f, 0.4144829213619232f, 0.30518484115600586f, -0.5003358721733093f, 0.390802264213562f, 0.4119834005832672f, 0.3643574118614197f, 0.4975000023841858f, 0.3371187150478363f, 0.31019774079322815f, 0.22378814220428467f, -0.3334845304489136f, 0.1654045134782791f, 0.14211028814315796f, 0.4448322653770447f, -0.4171973168849945f, 0.03768457472324371f, 0.0f, 0.5231057405471802f, -0.3215390741825104f, -0.14276351034641266f, 0.5695204138755798f, -0.20522691309452057f, 0.0f, 0.5936559438705444f, -0.08099491894245148f, 0.6017009019851685f, 0.0f, 0.5980119705200195f, 0.0f, 0.282094806432724f, -0.2403593808412552f, 0.0889744758605957f, 0.09286528080701828f, 0.4688291847705841f, -0.264663428068161f, 0.009497372433543205f, 0.24327048659324646f, 0.502954363822937f, -0.1937839388847351f, -0.09324891865253448f, 0.521267831325531f, -0.12374024838209152f, -0.18446695804595947f, 0.5305131077766418f, -0.05461635813117027f, 0.5338895320892334f, 0.013045242987573147f, 0.5332015156745911f, 0.5295804738998413f, 0.13759219646453857f, -0.27359575033187866f, 0.3242362141609192f, -0.27236804366111755f, 0.29521456360816956f, -0.44199138879776f, 0.4452876150608063f, 0.0f, 0.37472763657569885f, -0.4735797047615051f, 0.41168612241744995f, 0.44037261605262756f, -0.4876188635826111f, 0.0f, 0.4954850971698761f, -0.4878280460834503f, 0.5420773029327393f, 0.0f, 0.5815340280532837f, 0.0f, 0.282094806432724f, -0.3068500757217407f, 0.2890093922615051f, -0.2592114210128784f, 0.4863921105861664f, -0.43444186449050903f, 0.394683301448822f, -0.34362509846687317f, 0.5413427948951721f, -0.4391913115978241f, 0.38350313901901245f, 0.582071840763092f, -0.44341665506362915f, 0.37287411093711853f, 0.6145874261856079f, -0.4462928771972656f, 0.6416686773300171f, -0.44775089621543884f, 0.6648485660552979f, 0.6850703358650208f, 0.046423349529504776f, -0.10476886481046677f, 0.15971150994300842f, -0.2089904397726059f, 0.1033361628651619f, -0.1858418732881546f, 0.2607538104057312f, 0.0f, 0.1360824704170227f, -0.21955569088459015f, 0.2920544147491455f, 0.16591231524944305f, -0.2504565119743347f, 0.0f, 0.19366930425167084f, -0.27913984656333923f, 0.21981802582740784f, 0.0f, 0.24465221166610718f, 0.0f, 0.0015039525460451841f, 0.0032565747387707233f, 0.0040449537336826324f, 0.004278239328414202f, 0.0003782593703363091f, 0.001378013170324266f, 0.0026014926843345165f, 0.0038629574701189995f, 6.141007906990126e-05f, 0.00031124631641432643f, 0.0007768202922306955f, 9.631811735744122e-06f, 6.237463821889833e-05f, 0.00019263618742115796f, 1.4834713510936126e-06f, 1.1682720469252672e-05f, 2.2592820414502057e-07f, 2.094382807626971e-06f, 3.4146520278000025e-08f, 5.132429592435983e-09f, 0.002577312523499131f, 0.0037293776404112577f, 0.004224022384732962f, 0.0042162248864769936f, 0.000836848805192858f, 0.0019742127042263746f, 0.0032379121985286474f, 0.0f, 0.00016075369785539806f, 0.000516296538989991f, 0.0010915271705016494f, 2.8589169232873246e-05f, 0.00011557528341654688f, 0.0f, 4.867969437327702e-06f, 2.367265369684901e-05f, 8.059617471189995e-07f, 0.0f, 1.3084718375466764e-07f, 0.0f, 0.0034481717739254236f, 0.006463837809860706f, 0.005295671056956053f, 0.0015501659363508224f, 0.0019607157446444035f, 0.006347957998514175f, 0.009499224834144115f, 0.009462045505642891f, 0.0007196722435764968f, 0.0032693147659301758f, 0.00680229626595974f, 0.0002551956567913294f, 0.001487526809796691f, 0.003921412397176027f, 8.886170689947903e-05f, 0.000631489499937743f, 3.059680602746084e-05f, 0.0002563753805588931f, 1.0454957191541325e-05f, 3.552785528881941e-06f, 0.005641388241201639f, 0.006295457016676664f, 0.0036407518200576305f, -0.0007231116760522127f, 0.004141294397413731f, 0.008230771869421005f, 0.009945230558514595f, 0.0f, 0.001798540586605668f, 0.005000726785510778f, 0.00845090951770544f, 0.0007231542840600014f, 0.0025645566638559103f, 0.0f, 0.00027838602545671165f, 0.001196904806420207f, 0.00010420395847177133f, 0.0f, 3.8247613701969385e-05f, 0.0f, 0.005270752124488354f, 0.007354032248258591f, 0.0003402744769118726f, -0.0071259066462516785f, 0.004570832941681147f, 0.01174336951225996f, 0.009748122654855251f, -0.0010836750734597445f, 0.0025586592964828014f, 0.009406833909451962f, 0.013032806105911732f, 0.0013837191509082913f, 0.006590037606656551f, 0.012414973229169846f, 0.0007348291110247374f, 0.004290727898478508f, 0.00038587336894124746f, 0.0026665651239454746f, 0.00020108884200453758f, 0.00010421535262139514f, 0.007902529090642929f, 0.004506142344325781f, -0.003932847175747156f, -0.008368808776140213f, 0.008847351185977459f, 0.012164327315986156f, 0.00495015736669302f, 0.0f, 0.00585995614528656f, 0.012127147056162357f, 0.011542540974915028f, 0.003593371482565999f, 0.009803719818592072f, 0.0f, 0.0021096752025187016f, 0.0071107931435108185f, 0.0012043407186865807f, 0.0f, 0.0006741654360666871f, 0.0f, 0.006903097033500671f, 0.0054944283328950405f, -0.007046831306070089f, -0.0073615084402263165f, 0.007834612391889095f, 0.013581224717199802f, -0.0010950349969789386f, -0.013665626756846905f, 0.005739650223404169f, 0.01488446444272995f, 0.007134343963116407f, 0.004062297288328409f, 0.013930266723036766f, 0.012821067124605179f, 0.0028233251068741083f, 0.012011690996587276f, 0.0019403055775910616f, 0.00984527450054884f, 0.0013233176432549953f, 0.0008975499076768756f, 0.009032003581523895f, -0.0010128156282007694f, -0.009577343240380287f, -0.0015072000678628683f, 0.013233722187578678f, 0.008058995939791203f, -0.009692547842860222f, 0.0f, 0.011471334844827652f, 0.013542655855417252f, -0.002117132069543004f, 0.009206032380461693f, 0.01569998264312744f, 0.0f, 0.007073538843542337f, 0.015626385807991028f, 0.005284711718559265f, 0.0f, 0.003871588734909892f, 0.0f, 0.008285999298095703f, 0.0013461853377521038f, -0.01041522715240717f, 0.0037876085843890905f, 0.011284444481134415f, 0.009593541733920574f, -0.01343253068625927f, -0.0036216473672538996f, 0.009919959120452404f, 0.01436745934188366f, -0.008884121663868427f, 0.008424768224358559f, 0.017016129568219185f, -0.0030264779925346375f, 0.00702601158991456f, 0.018123628571629524f, 0.005794018507003784f, 0.01815292239189148f, 0.004741716664284468f, 0.003859151853248477f, 0.008867619559168816f, -0.007390057202428579f, -0.00539498683065176f, 0.010068580508232117f, 0.01559073943644762f, -0.0031277332454919815f, -0.013663386926054955f, 0.0f, 0.016216622665524483f, 0.0039077941328287125f, -0.015274993143975735f, 0.015616391785442829f, 0.009748220443725586f, 0.0f, 0.014398150146007538f, 0.014131954871118069f, 0.012907824479043484f, 0.0f, 0.011347043327987194f, 0.0f, 0.00936944130808115f, -0.0038828144315630198f, -0.006159667391330004f, 0.011184087023139f, 0.014426086097955704f, 0.0006598319741897285f, -0.0135439308360219f, 0.01466087345033884f, 0.014337641187012196f, 0.005816700868308544f, -0.01600334793329239f, 0.013766555115580559f, 0.010136350058019161f, -0.01661805808544159f, 0.012980030849575996f, 0.013683537021279335f, 0.012101695872843266f, 0.01652386784553528f, 0.01119699515402317f, 0.010302847251296043f, 0.007432855665683746f, -0.011076290160417557f, 0.005493713077157736f, 0.004720023367553949f, 0.014774571172893047f, -0.013856709934771061f, 0.0012516481801867485f, 0.0f, 0.017374331131577492f, -0.010679536499083042f, -0.0047417194582521915f, 0.018915940076112747f, -0.00681636668741703f, 0.0f, 0.019717572256922722f, -0.002690149238333106f, 0.0199847761541605f, 0.0f, 0.019862251356244087f, 0.0f, 0.010114253498613834f, -0.008617868646979332f, 0.0031900994945317507f, 0.0033296009059995413f, 0.01680944673717022f, -0.009489268064498901f, 0.0003405197348911315f, 0.008722243830561638f, 0.018032973632216454f, -0.006947948131710291f, -0.0033433556091040373f, 0.018689587712287903f, -0.004436594899743795f, -0.006613896228373051f, 0.019021067768335342f, -0.0019582202658057213f, 0.01914212666451931f, 0.0004677253891713917f, 0.019117459654808044f, 0.0189876276999712f, 0.0049332440830767155f, -0.009809528477489948f, 0.011625195853412151f, -0.009765510447323322f, 0.010584651492536068f, -0.015847202390432358f, 0.015965385362505913f, 0.0f, 0.01343552116304636f, -0.016979772597551346f, 0.014760633930563927f, 0.01578916236758232f, -0.01748313382267952f, 0.0f, 0.017765169963240623f, -0.017490632832050323f, 0.019435690715909004f, 0.0f, 0.020850377157330513f, 0.0f, 0.010493514128029346f, -0.01141437515616417f, 0.010750727728009224f, -0.009642287157475948f, 0.018093077465891838f, -0.01616060361266136f, 0.01468164287507534f, -0.012782352045178413f, 0.020137161016464233f, -0.016337275505065918f, 0.0142657570540905f, 0.0216522216796875f, -0.016494451090693474f, 0.01387037243694067f, 0.022861754521727562f, -0.01660144329071045f, 0.023869138211011887f, -0.016655679792165756f, 0.02473139576613903f, 0.025483615696430206f, 0.0017268809024244547f, -0.003897249000146985f, 0.005941035225987434f, -0.007774139288812876f, 0.003843954298645258f, -0.0069130463525652885f, 0.00969966035336256f, 0.0f, 0.0050620692782104015f, -0.008167151361703873f, 0.010863997973501682f, 0.00617169588804245f, -0.00931661669164896f, 0.0f, 0.007204215507954359f, -0.010383594781160355f, 0.008176909759640694f, 0.0f, 0.00910070538520813f, 0.0f};
static __constant__ float kLpTrig8[90] = {1.0f, 0.9914448857307434f, 0.13052618503570557f, 0.9659258127212524f, 0.258819043636322f, 0.9238795042037964f, 0.3826834261417389f, 0.8660253882408142f, 0.5f, 0.7933533191680908f, 0.6087614297866821f, 0.7071067690849304f, 0.7071067690849304f, 0.6087614297866821f, 0.7933533191680908f, 1.0f, 0.9238795042037964f, 0.3826834261417389f, 0.7071067690849304f, 0.7071067690849304f, 0.3826834261417389f, 0.9238795042037964f, 6.123234262925839e-17f, 1.0f, -0.3826834261417389f, 0.9238795042037964f, -0.7071067690849304f, 0.7071067690849304f, -0.9238795042037964f, 0.3826834261417389f, 1.0f, 0.7933533191680908f, 0.6087614297866821f, 0.258819043636322f, 0.9659258127212524f, -0.3826834261417389f, 0.9238795042037964f, -0.8660253882408142f, 0.5f, -0.9914448857307434f, -0.13052618503570557f, -0.7071067690849304f, -0.7071067690849304f, -0.13052618503570557f, -0.9914448857307434f, 1.0f, 0.6087614297866821f, 0.7933533191680908f, -0.258819043636322f, 0.9659258127212524f, -0.9238795042037964f, 0.3826834261417389f, -0.8660253882408142f, -0.5f, -0.13052618503570557f, -0.9914448857307434f, 0.7071067690849304f, -0.7071067690849304f, 0.9914448857307434f, 0.13052618503570557f, 1.0f, 0.3826834261417389f, 0.9238795042037964f, -0.7071067690849304f, 0.7071067690849304f, -0.9238795042037964f, -0.3826834261417389f, -1.8369701465288538e-16f, -1.0f, 0.9238795042037964f, -0.3826834261417389f, 0.7071067690849304f, 0.7071067690849304f, -0.3826834261417389f, 0.9238795042037964f, 1.0f, 0.13052618503570557f, 0.9914448857307434f, -0.9659258127212524f, 0.258819043636322f, -0.3826834261417389f, -0.9238795042037964f, 0.8660253882408142f, -0.5f, 0.6087614297866821f, 0.7933533191680908f, -0.7071067690849304f, 0.7071067690849304f, -0.7933533191680908f, -0.6087614297866821f};
#endif
template <> struct SH<8> {
    static constexpr int K = 64;
    static constexpr int NNZ_SYM = 6588;   // entries (i, j <= k)
    __device__ __forceinline__ static float norm(int i) {
        switch (i) {
            case 0: return 0.282094806432724f;
            case 1: return 0.48860251903533936f;
            case 2: return 0.48860251903533936f;
            case 3: return 0.48860251903533936f;
            case 4: return 0.18209140002727509f;
            case 5: return 0.36418280005455017f;
            case 6: return 0.6307831406593323f;
            case 7: return 0.36418280005455017f;
            case 8: return 0.18209140002727509f;
            case 9: return 0.03933623805642128f;
            case 10: return 0.09635371714830399f;
            case 11: return 0.304697185754776f;
            case 12: return 0.7463526725769043f;
            case 13: return 0.304697185754776f;
            case 14: return 0.09635371714830399f;
            case 15: return 0.03933623805642128f;
            case 16: return 0.005960340145975351f;
            case 17: return 0.016858387738466263f;
            case 18: return 0.06307831406593323f;
            case 19: return 0.2676186263561249f;
            case 20: return 0.8462843894958496f;
            case 21: return 0.2676186263561249f;
            case 22: return 0.06307831406593323f;
            case 23: return 0.016858387738466263f;
            case 24: return 0.005960340145975351f;
            case 25: return 0.0006945841596461833f;
            case 26: return 0.002196467947214842f;
            case 27: return 0.009318824857473373f;
            case 28: return 0.045652732253074646f;
            case 29: return 0.2415715456008911f;
            case 30: return 0.935602605342865f;
            case 31: return 0.2415715456008911f;
            case 32: return 0.045652732253074646f;
            case 33: return 0.009318824857473373f;
            case 34: return 0.002196467947214842f;
            case 35: return 0.0006945841596461833f;
            case 36: return 6.572237907676026e-05f;
            case 37: return 0.00022766899201087654f;
            case 38: return 0.00106786226388067f;
            case 39: return 0.005848922301083803f;
            case 40: return 0.035093534737825394f;
            case 41: return 0.22195099294185638f;
            case 42: return 1.0171072483062744f;
            case 43: return 0.22195099294185638f;
            case 44: return 0.035093534737825394f;
            case 45: return 0.005848922301083803f;
            case 46: return 0.00106786226388067f;
            case 47: return 0.00022766899201087654f;
            case 48: return 6.572237907676026e-05f;
            case 49: return 5.233009233052144e-06f;
            case 50: return 1.9580127627705224e-05f;
            case 51: return 9.983946074498817e-05f;
            case 52: return 0.0005990367499180138f;
            case 53: return 0.003973560407757759f;
            case 54: return 0.02809731289744377f;
            case 55: return 0.206472247838974f;
            case 56: return 1.0925484895706177f;
            case 57: return 0.206472247838974f;
            case 58: return 0.02809731289744377f;
            case 59: return 0.003973560407757759f;
            case 60: return 0.0005990367499180138f;
            case 61: return 9.983946074498817e-05f;
            case 62: return 1.9580127627705224e-05f;
            case 63: return 5.233009233052144e-06f;
            default: return 0.0f;
        }
    }
    __device__ __forceinline__ static float ahat(int l) {
        switch (l) {
            case 0: return 3.1415927410125732f;
            case 1: return 2.094395160675049f;
            case 2: return 0.7853981852531433f;
            case 3: return 0.0f;
            case 4: return -0.13089969754219055f;
            case 5: return 0.0f;
            case 6: return 0.04908738657832146f;
            case 7: return 0.0f;
            default: return 0.0f;
        }
    }
    static constexpr int LPS = 6;   // lane-pair product rule: node pairs
    static constexpr int LPQ = 6;   // ... and azimuth quads
    static constexpr int LES = 8;   // lane-pair projected-exponential rule: node pairs
    static constexpr int LEQ = 8;   // ... and azimuth quads
#if defined(SHS_NB) && SHS_NB == 8
    __device__ __forceinline__ static const float* lp_leg() { return kLpLeg8; }
    __device__ __forceinline__ static const float* le_leg() { return kLeLeg8; }
    __device__ __forceinline__ static const float* lp_trig_row(int b) { return kLpTrig8 + b * 15; }
#endif
    __device__ __forceinline__ static float lp_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 15 + h) {
            case 1: return 0.9914448857307434f;
            case 2: return 0.13052618503570557f;
            case 3: return 0.9659258127212524f;
            case 4: return 0.258819043636322f;
            case 5: return 0.9238795042037964f;
            case 6: return 0.3826834261417389f;
            case 7: return 0.8660253882408142f;
            case 8: return 0.5f;
            case 9: return 0.7933533191680908f;
            case 10: return 0.6087614297866821f;
            case 11: return 0.7071067690849304f;
            case 12: return 0.7071067690849304f;
            case 13: return 0.6087614297866821f;
            case 14: return 0.7933533191680908f;
            case 16: return 0.9238795042037964f;
            case 17: return 0.3826834261417389f;
            case 18: return 0.7071067690849304f;
            case 19: return 0.7071067690849304f;
            case 20: return 0.3826834261417389f;
            case 21: return 0.9238795042037964f;
            case 22: return 6.123234262925839e-17f;
            case 23: return 1.0f;
            case 24: return -0.3826834261417389f;
            case 25: return 0.9238795042037964f;
            case 26: return -0.7071067690849304f;
            case 27: return 0.7071067690849304f;
            case 28: return -0.9238795042037964f;
            case 29: return 0.3826834261417389f;
            case 31: return 0.7933533191680908f;
            case 32: return 0.6087614297866821f;
            case 33: return 0.258819043636322f;
            case 34: return 0.9659258127212524f;
            case 35: return -0.3826834261417389f;
            case 36: return 0.9238795042037964f;
            case 37: return -0.8660253882408142f;
            case 38: return 0.5f;
            case 39: return -0.9914448857307434f;
            case 40: return -0.13052618503570557f;
            case 41: return -0.7071067690849304f;
            case 42: return -0.7071067690849304f;
            case 43: return -0.13052618503570557f;
            case 44: return -0.9914448857307434f;
            case 46: return 0.6087614297866821f;
            case 47: return 0.7933533191680908f;
            case 48: return -0.258819043636322f;
            case 49: return 0.9659258127212524f;
            case 50: return -0.9238795042037964f;
            case 51: return 0.3826834261417389f;
            case 52: return -0.8660253882408142f;
            case 53: return -0.5f;
            case 54: return -0.13052618503570557f;
            case 55: return -0.9914448857307434f;
            case 56: return 0.7071067690849304f;
            case 57: return -0.7071067690849304f;
            case 58: return 0.9914448857307434f;
            case 59: return 0.13052618503570557f;
            case 61: return 0.3826834261417389f;
            case 62: return 0.9238795042037964f;
            case 63: return -0.7071067690849304f;
            case 64: return 0.7071067690849304f;
            case 65: return -0.9238795042037964f;
            case 66: return -0.3826834261417389f;
            case 67: return -1.8369701465288538e-16f;
            case 68: return -1.0f;
            case 69: return 0.9238795042037964f;
            case 70: return -0.3826834261417389f;
            case 71: return 0.7071067690849304f;
            case 72: return 0.7071067690849304f;
            case 73: return -0.3826834261417389f;
            case 74: return 0.9238795042037964f;
            case 76: return 0.13052618503570557f;
            case 77: return 0.9914448857307434f;
            case 78: return -0.9659258127212524f;
            case 79: return 0.258819043636322f;
            case 80: return -0.3826834261417389f;
            case 81: return -0.9238795042037964f;
            case 82: return 0.8660253882408142f;
            case 83: return -0.5f;
            case 84: return 0.6087614297866821f;
            case 85: return 0.7933533191680908f;
            case 86: return -0.7071067690849304f;
            case 87: return 0.7071067690849304f;
            case 88: return -0.7933533191680908f;
            case 89: return -0.6087614297866821f;
            default: return 1.0f;
        }
    }
    __device__ __forceinline__ static float le_trig(int b, int h) {   // h = 2m - 1: cos(m phi_b), 2m: sin
        switch (b * 15 + h) {
            case 1: return 0.9951847195625305f;
            case 2: return 0.0980171412229538f;
            case 3: return 0.9807852506637573f;
            case 4: return 0.19509032368659973f;
            case 5: return 0.9569403529167175f;
            case 6: return 0.290284663438797f;
            case 7: return 0.9238795042037964f;
            case 8: return 0.3826834261417389f;
            case 9: return 0.8819212913513184f;
            case 10: return 0.4713967442512512f;
            case 11: return 0.8314695954322815f;
            case 12: return 0.5555702447891235f;
            case 13: return 0.7730104327201843f;
            case 14: return 0.6343932747840881f;
            case 16: return 0.9569403529167175f;
            case 17: return 0.290284663438797f;
            case 18: return 0.8314695954322815f;
            case 19: return 0.5555702447891235f;
            case 20: return 0.6343932747840881f;
            case 21: return 0.7730104327201843f;
            case 22: return 0.3826834261417389f;
            case 23: return 0.9238795042037964f;
            case 24: return 0.0980171412229538f;
            case 25: return 0.9951847195625305f;
            case 26: return -0.19509032368659973f;
            case 27: return 0.9807852506637573f;
            case 28: return -0.4713967442512512f;
            case 29: return 0.8819212913513184f;
            case 31: return 0.8819212913513184f;
            case 32: return 0.4713967442512512f;
            case 33: return 0.5555702447891235f;
            case 34: return 0.8314695954322815f;
            case 35: return 0.0980171412229538f;
            case 36: return 0.9951847195625305f;
            case 37: return -0.3826834261417389f;
            case 38: return 0.9238795042037964f;
            case 39: return -0.7730104327201843f;
            case 40: return 0.6343932747840881f;
            case 41: return -0.9807852506637573f;
            case 42: return 0.19509032368659973f;
            case 43: return -0.9569403529167175f;
            case 44: return -0.290284663438797f;
            case 46: return 0.7730104327201843f;
            case 47: return 0.6343932747840881f;
            case 48: return 0.19509032368659973f;
            case 49: return 0.9807852506637573f;
            case 50: return -0.4713967442512512f;
            case 51: return 0.8819212913513184f;
            case 52: return -0.9238795042037964f;
            case 53: return 0.3826834261417389f;
            case 54: return -0.9569403529167175f;
            case 55: return -0.290284663438797f;
            case 56: return -0.5555702447891235f;
            case 57: return -0.8314695954322815f;
            case 58: return 0.0980171412229538f;
            case 59: return -0.9951847195625305f;
            case 61: return 0.6343932747840881f;
            case 62: return 0.7730104327201843f;
            case 63: return -0.19509032368659973f;
            case 64: return 0.9807852506637573f;
            case 65: return -0.8819212913513184f;
            case 66: return 0.4713967442512512f;
            case 67: return -0.9238795042037964f;
            case 68: return -0.3826834261417389f;
            case 69: return -0.290284663438797f;
            case 70: return -0.9569403529167175f;
            case 71: return 0.5555702447891235f;
            case 72: return -0.8314695954322815f;
            case 73: return 0.9951847195625305f;
            case 74: return -0.0980171412229538f;
            case 76: return 0.4713967442512512f;
            case 77: return 0.8819212913513184f;
            case 78: return -0.5555702447891235f;
            case 79: return 0.8314695954322815f;
            case 80: return -0.9951847195625305f;
            case 81: return -0.0980171412229538f;
            case 82: return -0.3826834261417389f;
            case 83: return -0.9238795042037964f;
            case 84: return 0.6343932747840881f;
            case 85: return -0.7730104327201843f;
            case 86: return 0.9807852506637573f;
            case 87: return 0.19509032368659973f;
            case 88: return 0.290284663438797f;
            case 89: return 0.9569403529167175f;
            case 91: return 0.290284663438797f;
            case 92: return 0.9569403529167175f;
            case 93: return -0.8314695954322815f;
            case 94: return 0.5555702447891235f;
            case 95: return -0.7730104327201843f;
            case 96: return -0.6343932747840881f;
            case 97: return 0.3826834261417389f;
            case 98: return -0.9238795042037964f;
            case 99: return 0.9951847195625305f;
            case 100: return 0.0980171412229538f;
            case 101: return 0.19509032368659973f;
            case 102: return 0.9807852506637573f;
            case 103: return -0.8819212913513184f;
            case 104: return 0.4713967442512512f;
            case 106: return 0.0980171412229538f;
            case 107: return 0.9951847195625305f;
            case 108: return -0.9807852506637573f;
            case 109: return 0.19509032368659973f;
            case 110: return -0.290284663438797f;
            case 111: return -0.9569403529167175f;
            case 112: return 0.9238795042037964f;
            case 113: return -0.3826834261417389f;
            case 114: return 0.4713967442512512f;
            case 115: return 0.8819212913513184f;
            case 116: return -0.8314695954322815f;
            case 117: return 0.5555702447891235f;
            case 118: return -0.6343932747840881f;
            case 119: return -0.7730104327201843f;
            default: return 1.0f;
        }
    }
};

}  // namespace shsgen
