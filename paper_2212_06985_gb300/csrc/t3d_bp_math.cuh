// Check-node arithmetic shared by the BP kernels (Sec. 4.1, Eq. 2), FP32.
// For an input x (a variable->check message) the pair t = tanh(|x|/2),
// d = 1 - t = 2 e^{-|x|} / (1 + e^{-|x|}) is formed without cancellation;
// products of pairs are (tA tB, dA + tA dB), exact algebra, so P = prod t and
// D = 1 - P stay accurate even when P rounds to 1 in FP32; the output
// magnitude is 2 atanh(P) = log((1 + P) / D).  Also the flooding check node
// over a fixed number of inputs built from those pairs, and the four-samples-
// per-thread row accessors of the sample-innermost message layouts.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace t3d {
namespace bpm {

struct TD {
    float t;  // tanh(|x|/2)
    float d;  // 1 - tanh(|x|/2)
};

__device__ __forceinline__ TD td_mul(TD A, TD B) { return TD{A.t * B.t, fmaf(A.t, B.d, A.d)}; }

// MUFU approximations (PTX ex2/rcp/lg2 .approx.ftz, a few ulp); the
// formulations below only feed them arguments where that relative accuracy
// carries through without cancellation.
__device__ __forceinline__ float ex2_approx(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float rcp_approx(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

__device__ __forceinline__ float lg2_approx(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// (tanh(|x|/2), 1 - tanh(|x|/2)) = ((1 - E), 2E) / (1 + E) with E = e^{-|x|}.
// For |x| < 0.1 the difference 1 - E is taken from its Taylor series
// |x| - |x|^2/2 + |x|^3/6 - |x|^4/24 (truncation < 1e-6 relative) instead of
// subtracting two nearly equal numbers; above 0.1 the subtraction loses at
// most a factor E/(1-E) < 10 on E's few-ulp error.  Both forms are evaluated
// and one selected.
__device__ __forceinline__ TD td_of(float x)
{
    const float a = fabsf(x);
    const float E = ex2_approx(-a * kLog2e);
    const float r = rcp_approx(1.0f + E);
    float h = fmaf(a, -1.0f / 24.0f, 1.0f / 6.0f);
    h = fmaf(a, h, -0.5f);
    h = fmaf(a, h, 1.0f);
    const float om = (a < 0.1f) ? a * h : 1.0f - E;
    return TD{om * r, (E + E) * r};
}

// 2 atanh(P) for P = prod t, D = 1 - P: for P < 0.05 the odd series
// 2P (1 + P^2/3 + P^4/5) (truncation < 3e-10 relative); above it
// log((1 + P) / D), whose argument exceeds 1.1 so the approximate logarithm's
// absolute error stays below 2e-6 of the result.  D = 0 (underflow) gives +inf,
// which the clamp turns into 30.
__device__ __forceinline__ float two_atanh(float P, float D)
{
    const float u = P * P;
    const float series = 2.0f * P * fmaf(u, fmaf(u, 1.0f / 5.0f, 1.0f / 3.0f), 1.0f);
    const float logv = kLn2 * lg2_approx((1.0f + P) * rcp_approx(D));
    return (P < 0.05f) ? series : logv;
}


// Flooding check node over K inputs (Eq. 2): out[i] = (-1)^{syn} times the
// product of the other inputs' signs times 2 atanh(prod_{j != i} tanh(|x_j|/2)),
// from prefix and suffix products of the (t, d) pairs, clamped to |M| <= 30.
constexpr float kCheckClamp = 30.0f;

template <int K>
__device__ __forceinline__ void check_node(const float (&x)[K], bool syn, float (&out)[K])
{
    TD v[K], pre[K], suf[K];
    uint32_t sgn_all = syn ? 0x80000000u : 0u;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        v[i] = td_of(x[i]);
        sgn_all ^= __float_as_uint(x[i]);
    }
    pre[0] = TD{1.0f, 0.0f};
#pragma unroll
    for (int i = 1; i < K; ++i) pre[i] = td_mul(pre[i - 1], v[i - 1]);
    suf[K - 1] = TD{1.0f, 0.0f};
#pragma unroll
    for (int i = K - 2; i >= 0; --i) suf[i] = td_mul(v[i + 1], suf[i + 1]);
#pragma unroll
    for (int i = 0; i < K; ++i) {
        const TD o = td_mul(pre[i], suf[i]);
        const float mag = fminf(two_atanh(o.t, o.d), kCheckClamp);
        const uint32_t sgn = (sgn_all ^ __float_as_uint(x[i])) & 0x80000000u;
        out[i] = __uint_as_float(__float_as_uint(mag) | sgn);
    }
}

// The check node on a lane's two samples at once with the packed two-wide FP32
// instructions (__fadd2_rn, __fmul2_rn, __ffma2_rn): every operation is the scalar
// one of td_of / td_mul / two_atanh (t3d_bp_math.cuh) in the same order and
// rounding, applied to both samples, so the messages are bit for bit those of the
// scalar code; the MUFU approximations and the selects stay per sample.
struct TD2 {
    float2 t, d;
};

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

__device__ __forceinline__ TD2 td2_mul(const TD2& A, const TD2& B)
{
    return TD2{__fmul2_rn(A.t, B.t), __ffma2_rn(A.t, B.d, A.d)};
}

__device__ __forceinline__ TD2 td2_of(float2 x)
{
    const float2 a = make_float2(fabsf(x.x), fabsf(x.y));
    const float2 m = __fmul2_rn(make_float2(-a.x, -a.y), f2(kLog2e));
    const float2 E = make_float2(ex2_approx(m.x), ex2_approx(m.y));
    const float2 e1 = __fadd2_rn(f2(1.0f), E);
    const float2 r = make_float2(rcp_approx(e1.x), rcp_approx(e1.y));
    float2 h = __ffma2_rn(a, f2(-1.0f / 24.0f), f2(1.0f / 6.0f));
    h = __ffma2_rn(a, h, f2(-0.5f));
    h = __ffma2_rn(a, h, f2(1.0f));
    const float2 ah = __fmul2_rn(a, h);
    const float2 ome = __ffma2_rn(E, f2(-1.0f), f2(1.0f));
    const float2 om = make_float2(a.x < 0.1f ? ah.x : ome.x, a.y < 0.1f ? ah.y : ome.y);
    return TD2{__fmul2_rn(om, r), __fmul2_rn(__fadd2_rn(E, E), r)};
}

__device__ __forceinline__ float2 two_atanh2(float2 P, float2 D)
{
    const float2 u = __fmul2_rn(P, P);
    const float2 poly = __ffma2_rn(u, __ffma2_rn(u, f2(1.0f / 5.0f), f2(1.0f / 3.0f)), f2(1.0f));
    const float2 series = __fmul2_rn(__fmul2_rn(f2(2.0f), P), poly);
    const float2 arg = __fmul2_rn(__fadd2_rn(f2(1.0f), P), make_float2(rcp_approx(D.x), rcp_approx(D.y)));
    const float2 logv = __fmul2_rn(f2(kLn2), make_float2(lg2_approx(arg.x), lg2_approx(arg.y)));
    return make_float2(P.x < 0.05f ? series.x : logv.x, P.y < 0.05f ? series.y : logv.y);
}

// check_node on a lane's two samples: the same products in the same order (a product with the
// neutral pair (1, 0) is exact, so the ends of the prefix and suffix chains are the inputs
// themselves), bit for bit.
template <int K>
__device__ __forceinline__ void check_node2(const float2 (&x)[K], bool syn0, bool syn1, float2 (&out)[K])
{
    TD2 v[K], suf[K];
    // the inputs' sign bits, packed (input i at bit K - 1 - i): the inputs themselves need not stay in
    // registers, which for K = 7 spilled.  (The toric code's four inputs fit either way, and t3d_bp.cu
    // keeps them: with packed signs its iteration takes 2.7% longer.)
    uint32_t sg0 = 0, sg1 = 0;
#pragma unroll
    for (int i = 0; i < K; ++i) {
        v[i] = td2_of(x[i]);
        sg0 = __funnelshift_l(__float_as_uint(x[i].x), sg0, 1);
        sg1 = __funnelshift_l(__float_as_uint(x[i].y), sg1, 1);
    }
    // an output's sign: the parity of the other inputs' and the syndrome
    const uint32_t all0 = ((uint32_t)__popc(sg0) + (syn0 ? 1u : 0u)) << 31;
    const uint32_t all1 = ((uint32_t)__popc(sg1) + (syn1 ? 1u : 0u)) << 31;
    if constexpr (K >= 2) suf[K - 2] = v[K - 1];
#pragma unroll
    for (int i = K - 3; i >= 0; --i) suf[i] = td2_mul(v[i + 1], suf[i + 1]);
    TD2 pre = v[0];
#pragma unroll
    for (int i = 0; i < K; ++i) {
        TD2 o;
        if constexpr (K == 1)
            o = TD2{f2(1.0f), f2(0.0f)};   // no other input
        else
            o = i == 0 ? suf[0] : (i == K - 1 ? pre : td2_mul(pre, suf[i]));
        if (i > 0 && i < K - 1) pre = td2_mul(pre, v[i]);
        const float2 a = two_atanh2(o.t, o.d);
        const float m0 = fminf(a.x, kCheckClamp), m1 = fminf(a.y, kCheckClamp);
        const uint32_t g0 = (all0 ^ (sg0 << (32 - K + i))) & 0x80000000u;
        const uint32_t g1 = (all1 ^ (sg1 << (32 - K + i))) & 0x80000000u;
        out[i] = make_float2(__uint_as_float(__float_as_uint(m0) | g0), __uint_as_float(__float_as_uint(m1) | g1));
    }
}

// Sample-innermost message rows (samples of a chunk padded to 64): a thread
// takes four consecutive samples of one row with 16-byte loads and stores.
__device__ __forceinline__ float4 ld4(const float* base, int64_t row, int64_t S, int64_t smp)
{
    return __ldg(reinterpret_cast<const float4*>(base + row * S + smp));
}

__device__ __forceinline__ void st4(float* base, int64_t row, int64_t S, int64_t smp, float4 v)
{
    *reinterpret_cast<float4*>(base + row * S + smp) = v;
}

__device__ __forceinline__ float comp(const float4& v, int c) { return c == 0 ? v.x : c == 1 ? v.y : c == 2 ? v.z : v.w; }

}  // namespace bpm
}  // namespace t3d
