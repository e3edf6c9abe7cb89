// Per-element server update rules, shared by the dense and sparse kernels.
#pragma once

#include "kernels.cuh"

namespace fasgd {

// Hardware approximations (PTX rsqrt.approx / rcp.approx).  Their error is a
// few ulp, far inside the 1e-5 relative bound the results are held to; see
// the rounding notes on fasgd_update below.  FTZ selects the forms that flush
// subnormal inputs and outputs to zero.  In fasgd_update they give the same
// results as the subnormal-preserving forms whenever eps >= 2^-126 and the
// gradients are finite: the radicand is then at least 2^-126, and v, a
// weighted mean of r >= (1 - beta) / sqrt(FLT_MAX) with 1 - beta >= 2^-24,
// is at least 2^-88; neither they nor their reciprocals are subnormal.
template <bool FTZ>
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    if (FTZ)
        asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    else
        asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <bool FTZ>
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    if (FTZ)
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    else
        asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

template <bool FTZ>
__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    if (FTZ)
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    else
        asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Smallest eps for which the flush-to-zero forms are exact substitutes.
constexpr float kFtzSafeEps = 1.17549435e-38f;  // 2^-126

// ASGD / SASGD (Eq. 1-2): theta <- theta - alpha(tau) * g.  Both operations
// are rounded separately (no fused multiply-add), so the result is the
// correctly rounded fp32 sequence.
__device__ __forceinline__ void sgd_update(float& theta, float g, float coef) {
    theta = __fsub_rn(theta, __fmul_rn(coef, g));
}

// FASGD (Eq. 4-8) for one parameter and one gradient entry g.
//   Eq. 4  n <- gamma n + (1 - gamma) g^2
//   Eq. 5  b <- gamma b + (1 - gamma) g
//   Eq. 6  v <- beta v + (1 - beta) / sqrt(max(n - b^2, 0) + eps)
//   Eq. 7-8 theta <- theta - alpha(tau) * g / v      (v just updated)
// n, b and the radicand are formed with one rounding per product and sum
// (no contraction), which makes them the exact fp32 sequence.  The inverse
// square root, the reciprocal of v and the two fused multiply-adds of the
// v and theta updates differ from a once-rounded sequence by a few ulp; v is
// a positive weighted mean, so that difference does not grow, and theta only
// accumulates it relative to the size of each step.
// STD selects the prose reading of Sec. 2.2: v averages the std itself
// (r = sqrt(max(n - b^2, 0) + eps)) and the step divides by it.  With
// eps >= 2^-126 the std is >= 2^-63 and v >= 2^-87, so the flush-to-zero
// forms stay exact substitutes there too.
template <bool FTZ = false, bool STD = false>
__device__ __forceinline__ void fasgd_update(float& theta, float& n, float& b, float& v,
                                             float g, float coef, const StatParams& sp) {
    n = __fadd_rn(__fmul_rn(sp.gamma, n), __fmul_rn(sp.one_m_gamma, __fmul_rn(g, g)));
    b = __fadd_rn(__fmul_rn(sp.gamma, b), __fmul_rn(sp.one_m_gamma, g));
    const float var = fmaxf(__fsub_rn(n, __fmul_rn(b, b)), 0.0f);
    const float rad = __fadd_rn(var, sp.eps);
    const float r = STD ? sqrt_approx<FTZ>(rad) : rsqrt_approx<FTZ>(rad);
    v = fmaf(sp.beta, v, sp.one_m_beta * r);
    theta = fmaf(-(coef * g), rcp_approx<FTZ>(v), theta);
}

// The same rule with every operation correctly rounded and none fused
// (IEEE square root and division, separate multiplies and adds): the exact
// fp32 sequence Eq. 4-8 define, bit for bit on any IEEE machine.  Selected
// per handle (fasgd_set_exact) where results must be reproducible bit for
// bit, e.g. in closed-loop simulations; it costs a division and a square
// root per element-push on the pipes the fast form leaves idle.
template <bool STD = false>
__device__ __forceinline__ void fasgd_update_exact(float& theta, float& n, float& b, float& v,
                                                   float g, float coef, const StatParams& sp) {
    n = __fadd_rn(__fmul_rn(sp.gamma, n), __fmul_rn(sp.one_m_gamma, __fmul_rn(g, g)));
    b = __fadd_rn(__fmul_rn(sp.gamma, b), __fmul_rn(sp.one_m_gamma, g));
    const float var = fmaxf(__fsub_rn(n, __fmul_rn(b, b)), 0.0f);
    const float root = __fsqrt_rn(__fadd_rn(var, sp.eps));
    const float r = STD ? root : __fdiv_rn(1.0f, root);
    v = __fadd_rn(__fmul_rn(sp.beta, v), __fmul_rn(sp.one_m_beta, r));
    theta = __fsub_rn(theta, __fdiv_rn(__fmul_rn(coef, g), v));
}

// ---- the exact sequence on pairs -------------------------------------------
// Two fp32 values in one 64-bit register pair, with the packed fp32
// instructions of sm_100 and later (each half rounded on its own, no
// flush to zero): one issue slot for two operations.
struct Pair {
    unsigned long long bits;
};
__device__ __forceinline__ Pair pair(float x, float y) {
    Pair p;
    asm("mov.b64 %0, {%1, %2};" : "=l"(p.bits) : "f"(x), "f"(y));
    return p;
}
__device__ __forceinline__ void unpack(Pair p, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(p.bits));
}
__device__ __forceinline__ Pair add2(Pair a, Pair b) {
    Pair d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.bits) : "l"(a.bits), "l"(b.bits));
    return d;
}
__device__ __forceinline__ Pair mul2(Pair a, Pair b) {
    Pair d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d.bits) : "l"(a.bits), "l"(b.bits));
    return d;
}
__device__ __forceinline__ Pair fma2(Pair a, Pair b, Pair c) {
    Pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.bits) : "l"(a.bits), "l"(b.bits), "l"(c.bits));
    return d;
}

// fl(a b) that stays a rounding of its own: a product made with mul2 and fed
// to add2 comes out as one fused multiply-add here (also under -fmad=false),
// so it is formed as fma(a, b, -0), with a -0 the compiler does not see.
__device__ __forceinline__ Pair product2(Pair a, Pair b, const StatParams& sp) {
    return fma2(a, b, pair(sp.minus_zero, sp.minus_zero));
}

// What the pushes of a pass saw, kept while they are applied: whether the
// chains of exact_update2 gave the correctly rounded sequence throughout.  That
// holds for rad in [2^-100, 2^100], v in [2^-60, 2^60] and a quotient q = a / v,
// a = fl(coef g), that is zero or of magnitude in [2^-66, 2^94]: a and q are then
// normal, no intermediate is subnormal and no residual rounded.  A smaller q does
// no harm either where |theta| is 2^-40 or more: half the gap to its neighbours is
// at least 2^-65, so theta stays as it is whatever q rounds to.  Gradients far
// below their neighbours, as a saturated softmax leaves them, would otherwise send
// whole passes the long way (25M, K = 8, one gradient in a hundred times 1e-22:
// 1114 us with a bound on a alone, 424 with CUDA's functions throughout, 247 so,
// as without such gradients).  NaN fails.  One add-and-compare instruction per
// bound, and no branch among the pushes: a pass looks once, at its end, and forms
// the quads that left the range again (exact_quad).
template <int ARITH> struct Guard {
    __device__ __forceinline__ bool ok() const { return true; }
};

// Square root, reciprocal and quotient of pairs.  CUDA's own square root and
// division are correctly rounded over the whole fp32 range and cost about 80
// issue slots per element-push here, which made the exact pass issue-bound
// (K = 8 at 25M parameters: 427 us, 55 % of the copy bandwidth).  Inside the
// range above, which every finite training run keeps to, the hardware
// approximations refined by fused multiply-adds are correctly rounded as well
// (Markstein, IBM J. Res. Dev. 34(1), 1990: the residual of an almost rounded
// root or quotient is exact in one fused multiply-add, and one correction by a
// rounded reciprocal then rounds correctly):
//   root:        s = rad y, y ~ rad^-1/2;   s + (rad - s^2) y / 2
//   reciprocal:  z ~ 1 / x;                 z + (1 - x z) z
//   quotient:    q = a z, z = fl(1/v);      twice q + (a - v q) z (the first
//                makes q faithful, the second rounds it).
// Reciprocal and quotient come negated (the sign is free at the approximation's
// input), which keeps the sign of a zero a.  tests/test_gpu_exact_sweep.py holds
// these three functions to CUDA's: root and reciprocal for every fp32 value of
// the range, the quotient on 4e10 pairs (random, near midpoints, mantissas at
// both ends).
__device__ __forceinline__ Pair root2(Pair rad, Pair minus_rad) {
    float x, y;
    unpack(rad, x, y);
    const Pair inv = pair(rsqrt_approx<true>(x), rsqrt_approx<true>(y));
    const Pair s = mul2(rad, inv);
    return fma2(fma2(s, s, minus_rad), mul2(inv, pair(-0.5f, -0.5f)), s);
}
__device__ __forceinline__ Pair minus_reciprocal2(Pair x) {
    float a, b;
    unpack(x, a, b);
    const Pair w = pair(rcp_approx<true>(-a), rcp_approx<true>(-b));
    return fma2(fma2(x, w, pair(1.f, 1.f)), w, w);
}
// -(a / v), given the correctly rounded -(1 / v).
__device__ __forceinline__ Pair minus_quotient2(Pair a, Pair v, Pair minus_z) {
    Pair minus_q = mul2(a, minus_z);
    minus_q = fma2(fma2(v, minus_q, a), minus_z, minus_q);
    return fma2(fma2(v, minus_q, a), minus_z, minus_q);
}

// Brings the lowest quotient in range, 2^-66, to theta's line, 2^-40.
constexpr float kQuotientScale = 67108864.0f;   // 2^26

// fasgd_update_exact on two parameters, the same bits.  25M, K = 8 / 16, push +
// apply + pull: 464 us with CUDA's functions (K = 8), 282 / 517 with the negations
// as operations of their own, 273 / 494 now.
template <bool STD, class G>
__device__ __forceinline__ void exact_update2(Pair& theta, Pair& n, Pair& b, Pair& v, Pair g, float coef,
                                              const StatParams& sp, G& guard) {
    const Pair minus1 = pair(-1.f, -1.f);
    const Pair gamma = pair(sp.gamma, sp.gamma), rest = pair(sp.one_m_gamma, sp.one_m_gamma);
    n = add2(product2(gamma, n, sp), product2(rest, mul2(g, g), sp));
    b = add2(product2(gamma, b, sp), product2(rest, g, sp));
    float x, y;
    unpack(fma2(product2(b, b, sp), minus1, n), x, y);     // n - b^2
    const Pair var = pair(fmaxf(x, 0.0f), fmaxf(y, 0.0f));
    const Pair rad = add2(var, pair(sp.eps, sp.eps));
    const Pair minus_rad = fma2(var, minus1, pair(-sp.eps, -sp.eps));
    unpack(rad, x, y);
    guard.see_rad(x, y);
    const Pair root = root2(rad, minus_rad);
    // v' = beta v + (1 - beta) r.
    const Pair step = STD ? product2(pair(sp.one_m_beta, sp.one_m_beta), root, sp)
                          : product2(pair(-sp.one_m_beta, -sp.one_m_beta), minus_reciprocal2(root), sp);
    v = add2(product2(pair(sp.beta, sp.beta), v, sp), step);
    unpack(v, x, y);
    guard.see_v(x, y);
    // a and q come times 2^26 (exact where a is normal): a small a then leaves no
    // rounded residual (its last bit is 2^-146 or more), and one comparison serves
    // q and theta.  The last operation scales q back and rounds once.
    const float up = coef * kQuotientScale;
    const Pair minus_q = minus_quotient2(mul2(pair(up, up), g), v, minus_reciprocal2(v));
    float tx, ty;
    unpack(minus_q, x, y);
    unpack(theta, tx, ty);
    guard.see_q(x, y, tx, ty);
    theta = fma2(minus_q, pair(1.f / kQuotientScale, 1.f / kQuotientScale), theta);
}

// Arithmetic of a pass: hardware approximations (subnormal-preserving or
// flush-to-zero forms) or the exact sequence.
enum : int { kArithApprox = 0, kArithApproxFtz = 1, kArithExact = 2 };

template <> struct Guard<kArithExact> {
    uint32_t rad = 0, v = 0, q_min = 0xffffffffu, q_max = 0;
    __device__ __forceinline__ void see_rad(float x, float y) {
        rad = __viaddmax_u32(__float_as_uint(x), 0u - kRadLo, rad);
        rad = __viaddmax_u32(__float_as_uint(y), 0u - kRadLo, rad);
    }
    __device__ __forceinline__ void see_v(float x, float y) {
        v = __viaddmax_u32(__float_as_uint(x), 0u - kLo, v);
        v = __viaddmax_u32(__float_as_uint(y), 0u - kLo, v);
    }
    // The larger of the scaled quotient and theta, NaN from either.
    static __device__ __forceinline__ uint32_t larger(float q, float t) {
        float m;
        asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(fabsf(q)), "f"(fabsf(t)));
        return __float_as_uint(m);
    }
    __device__ __forceinline__ void see_q(float x, float y, float tx, float ty) {
        const uint32_t mx = larger(x, tx), my = larger(y, ty);
        q_min = __viaddmin_u32(mx, 0xffffffffu, q_min);   // zeros wrap to the largest
        q_min = __viaddmin_u32(my, 0xffffffffu, q_min);
        q_max = max(q_max, max(mx, my));
    }
    __device__ __forceinline__ bool ok() const {
        return rad <= kRadHi - kRadLo && v <= kHi - kLo && q_min >= kQLo - 1 && q_max <= kQHi;
    }
    static constexpr uint32_t kRadLo = 27u << 23, kRadHi = 227u << 23;   // 2^-100, 2^100
    static constexpr uint32_t kLo = 67u << 23, kHi = 187u << 23;         // 2^-60, 2^60
    static constexpr uint32_t kQLo = 87u << 23, kQHi = 247u << 23;       // 2^-40, 2^120
};

template <int ARITH, bool STD>
__device__ __forceinline__ void rule_update(float& theta, float& n, float& b, float& v, float g,
                                            float coef, const StatParams& sp) {
    if (ARITH == kArithExact)
        fasgd_update_exact<STD>(theta, n, b, v, g, coef, sp);
    else
        fasgd_update<ARITH == kArithApproxFtz, STD>(theta, n, b, v, g, coef, sp);
}

// One push on four consecutive parameters.
template <int RULE, int ARITH>
__device__ __forceinline__ void update4(float4& th, float4& n, float4& b, float4& v, const float4& g,
                                        float coef, const StatParams& sp, Guard<ARITH>& guard) {
    constexpr bool STD = RULE == kRuleFasgdStd;
    if constexpr (RULE == kRuleSgd) {
        sgd_update(th.x, g.x, coef);
        sgd_update(th.y, g.y, coef);
        sgd_update(th.z, g.z, coef);
        sgd_update(th.w, g.w, coef);
    } else if constexpr (ARITH == kArithExact) {
        Pair t0 = pair(th.x, th.y), n0 = pair(n.x, n.y), b0 = pair(b.x, b.y), v0 = pair(v.x, v.y);
        Pair t1 = pair(th.z, th.w), n1 = pair(n.z, n.w), b1 = pair(b.z, b.w), v1 = pair(v.z, v.w);
        exact_update2<STD>(t0, n0, b0, v0, pair(g.x, g.y), coef, sp, guard);
        exact_update2<STD>(t1, n1, b1, v1, pair(g.z, g.w), coef, sp, guard);
        unpack(t0, th.x, th.y);
        unpack(n0, n.x, n.y);
        unpack(b0, b.x, b.y);
        unpack(v0, v.x, v.y);
        unpack(t1, th.z, th.w);
        unpack(n1, n.z, n.w);
        unpack(b1, b.z, b.w);
        unpack(v1, v.z, v.w);
    } else {
        rule_update<ARITH, STD>(th.x, n.x, b.x, v.x, g.x, coef, sp);
        rule_update<ARITH, STD>(th.y, n.y, b.y, v.y, g.y, coef, sp);
        rule_update<ARITH, STD>(th.z, n.z, b.z, v.z, g.z, coef, sp);
        rule_update<ARITH, STD>(th.w, n.w, b.w, v.w, g.w, coef, sp);
    }
}

// The quad of parameters at e (a multiple of 4) after K pushes in exact
// arithmetic, formed again from memory with CUDA's square root and division:
// for quads whose guard failed, before anything of them is stored.  g0
// replaces grad[0].
struct QuadState {
    float4 th, n, b, v;
};
template <bool STD>
__device__ __noinline__ QuadState exact_quad(const float* theta, const float* n, const float* b,
                                             const float* v, const float* g0, const float* const* grad,
                                             const float* coef, int K, int64_t e, const StatParams& sp) {
    QuadState q;
    q.th = *reinterpret_cast<const float4*>(theta + e);
    q.n = *reinterpret_cast<const float4*>(n + e);
    q.b = *reinterpret_cast<const float4*>(b + e);
    q.v = *reinterpret_cast<const float4*>(v + e);
    float4 g = *reinterpret_cast<const float4*>(g0 + e);
#pragma unroll 1
    for (int k = 0; k < K; ++k) {
        float4 next = g;
        if (k + 1 < K) next = *reinterpret_cast<const float4*>(grad[k + 1] + e);
        fasgd_update_exact<STD>(q.th.x, q.n.x, q.b.x, q.v.x, g.x, coef[k], sp);
        fasgd_update_exact<STD>(q.th.y, q.n.y, q.b.y, q.v.y, g.y, coef[k], sp);
        fasgd_update_exact<STD>(q.th.z, q.n.z, q.b.z, q.v.z, g.z, coef[k], sp);
        fasgd_update_exact<STD>(q.th.w, q.n.w, q.b.w, q.v.w, g.w, coef[k], sp);
        g = next;
    }
    return q;
}

}  // namespace fasgd
