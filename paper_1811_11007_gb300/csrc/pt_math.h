// Device arithmetic written for the latency of the Newton solves, with the bounds
// that tests/test_gpu_numerics.py checks.
#pragma once

#include <cmath>

#include <cuda_runtime.h>

namespace pt {

// 1/x rounded to nearest, for x in the middle of the FP32 range: the hardware's
// approximation and one residual correction (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990).
// Equal to __frcp_rn on every significand (tests/test_gpu_numerics.py checks all of
// them, at both signs); extreme exponents take __frcp_rn itself, whose call and
// branches cost about 240 dependent cycles in place of 80.
__device__ __forceinline__ float rcp_rn(float x) {
    if ((((unsigned)__float_as_int(x) >> 23 & 0xffu) - 64u) > 126u) return __frcp_rn(x);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return __fmaf_rn(r, __fmaf_rn(-x, r, 1.0f), r);
}

// ---------------------------------------------------------------- FP32 pairs
// The mixed path runs its Newton iterations on FP32 partials, but every score
// it reports comes from partials carried as unevaluated sums h + l of two FP32
// numbers (|l| <= ulp(h)/2, about 48 significant bits): FP32 rounding errors of
// a partial repeat at every site that shares its sub-pattern (a constant
// column below a node, say, at thousands of sites), so at 10^4 sites they add
// up to ~1e-3 nats; the pairs bring that below 1e-6.  Error-free steps:
// Dekker's product by FMA (a*b = p + fma(a, b, -p)) and Knuth's two-sum.
// Explicit _rn intrinsics keep the compiler from contracting them.
struct F2 {
    float h, l;
};
__device__ __forceinline__ F2 f2_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
// h + l renormalised, for |h| >= |l| (Dekker's fast two-sum)
__device__ __forceinline__ F2 f2_norm(float h, float l) {
    const float s = __fadd_rn(h, l);
    return F2{s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return f2_norm(p, e);
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    const F2 s = f2_two_sum(a.h, b.h);
    return f2_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 f2_of(double x) {
    const float h = (float)x;
    return F2{h, (float)(x - (double)h)};
}

// ---------------------------------------------------------------- transition matrices from pairs
// 2^(i/32) as pairs, for expm1_pair; init by 32 or more threads, then a barrier.
struct Exp2Tab {
    F2 t[32];
    __device__ __forceinline__ void init() {
        for (int i = threadIdx.x; i < 32; i += blockDim.x) t[i] = f2_of(exp2(i * 0.03125));
    }
};
// exp(x) - 1 of a pair x in [-80, 0], to a few units of 2^-47 relative: x = n ln2 / 32 + r,
// |r| <= ln2 / 64; expm1(r) = r + r^2 (1/2 + r / 6 + ...) by its Taylor series (terms
// past r / 6 need only FP32), then T - 1 + T expm1(r) with T = 2^(n/32).
__device__ __forceinline__ F2 expm1_pair(F2 x, const Exp2Tab& tab) {
    // ln2 / 32 = c1 + c2 + c3, c1 of 12 bits: n c1 is exact for |n| < 4096
    const float c1 = 0x1.62ep-6f, c2 = 0x1.0bfbe8p-20f, c3 = 0x1.cf79acp-45f;
    const float n = rintf(__fmul_rn(x.h, 46.166241f));
    const F2 a = f2_two_sum(x.h, -__fmul_rn(n, c1));
    const float p2 = __fmul_rn(n, c2);
    const F2 b = f2_two_sum(a.h, -p2);
    const float lo = __fadd_rn(__fadd_rn(a.l, b.l), __fsub_rn(x.l, __fmaf_rn(n, c3, __fmaf_rn(n, c2, -p2))));
    const F2 r = f2_norm(b.h, lo);
    const F2 r6 = f2_mul(r, F2{0x1.555556p-3f, -0x1.555556p-28f});
    const float tail = __fmul_rn(__fmul_rn(r.h, r.h), __fmaf_rn(r.h, 1.0f / 120.0f, 1.0f / 24.0f));
    const F2 h = f2_two_sum(0.5f, r6.h);
    const F2 q = f2_norm(h.h, __fadd_rn(h.l, __fadd_rn(r6.l, tail)));
    const F2 p = f2_add(r, f2_mul(f2_mul(r, r), q));
    const int ni = (int)n;
    const float sc = __int_as_float((127 + (ni >> 5)) << 23);
    const F2 T{tab.t[ni & 31].h * sc, tab.t[ni & 31].l * sc};
    const F2 one = f2_two_sum(-1.0f, T.h);
    return f2_add(f2_norm(one.h, __fadd_rn(one.l, T.l)), f2_mul(T, p));
}
// One entry of P(t) = I + sum_{k=1..3} W_k (exp(lam_k r t) - 1), rounded to FP32, from
// the pairs W_k (w[1..3]) and em_k = expm1(lam_k r t) (em[k * stride]).  certain: the
// rounding is that of the FP64 sum W_0 + sum W_k exp(lam_k r t) (Ziv's test: both ends
// of the error interval round alike).  Half-width of the interval, with u = 2^-24 and mag
// the sum of |W_k em_k|: the pairs W_k and em_k are good to a few 2^-47 and the sums here
// to 33 u^2, together below 2^-42 of mag; beside delta = 1 the sums lose up to 12 u^2
// more; and base is how far the FP64 sum may lie from the exact one (p_entry_base; the
// default holds where the W_k miss delta by at most 2^-49 and sum to less than one).
__device__ __forceinline__ float p_entry_pair(float delta, const F2* w, const F2* em, int stride, bool& certain,
                                              float base = 0x1p-48f) {
    float s = delta, c = 0.f, mag = 0.f;
#pragma unroll
    for (int k = 1; k < 4; ++k) {
        const F2 a = w[k], e = em[k * stride];
        const float p = __fmul_rn(a.h, e.h);
        const float pe = __fmaf_rn(a.l, e.h, __fmaf_rn(a.h, e.l, __fmaf_rn(a.h, e.h, -p)));
        const F2 t = f2_two_sum(s, p);
        s = t.h;
        c = __fadd_rn(c, __fadd_rn(t.l, pe));
        mag = __fadd_rn(mag, fabsf(p));
    }
    const float eps = __fmaf_rn(mag, 0x1p-42f, __fmaf_rn(delta, 0x1.8p-45f, base));
    const float a = __fadd_rn(s, __fsub_rn(c, eps)), b = __fadd_rn(s, __fadd_rn(c, eps));
    certain = a == b;
    return a;
}
// The base of p_entry_pair for an entry's W_0..3: what the W_k miss delta by (they are
// rounded products of eigenvectors, scaled by sqrt(pi_j / pi_i): 6e-15 at mild
// frequencies, 2e-13 at frequencies of 1e-3), and the rounding of the FP64 sum, of its
// exponentials and of this difference, below 9 * 2^-53 of the sum of |W_k|.
__device__ __forceinline__ float p_entry_base(double delta, const double* W) {
    const double miss = fabs(((W[0] + W[1]) + W[2]) + W[3] - delta);
    const double all = (fabs(W[0]) + fabs(W[1])) + (fabs(W[2]) + fabs(W[3]));
    return __double2float_ru(fma(all, 0x1p-49, miss));
}

}  // namespace pt
