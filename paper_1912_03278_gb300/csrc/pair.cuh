// pair.cuh -- two FP32 values per instruction (PTX add/sub/mul/fma.rn.f32x2,
// sm_100 and up) and the double-float algorithms of df32.cuh on such pairs.
// Each half is rounded exactly as by the scalar instruction, so a pair form
// gives the scalar form's bits; what it saves is issue slots.
#pragma once
#include <cuda_runtime.h>

#include "df32.cuh"

namespace ihmc {

typedef unsigned long long pair_t;

__device__ __forceinline__ pair_t pk(float a, float b) {
    pair_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ pair_t pk1(float a) { return pk(a, a); }
__device__ __forceinline__ void upk(pair_t v, float &a, float &b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ pair_t add2(pair_t a, pair_t b) {
    pair_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair_t sub2(pair_t a, pair_t b) {
    pair_t r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair_t mul2(pair_t a, pair_t b) {
    pair_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ pair_t fma2(pair_t a, pair_t b, pair_t c) {
    pair_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
// a value the compiler has to keep (not recompute from what it was made of)
__device__ __forceinline__ float kept(float x) {
    asm volatile("" : "+f"(x));
    return x;
}

// tanh of a pair: tanh_f's operations (device_common.cuh) without its clamp of
// |x| at 20, which changes no bit of a finite argument (1 - 2/(1 + e^{2|x|})
// is 1 from |x| = 9 on, up to e^{2|x|} = inf).
__device__ __forceinline__ pair_t tanh2(pair_t x) {
    const pair_t one = pk1(1.0f);
    float x0, x1, y0, y1, e0, e1, d0, d1, r0, r1, t0, t1;
    upk(x, x0, x1);
    upk(mul2(x, pk1(2.8853900817779268f)), y0, y1);   // 2 log2(e) x
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e0) : "f"(fabsf(y0)));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e1) : "f"(fabsf(y1)));
    upk(add2(pk(e0, e1), one), d0, d1);
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(d0));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r1) : "f"(d1));
    upk(fma2(pk1(-2.0f), pk(r0, r1), one), t0, t1);
    return pk(copysignf(t0, x0), copysignf(t1, x1));
}

// ---- double-floats, two at a time -----------------------------------------
struct f2x2 {
    pair_t hi, lo;
};

__device__ __forceinline__ f2x2 dup_df(f2 a) { return f2x2{pk1(a.hi), pk1(a.lo)}; }
__device__ __forceinline__ f2x2 two_sum(pair_t a, pair_t b) {
    const pair_t s = add2(a, b);
    const pair_t bb = sub2(s, a);
    return f2x2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ f2x2 fast_two_sum(pair_t a, pair_t b) {
    const pair_t s = add2(a, b);
    return f2x2{s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ f2x2 df_add_f(f2x2 a, pair_t b) {
    const f2x2 s = two_sum(a.hi, b);
    return fast_two_sum(s.hi, add2(s.lo, a.lo));
}
__device__ __forceinline__ f2x2 df_add_q(f2x2 a, f2x2 b) {
    const f2x2 s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ f2x2 df_sub_q(f2x2 a, f2x2 b) {   // a + (-b)
    const pair_t s = sub2(a.hi, b.hi);
    const pair_t bb = sub2(s, a.hi);
    const pair_t e = sub2(sub2(a.hi, sub2(s, bb)), add2(b.hi, bb));
    return fast_two_sum(s, add2(e, sub2(a.lo, b.lo)));
}
// Products.  m = -(a.hi b) stands in for p = a.hi b, whose sign the rounding
// error fma(a.hi, b, -p) needs reversed; the caller has -b or -a.hi for less.
__device__ __forceinline__ f2x2 df_mul_f(f2x2 a, pair_t b, pair_t neg_b) {
    const pair_t m = mul2(a.hi, neg_b);
    pair_t e = fma2(a.hi, b, m);
    e = fma2(a.lo, b, e);
    const pair_t s = sub2(e, m);
    return f2x2{s, sub2(e, add2(s, m))};
}
__device__ __forceinline__ f2x2 df_mul_fc(f2x2 a, pair_t neg_ahi, pair_t b) {   // a constant
    const pair_t m = mul2(neg_ahi, b);
    pair_t e = fma2(a.hi, b, m);
    e = fma2(a.lo, b, e);
    const pair_t s = sub2(e, m);
    return f2x2{s, sub2(e, add2(s, m))};
}
__device__ __forceinline__ f2x2 df_mul(f2x2 a, pair_t neg_ahi, f2x2 b) {
    const pair_t m = mul2(neg_ahi, b.hi);
    pair_t e = fma2(a.hi, b.hi, m);
    e = fma2(a.hi, b.lo, e);
    e = fma2(a.lo, b.hi, e);
    const pair_t s = sub2(e, m);
    return f2x2{s, sub2(e, add2(s, m))};
}

// Sums of addends given as exact pairs: acc_add of df32.cuh, one accumulator
// per half.
struct AccPair {
    f2x2 hi;
    pair_t lo;
};
__device__ __forceinline__ AccPair accp_zero() { return AccPair{{0ull, 0ull}, 0ull}; }
__device__ __forceinline__ void acc_add(AccPair &a, f2x2 v) {
    a.hi = df_add_f(a.hi, v.hi);
    a.lo = add2(a.lo, v.lo);
}
__device__ __forceinline__ double acc_val(const AccPair &a) {
    float h0, h1, l0, l1, r0, r1;
    upk(a.hi.hi, h0, h1);
    upk(a.hi.lo, l0, l1);
    upk(a.lo, r0, r1);
    return acc_val(f2{h0, l0}, r0) + acc_val(f2{h1, l1}, r1);
}
// v * v/2 as an exact pair sum
__device__ __forceinline__ f2x2 half_square(pair_t v) {
    const pair_t h = mul2(v, pk1(0.5f));
    const pair_t p = mul2(v, h);
    return f2x2{p, fma2(v, h, mul2(p, pk1(-1.0f)))};
}

// g(y) = log(1 + e^-y) of two double-floats y >= 0: log1pexp_neg (df32.cuh),
// the same operations on the same table, here in shared memory.  The
// double-float steps run on pairs; the FP32 series stays scalar, where its
// constants are immediate operands and cost no registers.
__device__ __forceinline__ f2x2 log1pexp_neg(f2x2 y, const float4 *tab) {
    float y0, y1;
    upk(y.hi, y0, y1);
    // round y 2^5 to the nearest integer by adding 1.5 * 2^23; the sum's bits
    // hold the table index.  y >= 36 (and NaN) is clamped here, set below.
    const float big = 12582912.0f;
    const float b0 = fminf(y0 * (float)LOG1PEXP_PER_UNIT, (float)LOG1PEXP_K) + big;
    const float b1 = fminf(y1 * (float)LOG1PEXP_PER_UNIT, (float)LOG1PEXP_K) + big;
    const float4 q0 = tab[__float_as_int(b0) - __float_as_int(big)];
    const float4 q1 = tab[__float_as_int(b1) - __float_as_int(big)];
    // y.hi - y_k is exact (Sterbenz), the low word carries the rest
    const f2x2 d = two_sum(pk(fmaf(b0 - big, -1.0f / LOG1PEXP_PER_UNIT, y0),
                              fmaf(b1 - big, -1.0f / LOG1PEXP_PER_UNIT, y1)), y.lo);
    const pair_t m1 = pk1(-1.0f);
    const pair_t sh = pk(q0.z, q1.z), sl = pk(q0.w, q1.w), nd = mul2(d.hi, m1);
    // -s d
    const pair_t m = mul2(sh, d.hi);
    pair_t e = fma2(sh, nd, m);
    e = fma2(sh, mul2(d.lo, m1), e);
    e = fma2(sl, nd, e);
    const pair_t t = sub2(e, m);
    const f2x2 t1{t, sub2(e, add2(t, m))};
    float dh0, dh1;
    upk(d.hi, dh0, dh1);
    auto series = [](float sf, float dh) {   // second to sixth order
        const float wf = fmaf(-sf, sf, sf), vf = fmaf(-2.0f, sf, 1.0f);
        const float c2 = 0.5f * wf;
        const float c3 = -wf * vf * (1.0f / 6.0f);
        const float c4 = wf * fmaf(-6.0f, wf, 1.0f) * (1.0f / 24.0f);
        const float c5 = -wf * vf * fmaf(-12.0f, wf, 1.0f) * (1.0f / 120.0f);
        const float c6 = wf * fmaf(wf, fmaf(120.0f, wf, -30.0f), 1.0f) * (1.0f / 720.0f);
        const float r = fmaf(dh, fmaf(dh, fmaf(dh, fmaf(dh, c6, c5), c4), c3), c2);
        return dh * dh * r;
    };
    f2x2 g = df_add_q(f2x2{pk(q0.x, q1.x), pk(q0.y, q1.y)},
                      df_add_f(t1, pk(series(q0.z, dh0), series(q1.z, dh1))));
    if (!(y0 < 36.0f && y1 < 36.0f)) {   // rare: |x| of 18 and more
        float h0, h1, l0, l1;
        upk(g.hi, h0, h1);
        upk(g.lo, l0, l1);
        if (y0 >= 36.0f) { h0 = __expf(-y0); l0 = 0.0f; }
        if (y1 >= 36.0f) { h1 = __expf(-y1); l1 = 0.0f; }
        g = f2x2{pk(h0, h1), pk(l0, l1)};
    }
    return g;
}

// Action terms of two sites, 1/2 psi a - |x| - log(1 + e^-2|x|), x = a + h'.
__device__ __forceinline__ f2x2 action_term(pair_t psi, f2x2 a, f2x2 x, const float4 *tab) {
    // |x|: the sign of the high word taken off both words
    float x0, x1, w0, w1;
    upk(x.hi, x0, x1);
    upk(x.lo, w0, w1);
    const uint32_t s0 = __float_as_uint(x0) & 0x80000000u, s1 = __float_as_uint(x1) & 0x80000000u;
    const f2x2 ax{pk(fabsf(x0), fabsf(x1)), pk(__uint_as_float(__float_as_uint(w0) ^ s0),
                                               __uint_as_float(__float_as_uint(w1) ^ s1))};
    const pair_t two = pk1(2.0f);
    const f2x2 g = log1pexp_neg(f2x2{mul2(ax.hi, two), mul2(ax.lo, two)}, tab);
    return df_sub_q(df_mul_f(a, mul2(psi, pk1(0.5f)), mul2(psi, pk1(-0.5f))), df_add_q(ax, g));
}

// Sums of two pairs of addends per step: column by column (two accumulator
// pairs) or, in the order of the four values, into one scalar accumulator --
// whichever the thread's columns had in the plane-streaming kernel, so that
// its partial sums are the same to the bit.
template <bool COLUMNS>
struct AccRow;
template <>
struct AccRow<true> {
    AccPair p[2];
    __device__ __forceinline__ void clear() { p[0] = p[1] = accp_zero(); }
    __device__ __forceinline__ void add(f2x2 a, f2x2 b) {
        acc_add(p[0], a);
        acc_add(p[1], b);
    }
    __device__ __forceinline__ double value() const { return acc_val(p[0]) + acc_val(p[1]); }
};
template <>
struct AccRow<false> {
    f2 hi;
    float lo;
    __device__ __forceinline__ void clear() {
        hi = f2{0.0f, 0.0f};
        lo = 0.0f;
    }
    __device__ __forceinline__ void add(f2 v) { acc_add(hi, lo, v); }
    __device__ __forceinline__ double value() const { return acc_val(hi, lo); }
};
__device__ __forceinline__ void upk(f2x2 v, f2 &a, f2 &b) {
    upk(v.hi, a.hi, b.hi);
    upk(v.lo, a.lo, b.lo);
}

}  // namespace ihmc
