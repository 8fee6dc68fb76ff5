// df.cuh -- "double-float" arithmetic: a value carried as the unevaluated sum
// hi + lo of two floats (about 44-48 significant bits), built from the
// error-free transformations two-sum (Knuth) and fused multiply-add products.
// Every float operation is written with the _rn intrinsics so that the compiler
// cannot contract or reorder it (the error terms depend on exact rounding).
#pragma once

namespace cplbm {

struct df {
    float hi, lo;
};

__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
__device__ __forceinline__ df quick_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ df df_add(df x, df y) {
    const df s = two_sum(x.hi, y.hi);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(x.lo, y.lo)));
}
__device__ __forceinline__ df df_sub(df x, df y) { return df_add(x, df{-y.hi, -y.lo}); }
__device__ __forceinline__ df df_add_f(df x, float y) {
    const df s = two_sum(x.hi, y);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, x.lo));
}
// x * c for DF x and DF c (products by fmaf are exact error terms)
__device__ __forceinline__ df df_mul(df x, float ch, float cl) {
    const float p = __fmul_rn(x.hi, ch);
    float e = fmaf(x.hi, ch, -p);
    e = fmaf(x.hi, cl, e);
    e = fmaf(x.lo, ch, e);
    return quick_two_sum(p, e);
}
__device__ __forceinline__ float df_round(df x) { return __fadd_rn(x.hi, x.lo); }

// x * c + y with the product left unnormalised before the sum (one
// renormalisation instead of two; same error bound to within a unit).
__device__ __forceinline__ df df_fma(df x, float ch, float cl, df y) {
    const float p = __fmul_rn(x.hi, ch);
    float e = fmaf(x.hi, ch, -p);
    e = fmaf(x.hi, cl, e);
    e = fmaf(x.lo, ch, e);
    const df s = two_sum(p, y.hi);
    return quick_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(e, y.lo)));
}

// Exact sum of nine positive floats as a double-float, for populations whose
// largest member is normally f[0]: accumulating from f[0] with the exact
// a + b = s + e split (valid when |running sum| >= |addend|, so exact here
// whenever f[0] is the largest; otherwise an error of at most one unit of the
// low part).
__device__ __forceinline__ df sum9_exact(const float g[9]) {
    float s = g[0], e = 0.0f;
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const float t = __fadd_rn(s, g[i]);
        e = __fadd_rn(e, __fsub_rn(g[i], __fsub_rn(t, s)));
        s = t;
    }
    return quick_two_sum(s, e);
}

// A float as a double, by integer operations: the conversion instruction runs on the
// FP64 pipe (2 lanes a clock and SM).  Zeros and subnormals, infinities and NaN take it.
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = u & 0x7fffffffu;
    if (e - 0x00800000u >= 0x7f000000u) return e == 0 ? __hiloint2double((int)u, 0) : (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | ((e >> 3) + 0x38000000u)), (int)(u << 29));
}

// Unevaluated sum of three floats: about 72 significant bits, more than a double's 53.
struct tf {
    float a, b, c;
};
__device__ __forceinline__ void tf_add(tf& s, float x) {
    const df h = two_sum(s.a, x), l = two_sum(s.b, h.lo);
    s.a = h.hi;
    s.b = l.hi;
    s.c = __fadd_rn(s.c, l.lo);
}
// n / r to about 68 bits, rounded once to double: three quotient digits of one float
// each, the remainder after the first kept as hi + lo.  inv: 1 / r.hi to a float's
// accuracy.  The digits' products reach 72 bits below the operands and need room in a
// float's range: operands outside it (the gas at reduced temperatures below 0.13) are first
// brought to about one by powers of 2^64, and the quotient's exponent is put back.
__device__ __forceinline__ double tf_div(tf n, df r, float inv) {
    df s = quick_two_sum(n.a, n.b);  // normalised: the head holds a float's accuracy
    int k = 0;                       // the quotient's exponent, in units of 64
    const float size = fabsf(s.hi);
    if (!(r.hi >= 0x1p-60f && r.hi <= 0x1p8f && size <= 0x1p32f &&
          (size >= 0x1p-84f || size == 0.0f))) {
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {  // (zero, infinite and NaN ones stay what they are)
            const float a = fabsf(r.hi), b = fabsf(s.hi);
            const int kr = a < 0x1p-32f ? 1 : (a > 0x1p32f ? -1 : 0);
            const int kn = b < 0x1p-32f ? 1 : (b > 0x1p32f ? -1 : 0);
            const float fr = __int_as_float((127 + 64 * kr) << 23);
            const float fn = __int_as_float((127 + 64 * kn) << 23);
            r.hi = __fmul_rn(r.hi, fr);
            r.lo = __fmul_rn(r.lo, fr);
            s.hi = __fmul_rn(s.hi, fn);
            s.lo = __fmul_rn(s.lo, fn);
            n.c = __fmul_rn(n.c, fn);
            k += kr - kn;
        }
        inv = __frcp_rn(r.hi);
    }
    const float q0 = __fmul_rn(s.hi, inv);
    const float p = __fmul_rn(q0, r.hi), t = __fmul_rn(q0, r.lo);
    float lo = __fsub_rn(n.c, fmaf(q0, r.lo, -t));
    df m = two_sum(__fsub_rn(s.hi, p), -fmaf(q0, r.hi, -p));
    lo = __fadd_rn(lo, m.lo);
    m = two_sum(m.hi, s.lo);
    lo = __fadd_rn(lo, m.lo);
    m = two_sum(m.hi, -t);
    lo = __fadd_rn(lo, m.lo);
    const float q1 = __fmul_rn(__fadd_rn(m.hi, lo), inv);
    const float p1 = __fmul_rn(q1, r.hi);
    float rem = __fsub_rn(m.hi, p1);
    rem = __fsub_rn(rem, fmaf(q1, r.hi, -p1));
    rem = __fadd_rn(rem, fmaf(-q1, r.lo, lo));
    const float q2 = __fmul_rn(rem, inv);
    const double q = __dadd_rn(widen(q0), __dadd_rn(widen(q1), widen(q2)));
    // (a NaN keeps its exponent: its high word has bits 19 to 30 set)
    const unsigned hi = (unsigned)__double2hiint(q);
    return k == 0 || q == 0.0 || (~hi & 0x7ff80000u) == 0u
               ? q
               : __hiloint2double((int)hi + k * (64 << 20), __double2loint(q));
}

}  // namespace cplbm
