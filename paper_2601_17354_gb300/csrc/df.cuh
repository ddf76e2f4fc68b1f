// Arithmetic on unevaluated sums of two floats.
#pragma once

namespace pgs {

// Unevaluated sums of two floats (about 47 bits), by the error-free transformations of Dekker (1971) and
// Knuth (TAOCP 2, 4.2.2).  GB300 runs FP64 at 1/64 of its FP32 rate, so what needs more than 24 bits on many
// threads is kept this way.  Every operation is an explicitly rounded intrinsic, so neither contraction
// nor reordering touches them.
struct Df {
    float h, l;
};
__device__ __forceinline__ Df df_fast(float a, float b) {  // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return {s, __fadd_rn(b, -__fadd_rn(s, -a))};
}
__device__ __forceinline__ Df df_two(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fadd_rn(s, -a);
    return {s, __fadd_rn(__fadd_rn(a, -__fadd_rn(s, -bb)), __fadd_rn(b, -bb))};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
    const Df s = df_two(a.h, b.h), t = df_two(a.l, b.l);
    const Df u = df_fast(s.h, __fadd_rn(s.l, t.h));
    return df_fast(u.h, __fadd_rn(u.l, t.l));
}
__device__ __forceinline__ Df df_neg(Df a) { return {-a.h, -a.l}; }
__device__ __forceinline__ Df df_sub(Df a, Df b) { return df_add(a, df_neg(b)); }
__device__ __forceinline__ Df df_mul(Df a, Df b) {
    const float p = __fmul_rn(a.h, b.h);
    return df_fast(p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p))));
}
__device__ __forceinline__ Df df_scale(Df a, float f) { return {__fmul_rn(a.h, f), __fmul_rn(a.l, f)}; }  // f a power of two
// a / b rounded to FP32 (both normalised); a zero divisor gives what a.h / b.h gives
__device__ __forceinline__ float df_ratio(Df a, Df b) {
    const float q = a.h / b.h;
    if (!isfinite(q)) return q;
    const float r = __fadd_rn(__fmaf_rn(-q, b.h, a.h), __fmaf_rn(-q, b.l, a.l));
    return __fadd_rn(q, r / b.h);
}
__device__ __forceinline__ Df df_from(double a) {
    const float h = (float)a;
    return {h, (float)(a - (double)h)};
}
__device__ __forceinline__ double df_double(Df a) { return (double)a.h + (double)a.l; }
// sqrt(x), x >= 0, and 1 / x to about 45 bits
__device__ __forceinline__ Df df_sqrt(Df x) {
    if (!(x.h > 0.0f)) return {x.h, 0.0f};
    const float r = __fsqrt_rn(x.h);
    const float e = __fadd_rn(__fmaf_rn(-r, r, x.h), x.l);
    return df_fast(r, __fdividef(0.5f * e, r));
}
__device__ __forceinline__ Df df_recip(Df x) {
    const float r = __frcp_rn(x.h);
    return df_fast(r, __fmul_rn(r, __fmaf_rn(-x.l, r, __fmaf_rn(-x.h, r, 1.0f))));
}
// |(x, y, z)|
__device__ __forceinline__ Df df_norm(Df x, Df y, Df z) {
    const float a = __fmul_rn(x.h, x.h), b = __fmul_rn(y.h, y.h), c = __fmul_rn(z.h, z.h);
    const Df s = df_two(a, b), t = df_two(s.h, c);
    float e = __fadd_rn(__fadd_rn(__fmaf_rn(x.h, x.h, -a), __fmaf_rn(y.h, y.h, -b)), __fmaf_rn(z.h, z.h, -c));
    const float l = __fmaf_rn(x.h, x.l, __fmaf_rn(y.h, y.l, __fmul_rn(z.h, z.l)));
    e = __fadd_rn(__fmaf_rn(2.0f, l, e), __fadd_rn(s.l, t.l));
    return df_sqrt(df_fast(t.h, e));
}
// sums whose low parts stay unnormalised until the end
__device__ __forceinline__ void df_acc(Df& s, Df v) {
    const Df t = df_two(s.h, v.h);
    s.h = t.h;
    s.l = __fadd_rn(__fadd_rn(s.l, v.l), t.l);
}
__device__ __forceinline__ void df_acc(Df& s, float v) { df_acc(s, Df{v, 0.0f}); }
// one product-sum step: acc += a b, acc kept as a sum and the lost parts' sum (normalised by the caller)
__device__ __forceinline__ void df_dot(Df& acc, Df a, Df b) {
    const float p = __fmul_rn(a.h, b.h);
    const float e = __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)));
    const Df s = df_two(acc.h, p);
    acc.h = s.h;
    acc.l = __fadd_rn(acc.l, __fadd_rn(s.l, e));
}

}  // namespace pgs
