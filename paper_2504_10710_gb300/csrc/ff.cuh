// Float-float arithmetic: a value is the unevaluated sum hi + lo of two FP32
// numbers, |lo| <= ulp(hi) / 2 after normalisation: about 48 significant bits
// within the FP32 exponent range.  Built from two error-free transformations:
// Knuth's two-sum (The Art of Computer Programming, vol. 2, 4.2.2, Theorem B)
// and the exact product a b = p + e with e = fma(a, b, -p) (Dekker 1971 wrote
// the product without an FMA; with one the error term is a single rounding-
// free operation).  The _rn intrinsics are never contracted or reassociated
// by the compiler, which the transformations rely on.
#pragma once
#include "f32x2.cuh"

namespace glls {

struct __align__(8) ffloat {   // 8-byte aligned: one 64-bit shared-memory access per value
    float hi, lo;
};

__device__ __forceinline__ ffloat ff_from_double(double x) {
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - (double)hi)};
}

__device__ __forceinline__ double ff_to_double(ffloat a) { return (double)a.hi + (double)a.lo; }

// s + e = a + b exactly (Knuth's two-sum: no condition on |a|, |b|)
__device__ __forceinline__ void ff_two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// hi + lo rewritten with |lo| <= ulp(hi) / 2 (the fast two-sum, valid when
// |hi| >= |lo| or hi = 0)
__device__ __forceinline__ ffloat ff_norm(ffloat a) {
    const float s = __fadd_rn(a.hi, a.lo);
    return {s, __fsub_rn(a.lo, __fsub_rn(s, a.hi))};
}

// acc += a b for float-float a, b.  The exact product of the high parts plus
// the two cross terms (a.lo b.lo is below the format's precision); the sum's
// rounding error and the product's low part are collected in acc.lo, which
// is left unnormalised (a few terms in a row stay well inside its headroom).
__device__ __forceinline__ void ff_mac(ffloat& acc, ffloat a, ffloat b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = __fmaf_rn(a.hi, b.hi, -p);
    e = __fmaf_rn(a.hi, b.lo, e);
    e = __fmaf_rn(a.lo, b.hi, e);
    float s, es;
    ff_two_sum(acc.hi, p, s, es);
    acc.hi = s;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(es, e));
}

// a + b and a - b, normalised
__device__ __forceinline__ ffloat ff_add(ffloat a, ffloat b) {
    float s, e;
    ff_two_sum(a.hi, b.hi, s, e);
    return ff_norm({s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))});
}
__device__ __forceinline__ ffloat ff_sub(ffloat a, ffloat b) { return ff_add(a, {-b.hi, -b.lo}); }

// ---- two float-float values in the halves of FP32 pairs --------------------
// Every operation does to each half what the scalar one above does, in the
// same order, so the halves carry the same bits.
struct ffloat2 {
    f32x2 hi, lo;
};

__device__ __forceinline__ ffloat2 ff_pack(ffloat a, ffloat b) { return {pack2(a.hi, b.hi), pack2(a.lo, b.lo)}; }
__device__ __forceinline__ void ff_unpack(ffloat2 p, ffloat& a, ffloat& b) {
    unpack2(p.hi, a.hi, b.hi);
    unpack2(p.lo, a.lo, b.lo);
}
__device__ __forceinline__ ffloat ff_neg(ffloat a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ ffloat2 ff_norm(ffloat2 a) {
    const f32x2 s = add2(a.hi, a.lo);
    return {s, sub2(a.lo, sub2(s, a.hi))};
}

__device__ __forceinline__ ffloat2 ff_add(ffloat2 a, ffloat2 b) {
    const f32x2 s = add2(a.hi, b.hi), bb = sub2(s, a.hi);
    const f32x2 e = add2(sub2(a.hi, sub2(s, bb)), sub2(b.hi, bb));
    return ff_norm(ffloat2{s, add2(e, add2(a.lo, b.lo))});
}

// acc += a b, nahi = -a.hi: the product is formed with its sign turned (m =
// -fl(a.hi b.hi), exact negation), so that its error term needs no negation.
__device__ __forceinline__ void ff_mac(ffloat2& acc, ffloat2 a, f32x2 nahi, ffloat2 b) {
    const f32x2 m = mul2(nahi, b.hi);
    f32x2 e = fma2(a.hi, b.hi, m);
    e = fma2(a.hi, b.lo, e);
    e = fma2(a.lo, b.hi, e);
    const f32x2 s = sub2(acc.hi, m), bb = sub2(s, acc.hi);
    const f32x2 es = sub2(sub2(acc.hi, sub2(s, bb)), add2(m, bb));
    acc.hi = s;
    acc.lo = add2(acc.lo, add2(es, e));
}

}  // namespace glls
