// Unevaluated sums of two binary32 numbers (hi + lo, 48 significant bits) on the FP32 pipe.
//
// GB300 issues one warp-wide FP64 instruction per 16 cycles and SM quarter, so a stencil in binary64
// is bound by that pipe; in split form it is about 10 FP32 operations per neighbour and bound by
// memory.  The error-free transformations are Knuth's TwoSum (The Art of Computer Programming, vol. 2,
// 4.2.2) and Dekker's FastTwoSum (Numerische Mathematik 18, 1971), and the product's error is one
// fma.  They hold for round-to-nearest without intermediate overflow.
#pragma once

namespace emfuse {

struct alignas(8) Split {
    float hi, lo;  // hi = the value rounded to binary32
};

// s + e = a + b exactly, s = fl(a + b)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
}

// d + x
__device__ __forceinline__ Split split_add(Split d, float x) {
    float s, e;
    two_sum(d.hi, x, s, e);
    e = __fadd_rn(e, d.lo);
    Split r;
    r.hi = __fadd_rn(s, e);
    r.lo = __fadd_rn(__fsub_rn(s, r.hi), e);
    return r;
}

// a c - (s + lo), rounded once to binary32 at the end: sums and products before it carry their
// errors (lo collects those of the sum s), so what is lost is about 2^-46 of the largest term.
__device__ __forceinline__ float split_finish(Split a, Split c, float s, float lo) {
    const float p = __fmul_rn(a.hi, c.hi);
    float pe = __fmaf_rn(a.hi, c.hi, -p);
    pe = __fmaf_rn(a.hi, c.lo, pe);
    pe = __fmaf_rn(a.lo, c.hi, pe);
    float t, te;
    two_sum(p, -s, t, te);
    return __fadd_rn(t, __fadd_rn(te, __fsub_rn(pe, lo)));
}

}  // namespace emfuse
