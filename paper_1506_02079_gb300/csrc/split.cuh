// Unevaluated sums of two binary32 numbers (hi + lo, 48 significant bits) on the FP32 pipe.
//
// GB300 issues one warp-wide FP64 instruction per 16 cycles and SM quarter, so a stencil in binary64
// is bound by that pipe; in split form it is about 10 FP32 operations per neighbour and bound by
// memory.  The error-free transformations are Knuth's TwoSum (The Art of Computer Programming, vol. 2,
// 4.2.2) and Dekker's FastTwoSum (Numerische Mathematik 18, 1971), and the product's error is one
// fma.  They hold for round-to-nearest without intermediate overflow.
#pragma once

#include <stdint.h>

#include "fpconv.cuh"

namespace emfuse {

struct alignas(8) Split {
    float hi, lo;  // hi = the value rounded to binary32
};

// Integer-pipe split of a binary64 value (see fpconv.cuh for why no conversion instruction is
// used): hi = d rounded to binary32 (the value d2f_ieee returns), lo = the 29 bits below it, rounded
// to 24.  Values below 2^-74, whose rest is below binary32's normal range, and values beyond
// binary32 get lo = 0.
__device__ __forceinline__ Split split_of(double d) {
    const uint32_t hi = uint32_t(__double2hiint(d)), lo = uint32_t(__double2loint(d));
    const int e = int((hi >> 20) & 0x7ffu);
    Split r;
    if (e >= 949 && e <= 1149) {
        uint32_t bits = (uint32_t(e - 896) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
        const int m = int(lo & 0x1fffffffu);
        const int up = (m > 0x10000000 || (m == 0x10000000 && (bits & 1u))) ? 1 : 0;
        bits += uint32_t(up);
        const uint32_t sgn = hi & 0x80000000u;
        r.hi = __uint_as_float(sgn | bits);
        r.lo = __int2float_rn(m - (up << 29)) * __uint_as_float(sgn | (uint32_t(e - 948) << 23));
    } else {
        r.hi = d2f_ieee(d);
        r.lo = 0.f;
    }
    return r;
}

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

// a c - (w + e + n + s), rounded once to binary32.
__device__ __forceinline__ float split_apply(Split a, Split c, Split w, Split e, Split n, Split s) {
    float s1, e1, s2, e2, s3, e3;
    two_sum(w.hi, e.hi, s1, e1);
    two_sum(n.hi, s.hi, s2, e2);
    two_sum(s1, s2, s3, e3);
    return split_finish(a, c, s3, ((w.lo + e.lo) + (n.lo + s.lo)) + ((e1 + e2) + e3));
}

}  // namespace emfuse
