// Double-float values for the FP32 pipe: a value is the unevaluated sum hi + lo of two
// floats with |lo| <= ulp(hi)/2, about 48 significant bits.  GB300 issues FP32 64
// times as fast as FP64, so the block chains of the streamfunction solve, strings of
// dependent sums that an FP64 refinement follows, run in this form (their sums are
// beside them, in k_implicit.cu); here are the type and its conversions.
//
// Error-free transformation used (fast two-sum, Dekker 1971), |a| >= |b|:
// s = a + b,  e = b - (s - a),  a + b = s + e exactly.
// Range: that of float (|x| < 3.4e38; below ~1e-38 the trailing part loses bits).
// The _rn intrinsics are never contracted into fused multiply-adds: the
// transformation relies on each operation being rounded on its own.
#pragma once
#include <cuda_runtime.h>

namespace pz {

struct __align__(8) ddf {
    float hi, lo;
};
struct __align__(16) ddc {
    ddf x, y;
};

__device__ __forceinline__ ddf dd_renorm(float s, float e) {
    const float h = __fadd_rn(s, e);
    return ddf{h, __fsub_rn(e, __fsub_rn(h, s))};
}
// Conversions taken apart on the IEEE 754 fields with integer and FP32 instructions: on
// GB300 one between float and double issues on the FP64 unit (2 per clock per SM).
//
// v = (-1)^s 1.f 2^e (52 fraction bits f) splits into h = the first 24
// significant bits (truncated) and the remainder r 2^(e-52), r = the low 29 bits
// of f, rounded to a float; one fast two-sum renormalises (|h| >= |r 2^(e-52)|).
// The pair holds v to 2^-48 relative.  |v| below float's normal range gives a
// signed zero, |v| above it (and inf, NaN) a signed infinity.
__device__ __forceinline__ ddf dd_from_bits(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const unsigned hw = (unsigned)(u >> 32), lw = (unsigned)u;
    const unsigned sign = hw & 0x80000000u;
    const int E = (int)((hw >> 20) & 0x7ffu) - 896;  // biased float exponent of 2^e
    if (E <= 0) return ddf{__uint_as_float(sign), 0.f};
    if (E >= 255) return ddf{__uint_as_float(sign | 0x7f800000u), 0.f};
    const float h = __uint_as_float(sign | ((unsigned)E << 23) | ((hw & 0xfffffu) << 3) | (lw >> 29));
    // r = 64 (r >> 6) + (r & 63), both parts exact floats by the 2^23 offset
    const unsigned r = lw & 0x1fffffffu;
    const float r1 = __fsub_rn(__uint_as_float(0x4b000000u | (r >> 6)), 8388608.f);
    const float r0 = __fsub_rn(__uint_as_float(0x4b000000u | (r & 63u)), 8388608.f);
    const float rf = __fmul_rn(__fmaf_rn(r1, 64.f, r0), 2.220446049250313e-16f);  // r 2^-52
    const float l = __fmul_rn(rf, __uint_as_float((unsigned)E << 23));          // times 2^e
    return dd_renorm(h, __uint_as_float(__float_as_uint(l) ^ sign));
}

// a float as the double of the same value (exact); subnormal floats give zero
__device__ __forceinline__ double f2d_bits(float f) {
    const unsigned b = __float_as_uint(f);
    const unsigned e = (b >> 23) & 0xffu, sign = b & 0x80000000u;
    const unsigned ed = (e == 0xffu) ? 0x7ffu : e + 896u;
    const unsigned hw = (e == 0u) ? sign : sign | (ed << 20) | ((b & 0x7fffffu) >> 3);
    const unsigned lw = (e == 0u) ? 0u : b << 29;
    return __hiloint2double((int)hw, (int)lw);
}
// the float nearest v (ties away from zero), by an integer rounding of the
// fraction; below float's normal range a signed zero, above it a signed infinity
__device__ __forceinline__ float f32_from_bits(double v) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(v);
    const unsigned hw = (unsigned)(u >> 32), lw = (unsigned)u;
    const unsigned sign = hw & 0x80000000u;
    const int E = (int)((hw >> 20) & 0x7ffu) - 896;
    if (E <= 0) return __uint_as_float(sign);
    if (E >= 255) return __uint_as_float(sign | 0x7f800000u);
    // exponent and leading 23 fraction bits (mod 2^32), plus the rounding bit;
    // a carry out of the fraction steps the exponent, as rounding does
    unsigned t = ((hw << 3) | (lw >> 29)) - (896u << 23);
    t = (t & 0x7fffffffu) + ((lw >> 28) & 1u);
    return __uint_as_float(sign | min(t, 0x7f800000u));
}

// hi + lo rounded to double: one FP64 add
__device__ __forceinline__ double dd_to_bits(ddf a) { return f2d_bits(a.hi) + f2d_bits(a.lo); }

// hi + lo as a double with integer instructions only.  hi widened to double
// leaves 29 zero fraction bits below its 24; a renormalised lo (|lo| <= ulp(hi)/2,
// exponent at least 24 below hi's) is lo's significand shifted into them
// (truncated past the double's last place), added to the bit pattern when the
// signs agree and subtracted otherwise, at twice the shift when hi is a power of
// two (the difference then lies in the binade below).  Within one unit in the
// last place of the double nearest hi + lo; a subnormal lo counts as zero.
__device__ __forceinline__ double dd_compose(ddf a) {
    const unsigned hb = __float_as_uint(a.hi), lb = __float_as_uint(a.lo);
    const unsigned eh = (hb >> 23) & 0xffu, el = (lb >> 23) & 0xffu;
    if (eh == 0u || eh == 0xffu || el == 0u) return f2d_bits(a.hi);
    const int sh = 29 - (int)(eh - el);
    if (sh > 5) return dd_to_bits(a);  // not a renormalised pair
    const unsigned ml = (lb & 0x7fffffu) | 0x800000u;
    const unsigned L = (sh >= 0) ? (ml << sh) : ((sh > -24) ? (ml >> -sh) : 0u);
    unsigned long long H =
        ((unsigned long long)(((eh + 896u) << 20) | ((hb & 0x7fffffu) >> 3)) << 32) | (unsigned long long)(hb << 29);
    if ((hb ^ lb) & 0x80000000u)
        H -= ((hb & 0x7fffffu) == 0u) ? 2ull * L : (unsigned long long)L;
    else
        H |= L;
    return __longlong_as_double((long long)(H | ((unsigned long long)(hb & 0x80000000u) << 32)));
}

}  // namespace pz
