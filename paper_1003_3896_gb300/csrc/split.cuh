// split.cuh -- double-single split of a double (the paper's hi + lo
// coordinate format, Sect. 5.2) from its bits, the widening of a float from
// its bits, and inverse square-root powers in double refined from a float
// estimate: arithmetic kept off the FP64 pipe, which on this GPU runs at 1/77
// of the FP32 rate.
#pragma once

namespace nb {

// Double-single split of r: hi = RN_float(r), lo = RN_float(r - hi), taken
// from the bits of r with integer operations.  r = S 2^(E - 1075) with the
// 53-bit significand S; hi keeps the top 24 bits of S rounded to nearest
// even, and r - hi = d 2^(E - 1075) exactly, d = S - q 2^29 with |d| <= 2^28,
// whose float rounding is lo.  Equal bit for bit to the plain conversions
// for 2^-70 <= |r| < 2^101 (hi and lo normal floats); other r (zero, tiny,
// huge, non-finite) take the plain conversions.  The FP64 pipe, which runs at
// 1/77 of the FP32 rate here, otherwise carries three conversions and a
// subtraction per coordinate.
__device__ __forceinline__ void split_ds(double r, float &hi, float &lo)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(r);
    const int E = (int)((b >> 52) & 0x7FF);
    if (E < 1023 - 70 || E > 1023 + 100) {
        hi = __double2float_rn(r);
        lo = __double2float_rn(r - (double)hi);
        return;
    }
    const unsigned long long S = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    unsigned int q = (unsigned int)(S >> 29);   // 24 bits, truncated
    const unsigned int rem = (unsigned int)(S & 0x1FFFFFFFu);
    const bool up = rem > 0x10000000u || (rem == 0x10000000u && (q & 1u));
    q += up ? 1u : 0u;
    const int d = (int)rem - (up ? 0x20000000 : 0);
    int ef = E - 1023 + 127;
    if (q == (1u << 24)) {   // rounding carried into the exponent
        q >>= 1;
        ++ef;
    }
    const unsigned int sign = (unsigned int)(b >> 63) << 31;
    hi = __int_as_float((int)(sign | ((unsigned int)ef << 23) | (q & 0x7FFFFFu)));
    const float scale = __int_as_float((E - 1075 + 127) << 23);   // 2^(E - 1075)
    lo = __fmul_rn(__int2float_rn(sign ? -d : d), scale);
}

// The double equal to float f, from its bits: the exponent rebiased, the
// fraction shifted into place (exact).  Zeros come from the sign bit alone;
// subnormal and non-finite f take the conversion instruction, which on this
// GPU runs on the FP64 pipe.
__device__ __forceinline__ double widen(float f)
{
    const unsigned int u = __float_as_uint(f);
    const unsigned int e = (u >> 23) & 0xFFu;
    if (e == 0u || e == 0xFFu) {
        if ((u & 0x7FFFFFFFu) == 0u)
            return __longlong_as_double((long long)((unsigned long long)u << 32));
        return (double)f;
    }
    const unsigned long long b = ((unsigned long long)(u & 0x80000000u) << 32) |
                                 ((unsigned long long)(e + 896u) << 52) |
                                 ((unsigned long long)(u & 0x7FFFFFu) << 29);
    return __longlong_as_double((long long)b);
}

// R^(-1/2) (POT) or R^(-3/2) in double for R >= 0, refined from the float
// estimate rsqrt.approx(R_f), R_f being R truncated to float from its bits.
// The FP64 pipe bounds the kernels that call this (2 lanes per SM clock), so it
// does three operations there and the rest goes to the integer and float pipes:
//   y0   the estimate rounded to 17 bits, y0 = M 2^k; then M^2 and M^3 are
//        integers of at most 34 and 51 bits, and y0^2 and y0^3 doubles built
//        from them exactly;
//   v    1 - R y0^2, one fused multiply-add: |v| < 2^-15.9, exact to 2^-69;
//   m    R^(-1/2) = y0 (1 + m), m = v / 2 + v^2 (3/8 + 5/16 v + O(v^2)), or
//        R^(-3/2) = y0^3 (1 + m), m = 3 v / 2 + v^2 (15/8 + 35/16 v + O(v^2)): the
//        dropped terms are below 2^-62, and the v^2 term, below 2^-30.8, needs
//        only float precision.
// Within 1.1 and 1.4 units of 2^-53 of the exact powers (emulated).  The form with
// y0 to 24 bits and its powers and the whole series in double takes five and six
// operations and is within 1.5 and 3.3 units: N = 16384 FP64 evaluation 4.65 ms
// with it, 3.83 with this one; energy of N = 32768 11.8 and 9.7 ms.  R outside the
// float range (the padding's 1e300, R = 0, non-finite R) takes the library rsqrt.
template <bool POT>
__device__ __forceinline__ double rsqrt_pow(double R)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(R);
    const int E = (int)(b >> 52);   // R >= 0: the sign bit is clear
    if (E < 1023 - 125 || E > 1023 + 126) {
        const double ri = rsqrt(R);
        return POT ? ri : ri * ri * ri;
    }
    const float rf = __int_as_float(((E - 1023 + 127) << 23) | (int)((b >> 29) & 0x7FFFFFu));
    float yf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(rf));
    const unsigned int yr = (__float_as_uint(yf) + 0x40u) & ~0x7Fu;   // 17 bits, to nearest
    const unsigned int M = ((yr >> 7) & 0xFFFFu) | 0x10000u;          // y0 = M 2^(ey - 143)
    const int ey = (int)(yr >> 23);
    // y0^2: the leading bit of M^2 is 32 or 33
    const unsigned long long P = (unsigned long long)M * M;
    const int s2 = (int)(P >> 33);
    const unsigned long long qb =
        (P << (20 - s2)) + ((unsigned long long)(2 * ey + 768 + s2) << 52);
    const double v = __fma_rn(-R, __longlong_as_double((long long)qb), 1.0);
    // v to float from its bits: v = 0 or 2^-90 < |v| < 2^-15 (its exponent field
    // is 0x380 to 0x3FF, whose low seven bits are the float's)
    const unsigned int vh = (unsigned int)((unsigned long long)__double_as_longlong(v) >> 32);
    const unsigned int vl = (unsigned int)__double_as_longlong(v);
    const unsigned int vt = __funnelshift_l(vl, vh, 3);
    const float vf = __uint_as_float((vt & 0x3FFFFFFFu) | (vh & ~0x3FFFFFFFu));
    const float w = __fmul_rn(__fmul_rn(vf, vf), POT ? __fmaf_rn(vf, 0.3125f, 0.375f)
                                                     : __fmaf_rn(vf, 2.1875f, 1.875f));
    // w >= 0 to double from its bits (0 gives 2^-127, of no effect)
    const unsigned long long wb =
        ((unsigned long long)__float_as_uint(w) << 29) + ((unsigned long long)896 << 52);
    const double m = __fma_rn(POT ? 0.5 : 1.5, v, __longlong_as_double((long long)wb));
    unsigned long long yb;
    if (POT) {
        yb = ((unsigned long long)yr << 29) + ((unsigned long long)896 << 52);
    } else {
        // y0^3: the leading bit of M^3 is 48, 49 or 50
        const unsigned long long Q = P * M;
        const int lz = __clz((int)(Q >> 32));   // 15, 14 or 13
        yb = (Q << (lz - 11)) + ((unsigned long long)(3 * ey + 656 - lz) << 52);
    }
    const double y = __longlong_as_double((long long)yb);
    return __fma_rn(y, m, y);
}

}  // namespace nb
