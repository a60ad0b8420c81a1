// arith.cuh -- the arithmetic the pair kernels share: the MUFU reciprocal
// square root, double-single accumulation, and float-float operations packed
// over two bodies per f32x2 instruction.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace nb {

__device__ __forceinline__ float rsqrt_mufu(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Add float t to the double-single number (hi, lo): Knuth's two-sum of hi and
// t, error folded into lo, then Dekker's fast two-sum to renormalise.
__device__ __forceinline__ void ds_add(float &hi, float &lo, float t)
{
    const float s = __fadd_rn(hi, t);
    const float bp = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(t, bp));
    const float l = __fadd_rn(lo, e);
    const float h = __fadd_rn(s, l);
    lo = __fsub_rn(l, __fsub_rn(h, s));
    hi = h;
}

// Add the float pair (p, e) to the float-float number (h, l): Knuth's
// two-sum of the high parts, the error and the low parts folded in, then
// Dekker's fast two-sum to renormalise.
__device__ __forceinline__ void ff_add(float &h, float &l, float p, float e)
{
    const float s = __fadd_rn(h, p);
    const float bp = __fsub_rn(s, h);
    const float err = __fadd_rn(__fadd_rn(__fsub_rn(h, __fsub_rn(s, bp)), __fsub_rn(p, bp)),
                                __fadd_rn(l, e));
    h = __fadd_rn(s, err);
    l = __fsub_rn(err, __fsub_rn(h, s));
}

__device__ __forceinline__ float2 f2neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return __fadd2_rn(a, f2neg(b)); }

// s + e = a + b exactly (Knuth).
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    const float2 bb = f2sub(s, a);
    e = __fadd2_rn(f2sub(a, f2sub(s, bb)), f2sub(b, bb));
}

// s + e = a + b exactly when |a| >= |b| (Dekker).
__device__ __forceinline__ void fast_two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    s = __fadd2_rn(a, b);
    e = f2sub(b, f2sub(s, a));
}

// s + e = a + b exactly for a, b >= 0: the larger operand first (max / min
// run on the ALU pipe, which this kernel leaves idle), then Dekker's fast
// two-sum, three FMA-pipe operations instead of Knuth's six.
__device__ __forceinline__ void pos_two_sum2(float2 a, float2 b, float2 &s, float2 &e)
{
    const float2 hi = make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y));
    const float2 lo = make_float2(fminf(a.x, b.x), fminf(a.y, b.y));
    s = __fadd2_rn(a, b);
    e = f2sub(lo, f2sub(s, hi));
}

// (ah + al) - (bh + bl), normalised.
__device__ __forceinline__ void ff_diff(float2 ah, float2 al, float2 bh, float2 bl, float2 &dh,
                                        float2 &dl)
{
    float2 s, e;
    two_sum2(ah, f2neg(bh), s, e);
    e = __fadd2_rn(e, f2sub(al, bl));
    fast_two_sum2(s, e, dh, dl);
}

// h^2 + (2 h l) as an unnormalised pair (p, e): p = fl(h^2), e its error plus
// the cross term.
__device__ __forceinline__ void ff_sq(float2 h, float2 l, float2 &p, float2 &e)
{
    p = __fmul2_rn(h, h);
    e = __ffma2_rn(h, h, f2neg(p));
    e = __ffma2_rn(__fadd2_rn(h, h), l, e);
}

// (ah + al)(bh + bl) without the al bl term, unnormalised.
__device__ __forceinline__ void ff_mul(float2 ah, float2 al, float2 bh, float2 bl, float2 &p,
                                       float2 &e)
{
    p = __fmul2_rn(ah, bh);
    e = __ffma2_rn(ah, bh, f2neg(p));
    e = __ffma2_rn(ah, bl, e);
    e = __ffma2_rn(al, bh, e);
}

// largest k in [0, K) with off[k] <= t
template <typename T>
__device__ __forceinline__ int32_t find_in(const T *off, int32_t K, int64_t t)
{
    int32_t lo = 0, hi = K;
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (off[mid] <= t) lo = mid; else hi = mid;
    }
    return lo;
}

}  // namespace nb
