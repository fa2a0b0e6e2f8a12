// Sums of compensated float32 accumulators across the threads of a CTA in
// float-float arithmetic (an unevaluated sum hi + lo of two floats, about 48
// significant bits; Dekker 1971, Knuth's two-sum).
//
// Why not double: GB300's FP64 pipe is narrow (a warp-wide double add holds
// it for 16 cycles or more). With double shuffles an iteration of the fused
// step with the objective took 16.6 us at 64^3, 40.7 at 101 x 147 x 183 and
// 23.3 at 128^3, of which 8.0, 17.1 and 9.3 were the sums (objective off: 8.6,
// 23.6, 13.9). With these sums the same iterations took 11.3, 30.7 and 18.6 us.
// A float-float add is 11 FP32 operations. The lanes also trade quantities
// first (lane groups of 8 end up with one of the 4 sums each), which takes 6
// adds and 12 shuffles per lane instead of 20 adds and 40 shuffles.
// Error of the recorded objective against float64, before and after: the
// same to all digits shown, 4.7e-10 (64^3), 1.8e-10 (101 x 147 x 183), 3.0e-10
// (128^3); the float32 terms set it.
//
// Range: a float-float overflows at 3.4e38 where a double does not, so a CTA
// with any accumulator at or above 1e30 (or not finite) takes the same tree in
// double. Both trees add in a fixed order.
#pragma once

#include <cuda_runtime.h>

namespace spg {
namespace ff {

struct FF {
    float hi, lo;
};

// s + e == a + b exactly (no ordering of |a|, |b| assumed)
__device__ __forceinline__ FF two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

__device__ __forceinline__ FF add(FF a, FF b)
{
    FF t = two_sum(a.hi, b.hi);
    t.lo = __fadd_rn(t.lo, __fadd_rn(a.lo, b.lo));
    const float s = __fadd_rn(t.hi, t.lo);
    return {s, __fsub_rn(t.lo, __fsub_rn(s, t.hi))};
}

__device__ __forceinline__ double add(double a, double b) { return a + b; }

__device__ __forceinline__ FF shfl_xor(FF a, int m)
{
    return {__shfl_xor_sync(0xffffffffu, a.hi, m), __shfl_xor_sync(0xffffffffu, a.lo, m)};
}

__device__ __forceinline__ double shfl_xor(double a, int m) { return __shfl_xor_sync(0xffffffffu, a, m); }

__device__ __forceinline__ double to_double(FF a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double to_double(double a) { return a; }

// True where a float-float sum of CTA-many such values could overflow.
__device__ __forceinline__ bool too_big(FF a) { return !(fabsf(a.hi) < 1e30f); }

// Warp sums of 4 quantities: lane l returns the sum over the warp of
// quantity l >> 3 (every lane of a group of 8 the same value).
template <class T>
__device__ __forceinline__ T warp_sum4(const T (&v)[4], int lane)
{
    const bool up = (lane & 16) != 0;
    T a = add(up ? v[2] : v[0], shfl_xor(up ? v[0] : v[2], 16));
    T b = add(up ? v[3] : v[1], shfl_xor(up ? v[1] : v[3], 16));
    const bool odd = (lane & 8) != 0;
    T s = add(odd ? b : a, shfl_xor(odd ? a : b, 8));
#pragma unroll
    for (int m = 4; m > 0; m >>= 1) s = add(s, shfl_xor(s, m));
    return s;
}

// Second level, by one warp: red[w * 4 + q] for nw <= 32 warps; lane q (< 4)
// returns the total of quantity q, added over the warps in a fixed tree.
template <class T>
__device__ __forceinline__ T cross_warp_sum4(const T *red, int nw, int lane, T zero)
{
    T s = lane < nw * 4 ? red[lane] : zero;
    for (int i = lane + 32; i < nw * 4; i += 32) s = add(s, red[i]);
#pragma unroll
    for (int m = 4; m < 32; m <<= 1) s = add(s, shfl_xor(s, m));
    return s;
}

}  // namespace ff
}  // namespace spg
