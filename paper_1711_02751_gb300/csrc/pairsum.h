// Sums across lanes, warps and blocks: FP64, or for FP32 terms FP32 pairs (hi + lo with |lo| <= ulp(hi) / 2,
// about 48 bits; TwoSum), which keeps reductions of FP32 kernels off GB300's FP64 pipe -- one FP64 warp
// instruction holds an SM partition's pipe for about 60 cycles.  Against exact sums, pairs and FP64 sums
// of the same FP32 terms (dots, nearly orthogonal dots and norms of 18 432 to 400 000 unit-scaled random
// values) are off by the same 4.74e-10 to 9.0e-11, equal to six digits: the terms' own rounding.
// FP64 sums instead, from the lanes to the exchange: 32^2, k = 2 5.96 -> 7.06 ms over ten steps, 91^2, k = 3
// 9.85 -> 11.1, 16 x 32^2, k = 3 28.8 -> 30.9; as 64-bit integers 6.5, 10.3 and 29.7; states the same bit
// for bit but one (4e-15 apart).
#pragma once

#include "compensated.h"

namespace hdgdg {

struct PairSum {
    float hi, lo;
};
__device__ __forceinline__ PairSum add(PairSum a, PairSum b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    PairSum r;
    r.hi = __fadd_rn(s, e);
    r.lo = __fsub_rn(e, __fsub_rn(r.hi, s));
    return r;
}
__device__ __forceinline__ PairSum add(PairSum a, float b) {
    float s, e;
    two_sum(a.hi, b, s, e);
    return PairSum{s, __fadd_rn(a.lo, e)};
}
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ PairSum shfl_xor(PairSum v, int o) {
    return PairSum{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double value(PairSum v) { return f32_to_f64(v.hi) + f32_to_f64(v.lo); }
__device__ __forceinline__ double value(double v) { return v; }
template <typename T>   // double
struct SumOf {
    using S = double;
};
template <>
struct SumOf<float> {
    using S = PairSum;
};
template <>
struct SumOf<PairSum> {
    using S = PairSum;
};

}  // namespace hdgdg
