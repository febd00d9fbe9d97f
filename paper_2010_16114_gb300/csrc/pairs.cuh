// pairs.cuh -- sums in pairs of floats (about 2^-47 relative), for reductions of
// FP32 values where GB300's two FP64 lanes per SM would be the bound.
#pragma once
#include <cmath>

namespace coxgb {
namespace {

struct tf {
    float h, l;  // value h + l, |l| <= ulp(h) / 2
};

// a + b exactly, as sum and error (Knuth's TwoSum); an infinite sum has no error term
__device__ __forceinline__ tf two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    const float e = (a - (s - bb)) + (b - bb);
    return {s, isinf(s) ? 0.f : e};
}
__device__ __forceinline__ tf tf_add(tf a, tf b)
{
    const tf s = two_sum(a.h, b.h);
    const float e = s.l + (a.l + b.l);
    const float h = s.h + e;
    return {h, e - (h - s.h)};
}
__device__ __forceinline__ double tf_double(tf a) { return static_cast<double>(a.h) + static_cast<double>(a.l); }
__device__ __forceinline__ tf tf_of(double v)
{
    const float h = static_cast<float>(v);
    return {h, isinf(h) ? 0.f : static_cast<float>(v - static_cast<double>(h))};
}
__device__ __forceinline__ tf shfl_xor(tf a, int o)
{
    return {__shfl_xor_sync(0xffffffffu, a.h, o), __shfl_xor_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double shfl_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ tf shfl_up(tf a, int o)
{
    return {__shfl_up_sync(0xffffffffu, a.h, o), __shfl_up_sync(0xffffffffu, a.l, o)};
}
__device__ __forceinline__ double shfl_up(double a, int o) { return __shfl_up_sync(0xffffffffu, a, o); }
__device__ __forceinline__ tf shfl_at(tf a, int l)
{
    return {__shfl_sync(0xffffffffu, a.h, l), __shfl_sync(0xffffffffu, a.l, l)};
}
__device__ __forceinline__ double shfl_at(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }

} // namespace
} // namespace coxgb
