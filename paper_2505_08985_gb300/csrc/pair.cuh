// Pair arithmetic: a value held as the unevaluated sum of two FP32 numbers,
// about 48 bits, for kernels that would otherwise be bound by the FP64 unit
// (1/64 of the FP32 rate on this device).  The error-free transformations are
// Knuth's two-sum and the FMA two-product; elementary functions are built on
// them from their series (see sample.cu).
#pragma once

namespace pndf {

struct Pair {
    float h, l;
};

__device__ __forceinline__ Pair quick_sum(float a, float b)  // |a| >= |b| or a = 0
{
    const float s = __fadd_rn(a, b);
    return Pair{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Pair two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return Pair{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return Pair{p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ Pair operator+(Pair a, Pair b)
{
    const Pair s = two_sum(a.h, b.h);
    return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Pair operator-(Pair a) { return Pair{-a.h, -a.l}; }
__device__ __forceinline__ Pair operator-(Pair a, Pair b) { return a + (-b); }
__device__ __forceinline__ Pair operator*(Pair a, Pair b)
{
    const Pair p = two_prod(a.h, b.h);
    return quick_sum(p.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l)));
}
__device__ __forceinline__ Pair operator*(Pair a, float b)
{
    const Pair p = two_prod(a.h, b);
    return quick_sum(p.h, __fmaf_rn(a.l, b, p.l));
}
__device__ __forceinline__ Pair operator+(Pair a, float b)
{
    const Pair s = two_sum(a.h, b);
    return quick_sum(s.h, __fadd_rn(s.l, a.l));
}
// One correction of the FP32 quotient / root; 0 for a root of 0.
__device__ __forceinline__ Pair divide(float a, Pair b)
{
    const float q = a / b.h;
    const float r = __fmaf_rn(-q, b.l, __fmaf_rn(-q, b.h, a));
    return quick_sum(q, r / b.h);
}
__device__ __forceinline__ Pair root(Pair a)
{
    const float s = sqrtf(a.h);
    if (!(s > 0.f)) return Pair{0.f, 0.f};
    const float r = __fadd_rn(__fmaf_rn(-s, s, a.h), a.l);
    return quick_sum(s, r * (0.5f / s));
}

}  // namespace pndf
