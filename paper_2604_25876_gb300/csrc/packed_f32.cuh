// packed_f32.cuh -- FP32 arithmetic shared by the streaming kernels: 4-vectors
// on the packed pair instructions, the Section 3 stencils without their 1/h
// factors, and error-free (compensated and double-float) sums.
#pragma once

#include <cuda_runtime.h>

#include "skyrme_device.cuh"

namespace skyrme {

// ------------------------------------------------- packed 4-vector helpers
struct P4 {
    float2 a, b;  // components (0,1) and (2,3)
};
__device__ __forceinline__ float2 bc(float s) { return make_float2(s, s); }
__device__ __forceinline__ P4 ld4(const float4 &v) { return {make_float2(v.x, v.y), make_float2(v.z, v.w)}; }
__device__ __forceinline__ float4 st4(const P4 &v) { return make_float4(v.a.x, v.a.y, v.b.x, v.b.y); }
__device__ __forceinline__ P4 add(const P4 &u, const P4 &v) { return {__fadd2_rn(u.a, v.a), __fadd2_rn(u.b, v.b)}; }
// u - v
__device__ __forceinline__ P4 sub(const P4 &u, const P4 &v)
{
    return {__ffma2_rn(v.a, bc(-1.f), u.a), __ffma2_rn(v.b, bc(-1.f), u.b)};
}
__device__ __forceinline__ P4 mul(float2 s, const P4 &v) { return {__fmul2_rn(s, v.a), __fmul2_rn(s, v.b)}; }
__device__ __forceinline__ P4 fma(float2 s, const P4 &v, const P4 &c)
{
    return {__ffma2_rn(s, v.a, c.a), __ffma2_rn(s, v.b, c.b)};
}
__device__ __forceinline__ float2 dot2(const P4 &u, const P4 &v, float2 acc)
{
    return __ffma2_rn(u.b, v.b, __ffma2_rn(u.a, v.a, acc));
}
__device__ __forceinline__ float hsum(float2 t) { return t.x + t.y; }
__device__ __forceinline__ float dot(const P4 &u, const P4 &v)
{
    return hsum(__ffma2_rn(u.b, v.b, __fmul2_rn(u.a, v.a)));
}
// The unscaled stencils' weights, the same for every lattice (compile-time
// constants: the compiler takes them from its constant bank instead of
// registers, which matters in the batched kernels, whose lattice
// descriptors live in global memory)
__device__ __forceinline__ float2 kW8() { return make_float2(8.f, 8.f); }
__device__ __forceinline__ float2 kWm16() { return make_float2(-16.f, -16.f); }
__device__ __forceinline__ float2 kW30() { return make_float2(30.f, 30.f); }
__device__ __forceinline__ float2 kXm1() { return make_float2(-2.f / 3.f, -2.f / 3.f); }
__device__ __forceinline__ float2 kXm2() { return make_float2(1.f / 12.f, 1.f / 12.f); }

// weighted first difference c1 (p1 - m1) + c2 (p2 - m2) (the mixed second
// derivatives, of the u_i)
__device__ __forceinline__ P4 fd1(const P4 &m2, const P4 &m1, const P4 &p1, const P4 &p2, float2 c1,
                                  float2 c2)
{
    return fma(c2, sub(p2, m2), mul(c1, sub(p1, m1)));
}
// 12h d phi = 8 (p1 - m1) - (p2 - m2), w8 = (8, 8)
__device__ __forceinline__ P4 fd1u(const P4 &m2, const P4 &m1, const P4 &p1, const P4 &p2,
                                   float2 w8)
{
    return fma(w8, sub(p1, m1), sub(m2, p2));
}
// -12h^2 d^2 phi = (p2 + m2) + 30 c - 16 (p1 + m1), wm16 = (-16, -16), w30 = (30, 30)
__device__ __forceinline__ P4 fd2n(const P4 &m2, const P4 &m1, const P4 &c, const P4 &p1,
                                   const P4 &p2, float2 wm16, float2 w30)
{
    return fma(wm16, add(p1, m1), fma(w30, c, add(p2, m2)));
}

// ------------------------------------------------- double-float sums
// The streaming kernel keeps its energy, charge and force sums as unevaluated
// sums hi + lo of two floats (|lo| <= ulp(hi)/2), combined with the error-free
// two-sum and FMA two-product transformations (Knuth, Dekker): about 48
// significant bits on the FP32 pipe.  GB300's FP64 pipe issues 2 operations
// per SM and cycle, so FP64 reductions at the end of a launch sit on the
// critical path; these do not.
struct DF {
    float hi, lo;
};
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}
__device__ __forceinline__ DF quick_two_sum(float a, float b)  // |a| >= |b|
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ DF df_add(DF a, DF b)
{
    float s, e, t, f;
    two_sum(a.hi, b.hi, s, e);
    two_sum(a.lo, b.lo, t, f);
    DF r = quick_two_sum(s, __fadd_rn(e, t));
    return quick_two_sum(r.hi, __fadd_rn(r.lo, f));
}
__device__ __forceinline__ DF df_add(DF a, float x)
{
    float s, e;
    two_sum(a.hi, x, s, e);
    return quick_two_sum(s, __fadd_rn(e, a.lo));
}
__device__ __forceinline__ DF df_mul(DF a, DF b)
{
    const float p = __fmul_rn(a.hi, b.hi);
    const float e = __fmaf_rn(a.hi, b.hi, -p);
    return quick_two_sum(p, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, e)));
}
__device__ __forceinline__ DF df_neg(DF a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ double df_value(DF a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ DF df_shfl_xor(DF a, int o)
{
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// The error-free addition of one quantity: s + x, the rounding error added to c
__device__ __forceinline__ void two_sum_acc1(float &s, float &c, float x)
{
    const float t = __fadd_rn(s, x);
    const float bb = __fsub_rn(t, s);
    c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bb)), __fsub_rn(x, bb)));
    s = t;
}

// s + x with the rounding error of the addition added to c (two quantities)
__device__ __forceinline__ void two_sum_acc(float2 &s, float2 &c, float2 x)
{
    const float2 m1 = make_float2(-1.f, -1.f);
    const float2 t = __fadd2_rn(s, x);
    const float2 bb = __ffma2_rn(s, m1, t);                      // t - s
    const float2 ea = __ffma2_rn(__ffma2_rn(bb, m1, t), m1, s);  // s - (t - bb)
    const float2 eb = __ffma2_rn(bb, m1, x);                     // x - bb
    c = __fadd2_rn(c, __fadd2_rn(ea, eb));
    s = t;
}

// Pairwise sum of x[0..K) into x[0] (K a power of two): a tree of depth log2 K
template <int K> __device__ __forceinline__ void df_tree(DF (&x)[K])
{
#pragma unroll
    for (int w = 1; w < K; w <<= 1) {
#pragma unroll
        for (int k = 0; k + w < K; k += 2 * w) x[k] = df_add(x[k], x[k + w]);
    }
}

}  // namespace skyrme
