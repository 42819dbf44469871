// lbdp_vec.cuh -- NP values of one arithmetic type side by side: the nodes a
// thread of a bulk kernel works on together.  Two FP32 values go through one
// packed instruction on sm_100-class GPUs (each lane rounds as the scalar
// operation does), so a pair of nodes costs the issue slots of one; FP64 has
// one lane.
#pragma once

#include <cuda_runtime.h>

#include "lbdp_lattice.cuh"

namespace lbdp {

template <class R, int NP>
struct Vec;

template <class R>
struct Vec<R, 1> {
    R v;
    static __device__ __forceinline__ Vec of(R a) { return {a}; }
    __device__ __forceinline__ R lane(int) const { return v; }
    __device__ __forceinline__ void set(int, R a) { v = a; }
};

template <>
struct alignas(8) Vec<float, 2> {
    float2 v;
    static __device__ __forceinline__ Vec of(float a) { return {make_float2(a, a)}; }
    __device__ __forceinline__ float lane(int h) const { return h == 0 ? v.x : v.y; }
    __device__ __forceinline__ void set(int h, float a)
    {
        if (h == 0)
            v.x = a;
        else
            v.y = a;
    }
};

template <class R>
__device__ __forceinline__ Vec<R, 1> operator+(Vec<R, 1> a, Vec<R, 1> b) { return {add_x(a.v, b.v)}; }
template <class R>
__device__ __forceinline__ Vec<R, 1> operator-(Vec<R, 1> a, Vec<R, 1> b) { return {add_x(a.v, -b.v)}; }
template <class R>
__device__ __forceinline__ Vec<R, 1> operator*(Vec<R, 1> a, Vec<R, 1> b) { return {mul_x(a.v, b.v)}; }
template <class R>
__device__ __forceinline__ Vec<R, 1> vfma(Vec<R, 1> a, Vec<R, 1> b, Vec<R, 1> c) { return {fma_x(a.v, b.v, c.v)}; }

__device__ __forceinline__ Vec<float, 2> operator+(Vec<float, 2> a, Vec<float, 2> b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ Vec<float, 2> operator-(Vec<float, 2> a, Vec<float, 2> b)
{
    Vec<float, 2> r;
    asm("{.reg .b64 a, b, c;\n mov.b64 a, {%2, %3};\n mov.b64 b, {%4, %5};\n sub.rn.f32x2 c, a, b;\n"
        " mov.b64 {%0, %1}, c;}"
        : "=f"(r.v.x), "=f"(r.v.y)
        : "f"(a.v.x), "f"(a.v.y), "f"(b.v.x), "f"(b.v.y));
    return r;
}
__device__ __forceinline__ Vec<float, 2> operator*(Vec<float, 2> a, Vec<float, 2> b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ Vec<float, 2> vfma(Vec<float, 2> a, Vec<float, 2> b, Vec<float, 2> c)
{
    return {__ffma2_rn(a.v, b.v, c.v)};
}

// 1 / a.  For a pair of FP32 values, the hardware approximation and one
// Newton-Raphson step r (2 - a r) with fused multiply-adds: the rounded quotient,
// bit for bit __frcp_rn over every value from 2^-126 to 2^126 (densities lie near
// 1); a zero, infinite or denormal a gives NaN or infinity, as the state it came
// from holds.  Measured on GB300, kz_fused with __frcp_rn instead: 128^3 112.8 ->
// 113.4 us, 256^3 592.5 -> 594.0.
template <class R>
__device__ __forceinline__ Vec<R, 1> recip(Vec<R, 1> a)
{
    return {rcp_rn(a.v)};
}
__device__ __forceinline__ Vec<float, 2> recip(Vec<float, 2> a)
{
    Vec<float, 2> r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r.v.x) : "f"(a.v.x));
    asm("rcp.approx.f32 %0, %1;" : "=f"(r.v.y) : "f"(a.v.y));
    const Vec<float, 2> one = Vec<float, 2>::of(1.0f);
    const Vec<float, 2> e = vfma(Vec<float, 2>{make_float2(-a.v.x, -a.v.y)}, r, one);
    return vfma(r, e, r);
}

// min(a, 0) and max(a, 0), NaN kept.  FP64 decides on the high word: comparing
// takes the FP64 pipe.
__device__ __forceinline__ float min0(float a)
{
    float r;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(0.0f));
    return r;
}
__device__ __forceinline__ float max0(float a)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(0.0f));
    return r;
}
__device__ __forceinline__ double min0(double a) { return (unsigned)__double2hiint(a) <= 0x7FF00000u ? 0.0 : a; }
__device__ __forceinline__ double max0(double a)
{
    const unsigned h = (unsigned)__double2hiint(a);
    return h >= 0x80000000u && h <= 0xFFF00000u ? 0.0 : a;
}
template <class R, int NP>
__device__ __forceinline__ Vec<R, NP> vmin0(Vec<R, NP> a)
{
    Vec<R, NP> r;
#pragma unroll
    for (int h = 0; h < NP; ++h) r.set(h, min0(a.lane(h)));
    return r;
}
template <class R, int NP>
__device__ __forceinline__ Vec<R, NP> vmax0(Vec<R, NP> a)
{
    Vec<R, NP> r;
#pragma unroll
    for (int h = 0; h < NP; ++h) r.set(h, max0(a.lane(h)));
    return r;
}

// a scalar factor or addend
template <class R, int NP>
__device__ __forceinline__ Vec<R, NP> operator*(R a, Vec<R, NP> b) { return Vec<R, NP>::of(a) * b; }
template <class R, int NP>
__device__ __forceinline__ Vec<R, NP> vfma(R a, Vec<R, NP> b, Vec<R, NP> c) { return vfma(Vec<R, NP>::of(a), b, c); }

}  // namespace lbdp
