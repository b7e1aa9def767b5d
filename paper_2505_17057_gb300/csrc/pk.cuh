// pk.cuh -- arithmetic on one node, or on two neighbouring nodes at once, every operation rounded as written:
// one rounding per multiply, add or fused multiply-add, none left to the compiler's choice of
// contraction.  Kernels that evaluate the same node's contributions in different contexts (a value with one
// use in one kernel, two in another) then round alike.
//
// MMFD_PAIRED, set by a source file before its includes, picks the FP32 form.  1: paired instructions
// (fma.f32x2 and the like), one issue slot for both nodes, at the price of register pairs for the
// coefficients.  0: two single instructions, which take a coefficient from constant memory for free.
// Paired is the faster where few coefficients meet many node values: three steps per launch of the 2D NSE
// class kernel ran 35.2 us per step against 43.5 with single ones (4096^2), and the 3D class kernels
// likewise; four steps of the LCDE, whose coefficients are as many as its operations, ran 48 us against 37
// (8192^2), and that kernel stays with single ones.
#pragma once

#include <cuda_runtime.h>

namespace mmfd {

__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }

#ifndef MMFD_PAIRED
#define MMFD_PAIRED 0
#endif
#if MMFD_PAIRED
#define MMFD_PK_NS pk_paired
#else
#define MMFD_PK_NS pk_single
#endif

inline namespace MMFD_PK_NS {

// Two neighbouring nodes' values.
template <typename T>
struct Pk {
    T x, y;
    __host__ __device__ __forceinline__ T lo() const { return x; }
    __host__ __device__ __forceinline__ T hi() const { return y; }
    __device__ static __forceinline__ Pk make(T a, T b) { return {a, b}; }
    __host__ __device__ static __forceinline__ Pk fill(T a) { return {a, a}; }
};
#if MMFD_PAIRED
template <>
struct Pk<float> {
    float2 v;
    __host__ __device__ __forceinline__ float lo() const { return v.x; }
    __host__ __device__ __forceinline__ float hi() const { return v.y; }
    __device__ static __forceinline__ Pk make(float a, float b) { return {make_float2(a, b)}; }
    __host__ __device__ static __forceinline__ Pk fill(float a) { return {make_float2(a, a)}; }
};
__device__ __forceinline__ Pk<float> pfma(Pk<float> a, Pk<float> b, Pk<float> c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ Pk<float> pmul(Pk<float> a, Pk<float> b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ Pk<float> padd(Pk<float> a, Pk<float> b) { return {__fadd2_rn(a.v, b.v)}; }
// a - b, as b (-1) + a (the product is exact)
__device__ __forceinline__ Pk<float> psub(Pk<float> a, Pk<float> b) { return {__ffma2_rn(b.v, make_float2(-1.f, -1.f), a.v)}; }
#endif
template <typename T> __device__ __forceinline__ Pk<T> pfma(Pk<T> a, Pk<T> b, Pk<T> c) { return {rfma(a.x, b.x, c.x), rfma(a.y, b.y, c.y)}; }
template <typename T> __device__ __forceinline__ Pk<T> pmul(Pk<T> a, Pk<T> b) { return {rmul(a.x, b.x), rmul(a.y, b.y)}; }
template <typename T> __device__ __forceinline__ Pk<T> padd(Pk<T> a, Pk<T> b) { return {radd(a.x, b.x), radd(a.y, b.y)}; }
template <typename T> __device__ __forceinline__ Pk<T> psub(Pk<T> a, Pk<T> b) { return {rsub(a.x, b.x), rsub(a.y, b.y)}; }

}  // namespace MMFD_PK_NS

}  // namespace mmfd
