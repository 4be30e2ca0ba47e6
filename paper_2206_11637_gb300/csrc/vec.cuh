// Arithmetic types of the collision: one FP64 cell (D1) or one FP32 cell (F1).
//
// Every operation rounds on its own (add, sub, mul, fma round-to-nearest; no
// contraction by the compiler), so every kernel that forms a quantity by the same
// expression forms the same number: the in-place engine, the fused step and the
// batched step stay bitwise equal.
//
// (Two FP32 cells per thread in packed f32x2 instructions were measured: they
// halve the issue slots of the arithmetic, 52 -> 45 warp instructions per FP16S
// cell, but not its time on the FMA pipe -- a packed FMA occupies it for two
// cycles -- and the registers of two cells leave 16 warps per SM instead of 24:
// FP16S 14.2 against 15.5 GLUPS, FP32 15.0 against 15.0 on a 256x192x256
// impact.)
#pragma once
#include <cuda_runtime.h>

namespace pfl {

struct D1 {
  typedef double R;
  double v;
};
struct F1 {
  typedef float R;
  float v;
};

template <class V>
__host__ __device__ __forceinline__ V vbc(double c) {  // a constant
  return V{(typename V::R)c};
}

__device__ __forceinline__ D1 operator+(D1 a, D1 b) { return D1{__dadd_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator-(D1 a, D1 b) { return D1{__dsub_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator*(D1 a, D1 b) { return D1{__dmul_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 operator-(D1 a) { return D1{-a.v}; }
__device__ __forceinline__ D1 vfma(D1 a, D1 b, D1 c) { return D1{__fma_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return F1{__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return F1{__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return F1{__fmul_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a) { return F1{-a.v}; }
__device__ __forceinline__ F1 vfma(F1 a, F1 b, F1 c) { return F1{__fmaf_rn(a.v, b.v, c.v)}; }

// reciprocal, quotient and square root (IEEE, round to nearest)
__device__ __forceinline__ D1 vrcp(D1 a) { return D1{__drcp_rn(a.v)}; }
__device__ __forceinline__ F1 vrcp(F1 a) { return F1{__frcp_rn(a.v)}; }
__device__ __forceinline__ D1 vdiv(D1 a, D1 b) { return D1{__ddiv_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 vdiv(F1 a, F1 b) { return F1{__fdiv_rn(a.v, b.v)}; }
__device__ __forceinline__ D1 vsqrt(D1 a) { return D1{__dsqrt_rn(a.v)}; }
__device__ __forceinline__ F1 vsqrt(F1 a) { return F1{__fsqrt_rn(a.v)}; }

}  // namespace pfl
