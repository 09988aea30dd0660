// Fused multiply-adds of real and complex numbers, for sums of products written as chains.
#pragma once
#include "pfmp_internal.cuh"

namespace pfmp {

// x y + z as one fused multiply-add, and z + a b as four of them.  `z + a * b` written with
// the operators above costs six instructions (the product's two roundings, then an add
// that cannot fuse): where the FP64 pipe or the issue slots bound a kernel, sums of
// products are written with cmad.
__host__ __device__ __forceinline__ float mad(float x, float y, float z) { return fmaf(x, y, z); }
__host__ __device__ __forceinline__ double mad(double x, double y, double z) { return fma(x, y, z); }
template <typename T>
__host__ __device__ __forceinline__ cplx<T> cmad(cplx<T> a, cplx<T> b, cplx<T> z) {
  return mk(mad(-a.im, b.im, mad(a.re, b.re, z.re)), mad(a.im, b.re, mad(a.re, b.im, z.im)));
}

}  // namespace pfmp
