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

// z + a conj(b) and z + conj(a) b
template <typename T>
__host__ __device__ __forceinline__ cplx<T> cmad_nj(cplx<T> a, cplx<T> b, cplx<T> z) {
  return mk(mad(a.im, b.im, mad(a.re, b.re, z.re)), mad(-a.re, b.im, mad(a.im, b.re, z.im)));
}
template <typename T>
__host__ __device__ __forceinline__ cplx<T> cmad_jn(cplx<T> a, cplx<T> b, cplx<T> z) {
  return mk(mad(a.im, b.im, mad(a.re, b.re, z.re)), mad(-a.im, b.re, mad(a.re, b.im, z.im)));
}

// C += A B, A B^dag, A^dag B: 108 fused multiply-adds (a product and a matrix sum written
// separately cost 144 and 18)
template <typename T>
__device__ __forceinline__ void mac(Mat3<T>& C, const Mat3<T>& A, const Mat3<T>& B) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) C.m[i][j] = cmad(A.m[i][k], B.m[k][j], C.m[i][j]);
}
template <typename T>
__device__ __forceinline__ void mac_nd(Mat3<T>& C, const Mat3<T>& A, const Mat3<T>& B) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) C.m[i][j] = cmad_nj(A.m[i][k], B.m[j][k], C.m[i][j]);
}
template <typename T>
__device__ __forceinline__ void mac_dn(Mat3<T>& C, const Mat3<T>& A, const Mat3<T>& B) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k) C.m[i][j] = cmad_jn(A.m[k][i], B.m[k][j], C.m[i][j]);
}
// A B (the first product of each chain is a multiplication)
template <typename T>
__device__ __forceinline__ Mat3<T> mm(const Mat3<T>& A, const Mat3<T>& B) {
  Mat3<T> C;
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j)
      C.m[i][j] = cmad(A.m[i][2], B.m[2][j], cmad(A.m[i][1], B.m[1][j], A.m[i][0] * B.m[0][j]));
  return C;
}

}  // namespace pfmp
