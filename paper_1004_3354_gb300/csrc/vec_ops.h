// Element-level arithmetic of the vector kernels (internal header): products,
// sums and stores of one vector element in each format, warp and block sums.
// FP64 vectors accumulate in double, double-float and float vectors in
// double-float.  Each translation unit gets its own copy (anonymous namespace).
#pragma once

#include "ed_internal.h"
#include "vec16.h"

namespace ed {

namespace {

constexpr int kRedThreads = 256;

// ------------------------------------------------ element-level helpers
__device__ __forceinline__ void dmac(double& a, double x, double y) { a = fma(x, y, a); }
__device__ __forceinline__ void dmac(float2& a, float2 x, float2 y) { df_mac(a, x, y); }
__device__ __forceinline__ void dmac(float2& a, float x, float y) { df_mac1(a, make_float2(x, 0.f), y); }

__device__ __forceinline__ double to_d(double a) { return a; }
__device__ __forceinline__ double to_d(float2 a) { return (double)a.x + (double)a.y; }

__device__ __forceinline__ double add_acc(double a, double b) { return a + b; }
__device__ __forceinline__ float2 add_acc(float2 a, float2 b) { return df_add(a, b); }

__device__ __forceinline__ double shfl_x(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ float2 shfl_x(float2 v, int o) {
  return make_float2(__shfl_xor_sync(0xffffffffu, v.x, o), __shfl_xor_sync(0xffffffffu, v.y, o));
}

template <class A>
__device__ __forceinline__ A block_reduce(A v, A* sh) {
  for (int o = 16; o > 0; o >>= 1) v = add_acc(v, shfl_x(v, o));
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  int nw = blockDim.x >> 5;
  if (w == 0) {
    v = (lane < nw) ? sh[lane] : A{};
    for (int o = 16; o > 0; o >>= 1) v = add_acc(v, shfl_x(v, o));
  }
  __syncthreads();
  return v;  // valid in thread 0
}

// accumulator initialised from a stored element
__device__ __forceinline__ double acc_of(double x) { return x; }
__device__ __forceinline__ float2 acc_of(float2 x) { return x; }
__device__ __forceinline__ float2 acc_of(float x) { return make_float2(x, 0.f); }

__device__ __forceinline__ void amac(double& a, const double* cd, const float2*, int k, double x) {
  a = fma(cd[k], x, a);
}
__device__ __forceinline__ void amac(float2& a, const double*, const float2* cf, int k, float2 x) {
  df_mac(a, cf[k], x);
}
__device__ __forceinline__ void amac(float2& a, const double*, const float2* cf, int k, float x) {
  df_mac1(a, cf[k], x);
}

__device__ __forceinline__ double store_v(double a, double*) { return a; }
__device__ __forceinline__ float2 store_v(float2 a, float2*) { return df_norm(a); }
__device__ __forceinline__ float store_v(float2 a, float*) { return __fadd_rn(a.x, a.y); }

template <class V>
struct AccOf;
template <>
struct AccOf<double> { using T = double; };
template <>
struct AccOf<float2> { using T = float2; };
template <>
struct AccOf<float> { using T = float2; };

}  // namespace

}  // namespace ed
