// Device helpers and launch arguments shared by the product kernels
// (matvec.cu, fiber.cuh).
#pragma once

#include "internal.cuh"

template <typename T>
__device__ __forceinline__ T fma_t(T a, T b, T c);
template <>
__device__ __forceinline__ float fma_t<float>(float a, float b, float c) {
  return __fmaf_rn(a, b, c);
}
template <>
__device__ __forceinline__ double fma_t<double>(double a, double b, double c) {
  return __fma_rn(a, b, c);
}
template <typename T>
__device__ __forceinline__ T mul_t(T a, T b);
template <>
__device__ __forceinline__ float mul_t<float>(float a, float b) { return __fmul_rn(a, b); }
template <>
__device__ __forceinline__ double mul_t<double>(double a, double b) { return __dmul_rn(a, b); }
template <typename T>
__device__ __forceinline__ T add_t(T a, T b);
template <>
__device__ __forceinline__ float add_t<float>(float a, float b) { return __fadd_rn(a, b); }
template <>
__device__ __forceinline__ double add_t<double>(double a, double b) { return __dadd_rn(a, b); }

// four consecutive values of a 16-byte aligned row segment
__device__ __forceinline__ void load4(const float *p, float *y) {
  const float4 v = __ldg(reinterpret_cast<const float4 *>(p));
  y[0] = v.x;
  y[1] = v.y;
  y[2] = v.z;
  y[3] = v.w;
}
__device__ __forceinline__ void load4(const double *p, double *y) {
  const double2 a = __ldg(reinterpret_cast<const double2 *>(p));
  const double2 b = __ldg(reinterpret_cast<const double2 *>(p) + 1);
  y[0] = a.x;
  y[1] = a.y;
  y[2] = b.x;
  y[3] = b.y;
}

__device__ __forceinline__ void store4(float *p, const float *y) {
  *reinterpret_cast<float4 *>(p) = make_float4(y[0], y[1], y[2], y[3]);
}
__device__ __forceinline__ void store4(double *p, const double *y) {
  reinterpret_cast<double2 *>(p)[0] = make_double2(y[0], y[1]);
  reinterpret_cast<double2 *>(p)[1] = make_double2(y[2], y[3]);
}

template <typename T>
struct HvLaunch {
  HvTables<T> tb;
  const T *v;
  T *w;
  T *b0, *b1, *b2;
  T *const *basis;  // Lanczos mode: vector j at basis[j] (else b[j % 3])
  T *psi;
  LanczosState *st;
  double *part;
  int64_t slice = 0;  // HV_SLICED: grid row y works on v + y * slice, w + y * slice
};

// Lazy scales of the Lanczos vectors (v_j = scale * the stored vector).  FP64, bound
// by its pipe, folds the scale into the recurrence's coefficients; FP32 scales
// each element before it is used, which keeps its rounding that of normalised
// vectors and costs nothing beside the memory traffic.
template <typename T>
__device__ __forceinline__ T vec_of(T x, T scale) {
  if constexpr (sizeof(T) == 8) return x;
  else return mul_t<T>(x, scale);
}
template <typename T>
__device__ __forceinline__ T coef_of(double c, double scale) {
  return (T)(sizeof(T) == 8 ? c * scale : c);
}
// what a sum over vec_of elements still has to be multiplied with
template <typename T>
__device__ __forceinline__ double fold_of(T scale) {
  return sizeof(T) == 8 ? (double)scale : 1.0;
}

// Sum over a CTA of NT threads (fixed order), in thread 0 of the first warp:
// the values cross shared memory and one warp adds them.  A shuffle tree in
// every warp would cost each thread 5 FP64 additions, as much FP64 issue as a
// third of an element's product (GB300 issues FP64 at 1/64 of the FP32 rate;
// the FP64 Lanczos-mode product at 1.18e7 elements: 588 -> 474 us with this and
// <v_j, w> summed before the scale of v_j is applied).
template <int NT>
__device__ __forceinline__ double warp_sum_of(const double *buf, int lane) {
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < NT / 32; ++k) s += buf[lane + 32 * k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  return s;
}
template <int NT>
__device__ __forceinline__ double cta_sum(double x, double *buf) {
  buf[threadIdx.x] = x;
  __syncthreads();
  return threadIdx.x < 32 ? warp_sum_of<NT>(buf, threadIdx.x) : 0.0;
}

template <typename T>
__device__ __forceinline__ double block_sum(double x, double *red) {
  for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) red[wid] = x;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) s += red[k];
  }
  return s;
}

// Asynchronous copy of one element from global to shared memory (cp.async,
// cached in L1), so that all the loads of a staging loop are in flight at
// once instead of each waiting in a register for its shared-memory store.
template <typename T>
__device__ __forceinline__ void cp_async_elem(T *dst_smem, const T *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst_smem);
  if (sizeof(T) == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.wait_all;\n" ::: "memory");
}
