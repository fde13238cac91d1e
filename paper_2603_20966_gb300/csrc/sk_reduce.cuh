// sk_reduce.cuh -- fixed-order sums of FP32 partials, shared by the reduction
// kernels of every form.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sk {

__device__ __forceinline__ void add_to(float& s, float v) { s = __fadd_rn(s, v); }
__device__ __forceinline__ void add_to(float4& s, float4 v) {
  s.x = __fadd_rn(s.x, v.x);
  s.y = __fadd_rn(s.y, v.y);
  s.z = __fadd_rn(s.z, v.z);
  s.w = __fadd_rn(s.w, v.w);
}
__device__ __forceinline__ void set_zero(float& s) { s = 0.0f; }
__device__ __forceinline__ void set_zero(float4& s) { s = make_float4(0.f, 0.f, 0.f, 0.f); }

__device__ __forceinline__ void store_scaled(float* y, float scale, float v) {
  *y = __fmul_rn(scale, v);
}
__device__ __forceinline__ void store_scaled(float* y, float scale, float4 v) {
  *reinterpret_cast<float4*>(y) = make_float4(__fmul_rn(scale, v.x), __fmul_rn(scale, v.y),
                                              __fmul_rn(scale, v.z), __fmul_rn(scale, v.w));
}

// scale v into columns c .. c + W - 1 of a row of Y, those past Q left alone.
template <int W, class V>
__device__ __forceinline__ void store_columns(float* row, int64_t c, int64_t Q, float scale,
                                              const V& v) {
  if (c + W <= Q) {
    store_scaled(row + c, scale, v);
  } else {
    const float* vv = reinterpret_cast<const float*>(&v);
#pragma unroll
    for (int u = 0; u < W; ++u)
      if (c + u < Q) row[c + u] = __fmul_rn(scale, vv[u]);
  }
}

// Adds `N` partials, all loaded before the first is added.
template <int N, class V>
__device__ __forceinline__ const float* add_run(V& s, const float* p, int64_t zstride) {
  V v[N];
#pragma unroll
  for (int u = 0; u < N; ++u) v[u] = *reinterpret_cast<const V*>(p + u * zstride);
#pragma unroll
  for (int u = 0; u < N; ++u) add_to(s, v[u]);
  return p + N * zstride;
}

// p[0] + p[zstride] + ... (n terms, in that order), eight loads in flight: a
// thread's sum is otherwise a chain of n loads, each waiting for the L2.
template <class V>
__device__ __forceinline__ V sum_partials(const float* p, int64_t zstride, int n) {
  V s;
  set_zero(s);
  int z = 0;
  for (; z + 8 <= n; z += 8) p = add_run<8>(s, p, zstride);
  if (n & 4) p = add_run<4>(s, p, zstride);
  if (n & 2) p = add_run<2>(s, p, zstride);
  if (n & 1) add_run<1>(s, p, zstride);
  return s;
}

}  // namespace sk
