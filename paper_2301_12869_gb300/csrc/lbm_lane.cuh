// A few neighbouring columns of a lattice row in one lane's registers: N values of a value type
// (lbm_vec.cuh, lbm_dd.cuh), pointwise arithmetic, and each column's left and right neighbour
// from the lane's own values and one shuffle.
#pragma once

#include "lbm_dd.cuh"
#include "lbm_vec.cuh"

#include <cuda_runtime.h>

namespace lbm {

template <typename V, int N>
struct Lane {
  V v[N];
};

template <typename V, int N>
__device__ __forceinline__ Lane<V, N> operator+(const Lane<V, N>& x, const Lane<V, N>& y) {
  Lane<V, N> o;
#pragma unroll
  for (int j = 0; j < N; ++j) o.v[j] = x.v[j] + y.v[j];
  return o;
}
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> operator-(const Lane<V, N>& x, const Lane<V, N>& y) {
  Lane<V, N> o;
#pragma unroll
  for (int j = 0; j < N; ++j) o.v[j] = x.v[j] - y.v[j];
  return o;
}
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> operator*(V s, const Lane<V, N>& x) {
  Lane<V, N> o;
#pragma unroll
  for (int j = 0; j < N; ++j) o.v[j] = s * x.v[j];
  return o;
}
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> fma_lane(V s, const Lane<V, N>& x, const Lane<V, N>& y) {
  Lane<V, N> o;
#pragma unroll
  for (int j = 0; j < N; ++j) o.v[j] = fmadd(s, x.v[j], y.v[j]);
  return o;
}
template <typename V, int N>
__device__ __forceinline__ Lane<V, N> splat_lane(V s) {
  Lane<V, N> o;
#pragma unroll
  for (int j = 0; j < N; ++j) o.v[j] = s;
  return o;
}
template <typename V, int N>
__device__ __forceinline__ V sum_lane(const Lane<V, N>& x) {
  V o = x.v[0];
#pragma unroll
  for (int j = 1; j < N; ++j) o = o + x.v[j];
  return o;
}

// ---- neighbours. `get` fetches a column value (a float, dd or double) from another lane:
// the neighbouring lane's nearest column
template <int N, class Get>
__device__ __forceinline__ Lane<f2, N> shift_left(const Lane<f2, N>& q, Get get) {  // value at x - 1
  Lane<f2, N> o;
  o.v[0] = make_f2(get(hi(q.v[N - 1])), lo(q.v[0]));
#pragma unroll
  for (int j = 1; j < N; ++j) o.v[j] = make_f2(hi(q.v[j - 1]), lo(q.v[j]));
  return o;
}
template <int N, class Get>
__device__ __forceinline__ Lane<f2, N> shift_right(const Lane<f2, N>& q, Get get) {  // value at x + 1
  Lane<f2, N> o;
  o.v[N - 1] = make_f2(hi(q.v[N - 1]), get(lo(q.v[0])));
#pragma unroll
  for (int j = 0; j + 1 < N; ++j) o.v[j] = make_f2(hi(q.v[j]), lo(q.v[j + 1]));
  return o;
}
template <typename V, int N, class Get>
__device__ __forceinline__ Lane<V, N> shift_left(const Lane<V, N>& q, Get get) {
  Lane<V, N> o;
  o.v[0] = get(q.v[N - 1]);
#pragma unroll
  for (int j = 1; j < N; ++j) o.v[j] = q.v[j - 1];
  return o;
}
template <typename V, int N, class Get>
__device__ __forceinline__ Lane<V, N> shift_right(const Lane<V, N>& q, Get get) {
  Lane<V, N> o;
  o.v[N - 1] = get(q.v[0]);
#pragma unroll
  for (int j = 0; j + 1 < N; ++j) o.v[j] = q.v[j + 1];
  return o;
}

// a value of lane `src` of the warp
__device__ __forceinline__ float lane_value(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double lane_value(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ dd lane_value(dd v, int src) {
  return dd{__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src)};
}

}  // namespace lbm
