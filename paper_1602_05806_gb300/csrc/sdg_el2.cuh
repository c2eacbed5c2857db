// Shared-memory layout of 2D FP32 elements for kernels that give a warp whole
// elements (one line per lane) and a thread two of them.
//
// For N1 = 8 rows of eight unpadded values, swizzled so that the column reads
// of four elements, and the 16-byte row reads of one, fall on distinct banks;
// otherwise rows padded by one value.
#pragma once

#include "sdg_device.cuh"

namespace sdg {

template <int N1>
struct El2 {
  static constexpr bool SW = N1 == 8;       // swizzled, unpadded
  static constexpr int ES = big_es(N1);  // floats per element
  // Byte offsets of a column (node k at col_at) and of a row of an element.
  // Swizzled: node (k, l) sits at float slot * 64 + ((k ^ s) << 3) +
  // (l ^ 4 (k >> 2)), s = slot & 3; bits 3-5 of slot * 64 are zero, so a step
  // along the column is one XOR with a constant.
  static __device__ __forceinline__ int col(int slot, int l) {
    if constexpr (SW) return 4 * (slot * 64 + ((slot & 3) << 3) + l);
    return 4 * (slot * ES + l);
  }
  static __device__ __forceinline__ int row(int slot, int k) {
    if constexpr (SW) return 4 * (slot * 64 + ((k ^ (slot & 3)) << 3) + ((k >> 2) << 2));
    return 4 * (slot * ES + k * (N1 + 1));
  }
  template <int K>
  static __device__ __forceinline__ int at(int c) {  // node K of column c
    if constexpr (SW) return c ^ (4 * ((K << 3) | ((K >> 2) << 2)));
    return c + 4 * K * (N1 + 1);
  }
  static __device__ __forceinline__ float* ptr(float* s, int off) {
    return reinterpret_cast<float*>(reinterpret_cast<char*>(s) + off);
  }
  static __device__ __forceinline__ void load_row(float* s, int slot, int k, float (&v)[N1]) {
    const int r = row(slot, k);
    if constexpr (SW) {
      const float4 a = *reinterpret_cast<const float4*>(ptr(s, r));
      const float4 b = *reinterpret_cast<const float4*>(ptr(s, r ^ 16));
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int m = 0; m < N1; ++m) v[m] = *ptr(s, r + 4 * m);
    }
  }
  static __device__ __forceinline__ void store_row(float* s, int slot, int k, const float (&v)[N1]) {
    const int r = row(slot, k);
    if constexpr (SW) {
      *reinterpret_cast<float4*>(ptr(s, r)) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(ptr(s, r ^ 16)) = make_float4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int m = 0; m < N1; ++m) *ptr(s, r + 4 * m) = v[m];
    }
  }
  // two elements at once
  template <int K = 0>
  static __device__ __forceinline__ void load_cols(float* s, int c0, int c1, P2 (&v)[N1]) {
    if constexpr (K < N1) {
      v[K] = P2(*ptr(s, at<K>(c0)), *ptr(s, at<K>(c1)));
      load_cols<K + 1>(s, c0, c1, v);
    }
  }
  template <int K = 0>
  static __device__ __forceinline__ void store_cols(float* s, int c0, int c1, const P2 (&v)[N1]) {
    if constexpr (K < N1) {
      *ptr(s, at<K>(c1)) = v[K].hi();
      *ptr(s, at<K>(c0)) = v[K].lo();
      store_cols<K + 1>(s, c0, c1, v);
    }
  }
  static __device__ __forceinline__ void load_rows(float* s, int s0, int s1, int k, P2 (&v)[N1]) {
    float a[N1], b[N1];
    load_row(s, s0, k, a);
    load_row(s, s1, k, b);
#pragma unroll
    for (int m = 0; m < N1; ++m) v[m] = P2(a[m], b[m]);
  }
  static __device__ __forceinline__ void store_rows(float* s, int s0, int s1, int k, const P2 (&v)[N1]) {
    float a[N1], b[N1];
#pragma unroll
    for (int m = 0; m < N1; ++m) {
      a[m] = v[m].lo();
      b[m] = v[m].hi();
    }
    store_row(s, s1, k, b);
    store_row(s, s0, k, a);
  }
  static __device__ __forceinline__ int node(int slot, int k, int l) {  // float offset
    if constexpr (SW) return slot * 64 + ((k ^ (slot & 3)) << 3) + (l ^ ((k >> 2) << 2));
    return slot * ES + k * (N1 + 1) + l;
  }
};

}  // namespace sdg
