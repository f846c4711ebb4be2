// Device helpers shared by the eviction kernels (evict.cu, evict_large.cu).
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace mkv {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ unsigned long long shfl_min_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(kFull, v, o);
    v = w < v ? w : v;
  }
  return v;
}

constexpr int kMaxClamp = 64;    // clamped entries corrected incrementally

// Bytes of staging per unit (K and V rows, positions), padded so that every
// unit's block starts on a 256-byte boundary.
__host__ __device__ inline size_t stage_stride(int cap, int D) {
  return align_up((size_t)cap * (4 * (size_t)D + 4), 256);
}

// A row is handled by a group of 8 lanes; lane q of the group owns the
// value/key dims of float4 chunks q, q+8, q+16, ... (NC = D/32 chunks), so
// the 8 lanes of a row touch 8 different bank groups.
template <int D>
__device__ __forceinline__ int chunk_dim(int q, int c) { return (q + 8 * c) * 4; }

__device__ __forceinline__ float group_sum(float v) {
  v += __shfl_xor_sync(kFull, v, 1);
  v += __shfl_xor_sync(kFull, v, 2);
  v += __shfl_xor_sync(kFull, v, 4);
  return v;
}

template <int D>
__device__ __forceinline__ void load4_bf16(const __nv_bfloat16* p, float* o) { load_bf16<4>(p, o); }

// Vectors of N floats in shared memory (aligned to 4N bytes).
template <int N>
__device__ __forceinline__ void ld_vec(const float* p, float* v) {
  if constexpr (N == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x; v[1] = t.y;
  }
}
template <int N>
__device__ __forceinline__ void st_vec(float* p, const float* v) {
  if constexpr (N == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}

// One round of a transposing butterfly: lanes with bit o set keep the upper
// W values, the others the lower W, and each adds its partner's copy.
template <int W>
__device__ __forceinline__ void tsum_round(float* v, int lane, int o) {
  const bool hi = (lane & o) != 0;
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const float send = hi ? v[i] : v[i + W];
    const float keep = hi ? v[i + W] : v[i];
    v[i] = keep + __shfl_xor_sync(kFull, send, o);
  }
}

// Warp sums of P (8 or 16) values per lane in P - 1 + 5 - log2(P) shuffles:
// returns, in every lane, the sum over the warp of v[lane >> (5 - log2 P)].
template <int P>
__device__ __forceinline__ float transpose_sum(float (&v)[P], int lane) {
  static_assert(P == 8 || P == 16, "8 or 16 values");
  if constexpr (P == 16) tsum_round<8>(v, lane, 16);
  tsum_round<4>(v, lane, P == 16 ? 8 : 16);
  tsum_round<2>(v, lane, P == 16 ? 4 : 8);
  tsum_round<1>(v, lane, P == 16 ? 2 : 4);
  float r = v[0];
#pragma unroll
  for (int o = (P == 16 ? 1 : 2); o >= 1; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
  return r;
}

template <int N>
__device__ __forceinline__ float select_n(const float (&v)[N], int i) {
  float r = v[0];
#pragma unroll
  for (int k = 1; k < N; ++k) r = (i == k) ? v[k] : r;
  return r;
}

}  // namespace mkv
