// Device helpers shared by the eviction kernels (evict.cu, evict_large.cu).
#pragma once

#include "common.cuh"
#include "kernels.h"

namespace mkv {

constexpr unsigned kFull = 0xffffffffu;

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

// A lane's DPL dims as pairs of floats, two per instruction (fma.f32x2).
__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpair(uint64_t p, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ float pair_sum(uint64_t p) {
  float a, b;
  unpair(p, a, b);
  return a + b;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t unpack2(uint32_t w) {  // two bf16
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(w << 16), "r"(w & 0xffff0000u));
  return r;
}
// the warp's smallest (hi, lo), in every lane
__device__ __forceinline__ void min_key(unsigned& hi, unsigned& lo) {
  const unsigned m = __reduce_min_sync(kFull, hi);
  lo = __reduce_min_sync(kFull, hi == m ? lo : ~0u);
  hi = m;
}
template <int HP>
__device__ __forceinline__ void ld_pairs(const float* p, uint64_t (&v)[HP]) {
  if constexpr (HP == 2) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
    v[0] = t.x;
    v[1] = t.y;
  } else {
    v[0] = *reinterpret_cast<const unsigned long long*>(p);
  }
}
template <int HP>
__device__ __forceinline__ void st_pairs(float* p, const uint64_t (&v)[HP]) {
  if constexpr (HP == 2) *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(v[0], v[1]);
  else *reinterpret_cast<unsigned long long*>(p) = v[0];
}
// a lane's DPL dims of a row, as raw bf16 words
template <int DPL>
__device__ __forceinline__ uint2 load_raw(const __nv_bfloat16* p) {
  if constexpr (DPL == 4) return *reinterpret_cast<const uint2*>(p);
  else return make_uint2(*reinterpret_cast<const uint32_t*>(p), 0u);
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

// Warp sums of P (2, 8 or 16) values per lane in P - 1 + 5 - log2(P) shuffles:
// returns, in every lane, the sum over the warp of v[lane >> (5 - log2 P)].
template <int P>
__device__ __forceinline__ float transpose_sum(float (&v)[P], int lane) {
  static_assert(P == 2 || P == 8 || P == 16, "2, 8 or 16 values");
  if constexpr (P == 16) tsum_round<8>(v, lane, 16);
  if constexpr (P >= 8) {
    tsum_round<4>(v, lane, P == 16 ? 8 : 16);
    tsum_round<2>(v, lane, P == 16 ? 4 : 8);
  }
  constexpr int kLast = 32 / P;
  tsum_round<1>(v, lane, kLast);
  float r = v[0];
#pragma unroll
  for (int o = kLast / 2; o >= 1; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
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
