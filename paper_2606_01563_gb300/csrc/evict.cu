// Moment-informed eviction (Algorithm 1: append step and Phase 1).
//
// Algorithm 1's loop literally: every iteration scores the surviving rows by
// alpha_j ||r_j||, alpha_j the softmax weight summed over the G query heads of
// the unit and r_j the moment residual
//   r_j = v_j - v_bar - scale * C' k_j,  C' = C with |n C_ab| < tau zeroed
// (Eq. residual with S_tilde = n C), evicts the argmin (ties: lower row =
// lower position), and folds the evicted row into (n, mu_k, mu_v, C) with the
// Welford form of Eq. app_update.  Rows are compacted in order at the end.
// Each row keeps y_j = S_tilde k_j, which a fold changes by a multiple of one
// vector: O(d) per row and eviction instead of O(d^2).  The clamp stays exact:
// every iteration lists the entries with 0 < |S_tilde_ab| < tau and takes
// their products out of y_j; above kMaxClamp such entries that iteration
// computes C' k_j directly.
//
// Two kernels, chosen by the capacity: evict_reg_kernel here (up to kRegCap =
// 1152 rows, the capacity up to which y rows are kept across calls), and
// evict_large_kernel (evict_large.cu).
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>

#include "evict_common.cuh"
#include "warp_mma.cuh"

namespace cg = cooperative_groups;

namespace mkv {

namespace {

// ---------------------------------------------------------------------------
// Register kernel: a cluster of 8, 4 or 2 CTAs of 512 threads per unit, each
// with a contiguous slice of at most 16 RPW rows (RPW the smallest of 2, 5, 9
// and 16 that holds a slice of the capacity: a warp computes all of its RPW
// rows, there or not).  Warp w owns the slice rows w, w + 16, ... and lane l
// the dims [l*DPL, (l+1)*DPL) of each, with y_j = S_tilde k_j (raw co-moment
// form, S_tilde = n C) in registers.  The CTAs share out S_tilde itself by
// rows, in shared memory: a fold costs a warp one row or a few, and every CTA
// lists the clamped entries of its own rows.
// Every thread computes the Welford fold of its own dims from the evicted row,
// so the only barriers of an iteration are one block barrier (the block's
// minimum key) and one cluster barrier (every CTA's key, candidate row, its
// softmax terms and its count of clamped entries, written into every CTA's
// mailbox beforehand).  Scores assume that no entry is clamped; when a mailbox
// says otherwise, the lists are exchanged and the rows scored again.
//
// What bounds it: a chain of dependent steps, not memory: about 2 us per
// further eviction (64 of 192, 576, 1152 rows: 119, 147, 177 us; 144 us
// for the first with five rows per warp instead of two) and a fixed part of a
// few round trips (length, rows and moments, one cluster exchange of the
// softmax maxima and sums, rows out).  The block's minimum key goes through one
// word pair per warp and warp-wide reductions: 64-bit minimum atomics on one
// shared word made the same evictions 157 and 160 us.  Logits and S_tilde k of
// rows without a kept y run on the tensor cores from the rows in shared memory;
// survivors are written straight from there to their compacted places (every
// CTA has seen every evicted row, so no count is exchanged).
constexpr int kRegCap = 1152;  // largest capacity of this kernel
constexpr int kRT = 512;       // threads per CTA
constexpr int kRW = kRT / 32;  // warps per CTA
constexpr int kMaxCL = 8;      // CTAs per unit at most
constexpr int kBlk = 32;       // rows per block of the set-up products

template <int D, int G, int RPW>
struct RegLayout {
  static constexpr int R = kRW * RPW;  // rows of a slice at most
  static constexpr int LDK = D + 8;    // row stride of K: conflict-free matrix loads
  static constexpr int LDY = D + 4;    // row stride of a block of set-up products
  static constexpr size_t K = 0, V = K + (size_t)R * LDK * 2, lg = V + (size_t)R * D * 2,
                          pos = lg + (size_t)G * R * 4, yb = pos + (size_t)R * 4, S = yb + (size_t)kBlk * LDY * 4;
  static __host__ __device__ size_t total(int cl) { return S + (size_t)(D / cl) * D * 4; }
};

template <int D, int G, int RPW>
__global__ void __launch_bounds__(kRT, 1) evict_reg_kernel(const EvictArgs a) {
  using L = RegLayout<D, G, RPW>;
  constexpr int DPL = D / 32;  // dims per lane
  constexpr int KS = D / 16, NT = D / 8, CH = D / 8;
  constexpr int P = RPW <= 2 ? 2 : RPW <= 8 ? 8 : 16;  // padded row count of the transposing sums
  constexpr int SH = P == 2 ? 4 : P == 8 ? 2 : 1;      // lane l scores row l >> SH
  extern __shared__ __align__(16) uint8_t dsmem[];
  __nv_bfloat16* Ks = reinterpret_cast<__nv_bfloat16*>(dsmem + L::K);  // [R][LDK]
  __nv_bfloat16* Vs = reinterpret_cast<__nv_bfloat16*>(dsmem + L::V);  // [R][D]
  float* lg = reinterpret_cast<float*>(dsmem + L::lg);                 // [G][R] logits, then e_hj
  int32_t* s_pos = reinterpret_cast<int32_t*>(dsmem + L::pos);
  float* yb = reinterpret_cast<float*>(dsmem + L::yb);  // [kBlk][LDY]
  float* S = reinterpret_cast<float*>(dsmem + L::S);    // [D / CL][D] this CTA's rows of S_tilde
  __shared__ __align__(16) __nv_bfloat16 s_q[8][L::LDK];  // heads past G are zero
  __shared__ float s_mw[kRW][8], s_zw[kRW][8];          // (max, sum) of each warp's rows
  __shared__ float mail_m[kMaxCL][G], mail_z[kMaxCL][G];  // every CTA's (max, sum)
  __shared__ float mail_e[2][kMaxCL][G];                  // e_h of each CTA's candidate row
  __shared__ uint2 s_key[kRW];  // each warp's minimum key: (row, score bits)
  __shared__ unsigned long long mail_key[2][kMaxCL];
  __shared__ int mail_nz[2][kMaxCL];
  __shared__ __align__(16) __nv_bfloat16 mail_row[2][kMaxCL][2 * D];
  __shared__ uint32_t s_zidx[kMaxClamp], s_gidx[kMaxClamp];  // this CTA's clamped entries, the unit's
  __shared__ float s_zval[kMaxClamp], s_gval[kMaxClamp];
  __shared__ int s_nz;
  __shared__ uint32_t s_mask[kRW];  // survivors of each warp

  // In mkv_decode_evict_step the decode kernel may be placed on free SMs while
  // this one runs: it waits before it reads.  After mkv_evict_append the next
  // launch may be a decode step with early_load, which does not.
  grid_dependency_wait();
  if (a.release) grid_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank()), CL = static_cast<int>(cluster.num_blocks());
  const int u = blockIdx.x / CL;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const size_t row0 = (size_t)u * a.cap;
  __nv_bfloat16* Kg = reinterpret_cast<__nv_bfloat16*>(a.K) + row0 * D;
  __nv_bfloat16* Vg = reinterpret_cast<__nv_bfloat16*>(a.V) + row0 * D;
  int32_t* Pg = a.pos + row0;
  const int len_in = a.len[u], seen_in = a.seen[u];
  int n = a.n[u];
  const bool has_y = a.Y != nullptr && a.y_len != nullptr;
  const int y_len_in = has_y ? a.y_len[u] : 0;
  const bool has_new = a.k_new != nullptr;
  if (len_in < 0 || len_in > a.cap || (has_new && len_in + 1 > a.cap)) {
    if (rank == 0 && tid == 0) record_error(a.ws, MKV_ERR_CAPACITY, u);
    return;  // uniform over the cluster
  }
  const int len = len_in + (has_new ? 1 : 0);
  const int rows_per = (len + CL - 1) / CL;
  const int j0 = min(len, rank * rows_per), j1 = min(len, j0 + rows_per);
  const int nr = j1 - j0;
  const int jn = has_new ? len_in - j0 : -1;  // the appended token's slice row, if it is here
  const __nv_bfloat16* kn = reinterpret_cast<const __nv_bfloat16*>(a.k_new) + (size_t)u * D;
  const __nv_bfloat16* vn = reinterpret_cast<const __nv_bfloat16*>(a.v_new) + (size_t)u * D;
  if (jn >= 0 && jn < nr) {  // the owning CTA appends the token
    for (int i = tid; i < D; i += kRT) {
      const __nv_bfloat16 k = kn[i], v = vn[i];
      Kg[(size_t)len_in * D + i] = k;
      Vg[(size_t)len_in * D + i] = v;
      Ks[jn * L::LDK + i] = k;
      Vs[jn * D + i] = v;
    }
    if (tid == 0) {
      Pg[len_in] = seen_in;
      s_pos[jn] = seen_in;
    }
  }
  cluster_arrive_release();  // every CTA has read the length; awaited before the first remote store
  if (len <= a.budget) {
    cluster_wait_acquire();
    if (rank == 0 && tid == 0) {
      a.len[u] = len;
      a.seen[u] = seen_in + (has_new ? 1 : 0);
    }
    return;
  }
  // rows 0..y_cur-1 of the cache's y rows are current (none without them)
  const int y_cur = max(0, min(y_len_in, len_in));

  // Continuous eviction: only the appended row has no y, and every CTA computes
  // the elements of its own rows of S_tilde for it.  Computed where the row is,
  // like a longer run of appended rows, n C k took 2.7 us of the call's 11 (all
  // of C in one CTA): a step at 512 rows with its decode 18.4 -> 16.4 us.
  // (the length is compared as read: nvcc 13.0.88 folded y_cur == len_in to true)
  const bool one_fresh = n > 0 && has_new && y_len_in >= len_in;
  const int y_have = one_fresh ? len : y_cur;  // rows from here on are computed row by row below
  float kf_new[DPL];
#pragma unroll
  for (int d = 0; d < DPL; ++d) kf_new[d] = one_fresh ? __bfloat162float(kn[lane * DPL + d]) : 0.f;

  // ---- this slice's rows, the query, this CTA's rows of S_tilde, the means
  for (int idx = tid; idx < nr * CH; idx += kRT) {
    const int r = idx / CH, c = idx % CH;
    if (r == jn) continue;
    const uint4 k4 = reinterpret_cast<const uint4*>(Kg + (size_t)(j0 + r) * D)[c];
    const uint4 v4 = reinterpret_cast<const uint4*>(Vg + (size_t)(j0 + r) * D)[c];
    *reinterpret_cast<uint4*>(Ks + r * L::LDK + c * 8) = k4;
    *reinterpret_cast<uint4*>(Vs + r * D + c * 8) = v4;
  }
  for (int r = tid; r < nr; r += kRT)
    if (r != jn) s_pos[r] = Pg[j0 + r];
  const __nv_bfloat16* qg = reinterpret_cast<const __nv_bfloat16*>(a.q) + (size_t)u * G * D;
  for (int i = tid; i < 8 * D; i += kRT)
    s_q[i / D][i % D] = i / D < G ? qg[i] : __float2bfloat16_rn(0.f);
  const float nf0 = static_cast<float>(n);
  const int SR = D / CL, a0 = rank * SR;  // rows [a0, a0 + SR) of S_tilde
  const float* Cg = a.C + (size_t)u * D * D;
  for (int idx = tid; idx < SR * (D / 4); idx += kRT) {
    float4 c4 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (n > 0) c4 = reinterpret_cast<const float4*>(Cg + (size_t)a0 * D)[idx];
    reinterpret_cast<float4*>(S)[idx] = make_float4(c4.x * nf0, c4.y * nf0, c4.z * nf0, c4.w * nf0);
  }
  float mk[DPL], mv[DPL], sdk[DPL], sdv[DPL];
#pragma unroll
  for (int d = 0; d < DPL; ++d) {
    mk[d] = n > 0 ? a.mu_k[(size_t)u * D + lane * DPL + d] : 0.f;
    mv[d] = n > 0 ? a.mu_v[(size_t)u * D + lane * DPL + d] : 0.f;
    sdk[d] = sdv[d] = 0.f;
  }
  if (tid == 0) s_nz = 0;
  __syncthreads();

  // ---- logits of this CTA's rows: warp w takes rows 16 w .. 16 w + 15 against
  // the heads as the 8-column side, and their (max, sum of exp) per head
  const float scale = rsqrtf(static_cast<float>(D));
  {
    const int g = lane >> 2, t = lane & 3;
    float m0 = -INFINITY, m1 = -INFINITY, z0 = 0.f, z1 = 0.f;  // heads 2t, 2t + 1
    if (warp * 16 < nr) {
      float c0[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kk = 0; kk < KS; ++kk) {
        uint32_t k4[4];
        ldsm_x4(k4, Ks + (warp * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * L::LDK + kk * 16 + (lane >> 4) * 8);
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(&s_q[g][kk * 16 + 2 * t]);
        const uint32_t b1 = *reinterpret_cast<const uint32_t*>(&s_q[g][kk * 16 + 8 + 2 * t]);
        if (kk & 1) mma_m16n8k16(c1, k4[0], k4[1], k4[2], k4[3], b0, b1);
        else mma_m16n8k16(c0, k4[0], k4[1], k4[2], k4[3], b0, b1);
      }
      const int ra = warp * 16 + g, rb = ra + 8;
      const float x0 = ra < nr ? (c0[0] + c1[0]) * scale : -INFINITY, x1 = ra < nr ? (c0[1] + c1[1]) * scale : -INFINITY;
      const float x2 = rb < nr ? (c0[2] + c1[2]) * scale : -INFINITY, x3 = rb < nr ? (c0[3] + c1[3]) * scale : -INFINITY;
      if (2 * t < G) {
        if (ra < nr) lg[2 * t * L::R + ra] = x0;
        if (rb < nr) lg[2 * t * L::R + rb] = x2;
      }
      if (2 * t + 1 < G) {
        if (ra < nr) lg[(2 * t + 1) * L::R + ra] = x1;
        if (rb < nr) lg[(2 * t + 1) * L::R + rb] = x3;
      }
      m0 = fmaxf(x0, x2);
      m1 = fmaxf(x1, x3);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        m0 = fmaxf(m0, __shfl_xor_sync(kFull, m0, o));
        m1 = fmaxf(m1, __shfl_xor_sync(kFull, m1, o));
      }
      if (m0 != -INFINITY) z0 = expf(x0 - m0) + expf(x2 - m0);
      if (m1 != -INFINITY) z1 = expf(x1 - m1) + expf(x3 - m1);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        z0 += __shfl_xor_sync(kFull, z0, o);
        z1 += __shfl_xor_sync(kFull, z1, o);
      }
    }
    if (g == 0) {
      s_mw[warp][2 * t] = m0;
      s_mw[warp][2 * t + 1] = m1;
      s_zw[warp][2 * t] = z0;
      s_zw[warp][2 * t + 1] = z1;
    }
  }
  __syncthreads();
  cluster_wait_acquire();  // every CTA of the cluster has started
  if (tid < CL * G) {      // this CTA's (max, sum) of head h to rank r
    const int r = tid / G, h = tid % G;
    float m = -INFINITY, z = 0.f;
#pragma unroll
    for (int w = 0; w < kRW; ++w) m = fmaxf(m, s_mw[w][h]);
#pragma unroll
    for (int w = 0; w < kRW; ++w)
      if (s_mw[w][h] != -INFINITY) z += s_zw[w][h] * expf(s_mw[w][h] - m);
    *cluster.map_shared_rank(&mail_m[rank][h], r) = m;
    *cluster.map_shared_rank(&mail_z[rank][h], r) = z;
  }
  if (one_fresh)
    for (int j = warp; j < SR; j += kRW) {
      float s[DPL], dot = 0.f;
      ld_vec<DPL>(S + (size_t)j * D + lane * DPL, s);
#pragma unroll
      for (int d = 0; d < DPL; ++d) dot = fmaf(s[d], kf_new[d], dot);
      dot = warp_sum(dot);
      if (lane == 0) *cluster.map_shared_rank(yb + a0 + j, len_in / rows_per) = dot;
    }
  cluster_arrive_release();

  // ---- y_j = S_tilde k_j.  Rows below the cache's y_len carry it from the call
  // that last changed the moments; the others (appended since) are computed
  // here: n (C k_j) on the tensor cores, C as three bf16 parts (exact to 24
  // bits), warp w taking 8 value dims, in blocks of 32 rows
  constexpr int HP = DPL / 2;
  uint64_t y[RPW][HP];  // pairs of floats
  unsigned alive = 0u;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    const int r = warp + kRW * i;
#pragma unroll
    for (int d = 0; d < HP; ++d) y[i][d] = 0ull;
    if (r < nr) {
      alive |= 1u << i;
      if (n > 0 && j0 + r < y_cur) ld_pairs<HP>(a.Y + (row0 + j0 + r) * D + lane * DPL, y[i]);
    }
  }
  if (n > 0 && nr > 0 && j1 > y_have) {  // uniform over the CTA
    constexpr int kHalves = kRW / NT;   // warps sharing 8 value dims: 1 at D = 128 (both 16-row halves), 2 at D = 64
    const int g = lane >> 2, t = lane & 3, nt = warp % NT, half = warp / NT;
    uint32_t b3[3][KS][2];
#pragma unroll
    for (int kk = 0; kk < KS; ++kk)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const float2 c2 = *reinterpret_cast<const float2*>(Cg + (size_t)(nt * 8 + g) * D + kk * 16 + hf * 8 + 2 * t);
        float x = c2.x, w = c2.y;
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          b3[part][kk][hf] = pack_bf16x2(x, w);
          x = bf16_residual(x);
          w = bf16_residual(w);
        }
      }
#pragma unroll
    for (int blk = 0; blk < (RPW + 1) / 2; ++blk) {
      const int rlo = blk * kBlk, rhi = min(nr, rlo + kBlk);
      if (rlo < nr && j0 + rhi > y_cur) {  // a row of the block has no kept y
#pragma unroll
        for (int hh = 0; hh < 2 / kHalves; ++hh) {
          const int rt = kHalves == 1 ? hh : half;
          if (rlo + rt * 16 < L::R) {
            float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int kk = 0; kk < KS; ++kk) {
              uint32_t k4[4];
              ldsm_x4(k4, Ks + (rlo + rt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * L::LDK + kk * 16 + (lane >> 4) * 8);
              mma_m16n8k16(d0, k4[0], k4[1], k4[2], k4[3], b3[0][kk][0], b3[0][kk][1]);
              mma_m16n8k16(d1, k4[0], k4[1], k4[2], k4[3], b3[1][kk][0], b3[1][kk][1]);
              mma_m16n8k16(d2, k4[0], k4[1], k4[2], k4[3], b3[2][kk][0], b3[2][kk][1]);
            }
            float* ya = yb + (rt * 16 + g) * L::LDY + nt * 8 + 2 * t;
            ya[0] = (d0[0] + (d1[0] + d2[0])) * nf0;
            ya[1] = (d0[1] + (d1[1] + d2[1])) * nf0;
            ya[8 * L::LDY] = (d0[2] + (d1[2] + d2[2])) * nf0;
            ya[8 * L::LDY + 1] = (d0[3] + (d1[3] + d2[3])) * nf0;
          }
        }
        __syncthreads();
#pragma unroll
        for (int i = 2 * blk; i < 2 * blk + 2 && i < RPW; ++i) {
          const int r = warp + kRW * i;
          if (r < nr && j0 + r >= y_cur) ld_pairs<HP>(yb + (r - rlo) * L::LDY + lane * DPL, y[i]);
        }
        __syncthreads();
      }
    }
  }
  // clamp list of the initial moments: this CTA's entries with 0 < |S_tilde_ab| < tau
  const float tau = a.tau;
  auto scan_row = [&](int j, const float (&s)[DPL]) {
#pragma unroll
    for (int d = 0; d < DPL; ++d)
      if (s[d] != 0.f && fabsf(s[d]) < tau) {
        const int slot = atomicAdd(&s_nz, 1);
        if (slot < kMaxClamp) {
          s_zidx[slot] = static_cast<uint32_t>((a0 + j) * D + lane * DPL + d);
          s_zval[slot] = s[d];
        }
      }
  };
  if (n > 0 && tau > 0.f)
    for (int j = warp; j < SR; j += kRW) {
      float s[DPL];
      ld_vec<DPL>(S + (size_t)j * D + lane * DPL, s);
      scan_row(j, s);
    }

  // ---- softmax is shift-invariant: e_hj = exp(l_hj - M_h) with M_h the unit's
  // largest logit.  Z_h lives in lane h < G of every warp as a compensated
  // (Kahan) float, decremented per eviction: value zf - zc.  Every CTA
  // combines the same partials in the same order, so all hold the same values.
  cluster_wait_acquire();
#pragma unroll
  for (int i = 0; i < RPW; ++i)
    if (one_fresh && warp + kRW * i == jn && jn < nr) ld_pairs<HP>(yb + lane * DPL, y[i]);
  float zf = 1.f, zc = 0.f, zinv = 1.f, Mh = 0.f;
  if (lane < G) {
    float m = -INFINITY, z = 0.f;
    for (int r = 0; r < CL; ++r) m = fmaxf(m, mail_m[r][lane]);
    for (int r = 0; r < CL; ++r)
      if (mail_m[r][lane] != -INFINITY) z += mail_z[r][lane] * expf(mail_m[r][lane] - m);
    Mh = m;
    zf = z;
    zinv = 1.f / zf;
  }
  for (int jj = warp * 32 + lane; jj - lane < nr; jj += kRT)  // whole warps: the maxima come by shuffles
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float m = __shfl_sync(kFull, Mh, h);
      if (jj < nr) lg[h * L::R + jj] = expf(lg[h * L::R + jj] - m);
    }
  __syncthreads();
  // e_hj of the row this lane scores
  float ereg[G];
  {
    const int i = lane >> SH, r = warp + kRW * i;
#pragma unroll
    for (int h = 0; h < G; ++h) ereg[h] = (i < RPW && r < nr) ? lg[h * L::R + r] : 0.f;
  }

  // y_j' = y_j + (dk . k_j) dv of the warp's rows, two elements per instruction.
  // Rows evicted before, and those past the slice, are carried along without
  // a test (their shared memory is this kernel's); only live rows are scored.
  auto fold_y = [&]() {
    uint64_t dk2[HP], dv2[HP];
#pragma unroll
    for (int d = 0; d < HP; ++d) {
      dk2[d] = pair(sdk[2 * d], sdk[2 * d + 1]);
      dv2[d] = pair(sdv[2 * d], sdv[2 * d + 1]);
    }
    float pv[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      pv[i] = 0.f;
      if (i < RPW) {
        const uint2 kw = load_raw<DPL>(Ks + (warp + kRW * i) * L::LDK + lane * DPL);
        uint64_t a2 = fma2(dk2[0], unpack2(kw.x), 0ull);
        if constexpr (HP == 2) a2 = fma2(dk2[HP - 1], unpack2(kw.y), a2);
        pv[i] = pair_sum(a2);
      }
    }
    const float dsum = transpose_sum<P>(pv, lane);
#pragma unroll
    for (int i = 0; i < RPW; ++i) {
      const float dot = __shfl_sync(kFull, dsum, i << SH);
#pragma unroll
      for (int d = 0; d < HP; ++d) y[i][d] = fma2(pair(dot, dot), dv2[d], y[i][d]);
    }
  };
  const int n_evict = len - a.budget;
  int base = j0;  // where this slice's first survivor goes: the evicted rows below the slice move it down
  for (int e = 0;; ++e) {
    const int par = e & 1;
    // ---- fold the previous eviction into this CTA's rows of S_tilde and list
    // its clamped entries: S_tilde' = S_tilde + dv dk^T
    if (e > 0)
      for (int j = warp; j < SR; j += kRW) {
        const int ra = a0 + j;
        const float vd = __shfl_sync(kFull, select_n<DPL>(sdv, ra % DPL), ra / DPL);  // dv[ra]
        float s[DPL];
        bool any = false;
        ld_vec<DPL>(S + (size_t)j * D + lane * DPL, s);
#pragma unroll
        for (int d = 0; d < DPL; ++d) {
          s[d] = fmaf(vd, sdk[d], s[d]);
          any |= fabsf(s[d]) < tau;
        }
        st_vec<DPL>(S + (size_t)j * D + lane * DPL, s);
        if (any) scan_row(j, s);
      }
    if (e == n_evict) break;  // uniform over the cluster

    // ---- y_j', then the residual norms of the warp's rows:
    // r_j = v_j - mu_v - (scale / n) y_j
    const float rs = (n > 0) ? scale / static_cast<float>(n) : 0.f;
    if (e > 0) fold_y();
    float invz[G];
#pragma unroll
    for (int h = 0; h < G; ++h) invz[h] = __shfl_sync(kFull, zinv, h);
    // residual norms reduced so that lane l holds row l >> SH's; those lanes
    // score their row, and the warp's minimum key goes to the block minimum
    auto post_keys = [&](const float (&ss)[P]) {
      float pv[P];
#pragma unroll
      for (int i = 0; i < P; ++i) pv[i] = ss[i];
      const float sum = transpose_sum<P>(pv, lane);
      const int i = lane >> SH;
      unsigned hi = ~0u, lo = ~0u;  // score bits, row
      if ((lane & ((1 << SH) - 1)) == 0 && i < RPW && ((alive >> i) & 1u)) {
        float alpha = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) alpha = fmaf(ereg[h], invz[h], alpha);
        const float score = alpha * sqrtf(sum);
        hi = __float_as_uint(score);
        lo = static_cast<unsigned>(j0 + warp + kRW * i);
      }
      min_key(hi, lo);
      if (lane == 0) s_key[warp] = make_uint2(lo, hi);
    };
    // warp w < CL posts this CTA's key, candidate row and clamp count into rank w's mailbox
    auto post_mail = [&](int nz) {
      if (warp < CL) {
        const uint2 wk = s_key[lane % kRW];
        unsigned hi = wk.y, lo = wk.x;
        min_key(hi, lo);
        const int jb = (hi & lo) == ~0u ? -1 : static_cast<int>(lo) - j0;
        if (lane == 0) {
          *cluster.map_shared_rank(&mail_key[par][rank], warp) = (static_cast<unsigned long long>(hi) << 32) | lo;
          *cluster.map_shared_rank(&mail_nz[par][rank], warp) = nz;
        }
        if (jb >= 0 && lane < G) *cluster.map_shared_rank(&mail_e[par][rank][lane], warp) = lg[lane * L::R + jb];
        if (jb >= 0 && lane < D / 4) {  // lanes 0..D/8-1 carry k, the next D/8 carry v
          const bool is_v = lane >= D / 8;
          const int i = is_v ? lane - D / 8 : lane;
          const uint4 w4 = *reinterpret_cast<const uint4*>(is_v ? Vs + jb * D + i * 8 : Ks + jb * L::LDK + i * 8);
          reinterpret_cast<uint4*>(cluster.map_shared_rank(&mail_row[par][rank][is_v ? D : 0], warp))[i] = w4;
        }
      }
    };
    float part[P];
    {
      uint64_t nmv2[HP];
#pragma unroll
      for (int d = 0; d < HP; ++d) nmv2[d] = pair(-mv[2 * d], -mv[2 * d + 1]);
      const uint64_t nrs2 = pair(-rs, -rs);
#pragma unroll
      for (int i = 0; i < P; ++i) {
        part[i] = 0.f;
        if (i < RPW) {
          const uint2 vw = load_raw<DPL>(Vs + (warp + kRW * i) * D + lane * DPL);
          uint64_t s2 = 0ull;
#pragma unroll
          for (int d = 0; d < HP; ++d) {
            const uint64_t rr = fma2(nrs2, y[i < RPW ? i : 0][d], add2(unpack2(d == 0 ? vw.x : vw.y), nmv2[d]));
            s2 = fma2(rr, rr, s2);
          }
          part[i] = pair_sum(s2);
        }
      }
    }
    post_keys(part);
    __syncthreads();
    post_mail(s_nz);
    cluster.sync();
    const int my_nz = lane < CL ? mail_nz[par][lane] : 0;
    if (__any_sync(kFull, my_nz > 0)) {  // uniform over the cluster: clamped entries of C' change y; score again
      const int nz = __reduce_add_sync(kFull, min(my_nz, kMaxClamp + 1));
      const bool direct = nz > kMaxClamp;
      float* St = a.C + (size_t)u * D * D;  // direct: S_tilde transposed, in C's memory (C is written at the end)
      if (direct) {
        for (int j = warp; j < SR; j += kRW)
#pragma unroll
          for (int d = 0; d < DPL; ++d) St[(size_t)(lane * DPL + d) * D + a0 + j] = S[(size_t)j * D + lane * DPL + d];
        __threadfence();
      } else if (tid < nz) {  // the unit's list: rank by rank
        int z = tid, r = 0;
        while (z >= mail_nz[par][r]) z -= mail_nz[par][r++];
        s_gidx[tid] = cluster.map_shared_rank(s_zidx, r)[z];
        s_gval[tid] = cluster.map_shared_rank(s_zval, r)[z];
      }
      cluster.sync();  // lists and mailboxes read, S_tilde written
#pragma unroll
      for (int i = 0; i < P; ++i) {
        part[i] = 0.f;
        if (i < RPW && ((alive >> i) & 1u)) {
          const int r = warp + kRW * i;
          float yc[DPL];
          if (!direct) {
#pragma unroll
            for (int d = 0; d < HP; ++d) unpair(y[i < RPW ? i : 0][d], yc[2 * d], yc[2 * d + 1]);
            for (int z = 0; z < nz; ++z) {  // y'_a -= S_tilde_ab k_b for clamped (a, b)
              const int va = static_cast<int>(s_gidx[z] / D), kb = static_cast<int>(s_gidx[z] % D);
              if (va / DPL == lane) {
                const float corr = s_gval[z] * __bfloat162float(Ks[r * L::LDK + kb]);
#pragma unroll
                for (int d = 0; d < DPL; ++d)
                  if (va % DPL == d) yc[d] -= corr;
              }
            }
          } else {
#pragma unroll
            for (int d = 0; d < DPL; ++d) yc[d] = 0.f;
            for (int c = 0; c < D; ++c) {
              const float kv = __bfloat162float(Ks[r * L::LDK + c]);
#pragma unroll
              for (int d = 0; d < DPL; ++d) {
                const float cv = __ldcg(St + (size_t)c * D + lane * DPL + d);
                yc[d] = fmaf((fabsf(cv) < tau) ? 0.f : cv, kv, yc[d]);
              }
            }
          }
          float vf[DPL];
          load_bf16<DPL>(Vs + r * D + lane * DPL, vf);
#pragma unroll
          for (int d = 0; d < DPL; ++d) {
            const float rr = vf[d] - mv[d] - rs * yc[d];
            part[i] = fmaf(rr, rr, part[i]);
          }
        }
      }
      post_keys(part);
      __syncthreads();
      if (tid == 0) s_nz = 0;  // the next entries are listed after the cluster barrier below
      post_mail(0);
      cluster.sync();
    }

    // ---- every warp: the cluster's minimum key (ties cannot happen: rows
    // differ), by two warp-wide minimum reductions (score bits, then row)
    const unsigned long long bk = (lane < CL) ? mail_key[par][lane] : ~0ull;
    const unsigned khi = static_cast<unsigned>(bk >> 32), klo = static_cast<unsigned>(bk);
    unsigned mhi = khi, mlo = klo;
    min_key(mhi, mlo);
    const int src = __ffs(__ballot_sync(kFull, khi == mhi && klo == mlo)) - 1;
    const int js = (mhi == 0xffffffffu && mlo == 0xffffffffu) ? -1 : static_cast<int>(mlo);
    if (js < 0) {  // uniform: every rank read the same keys
      if (rank == 0 && tid == 0) record_error(a.ws, MKV_ERR_INVALID_ARG, u);
      break;
    }
    // Welford fold of the evicted row for this lane's dims (Eq. app_update)
    {
      const float inv = 1.f / static_cast<float>(n + 1);
      float kx[DPL], vx[DPL];
      load_bf16<DPL>(&mail_row[par][src][lane * DPL], kx);
      load_bf16<DPL>(&mail_row[par][src][D + lane * DPL], vx);
#pragma unroll
      for (int d = 0; d < DPL; ++d) {
        const float dk = kx[d] - mk[d];
        mk[d] = fmaf(dk, inv, mk[d]);
        mv[d] = fmaf(vx[d] - mv[d], inv, mv[d]);
        sdk[d] = dk;
        sdv[d] = vx[d] - mv[d];
      }
      n += 1;
    }
    const int jr = js - j0;
    if (jr < 0) --base;
    if (jr >= 0 && jr < nr && jr % kRW == warp) alive &= ~(1u << (jr / kRW));
    if (lane < G) {  // compensated Z_h -= e_h,js
      const float yk = -mail_e[par][src][lane] - zc;
      const float tk = zf + yk;
      zc = (tk - zf) - yk;
      zf = tk;
      zinv = 1.f / zf;
    }
  }
  // every CTA's reads of the cache, y and C lie before the loop's cluster
  // barriers, and no remote access follows them

  // ---- survivors to their places, in order, from shared memory
  if (has_y) fold_y();  // the loop left the last eviction out of y
  if (lane == 0) s_mask[warp] = alive;
  __syncthreads();
  const uint32_t mask = lane < kRW ? s_mask[lane] : 0u;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    if ((alive >> i) & 1u) {  // warp-uniform
      const int r = warp + kRW * i;
      // survivors of the slice ahead of row r: lane w counts warp w's
      const int dst = base + static_cast<int>(__reduce_add_sync(
                                 kFull, __popc(mask & ((1u << i) - 1u)) + (lane < warp ? (mask >> i) & 1u : 0u)));
      if (dst != j0 + r) {
        const size_t o = (size_t)dst * D + lane * DPL;
        if constexpr (DPL == 4) {
          *reinterpret_cast<uint2*>(Kg + o) = *reinterpret_cast<const uint2*>(Ks + r * L::LDK + lane * DPL);
          *reinterpret_cast<uint2*>(Vg + o) = *reinterpret_cast<const uint2*>(Vs + r * D + lane * DPL);
        } else {
          *reinterpret_cast<uint32_t*>(Kg + o) = *reinterpret_cast<const uint32_t*>(Ks + r * L::LDK + lane * DPL);
          *reinterpret_cast<uint32_t*>(Vg + o) = *reinterpret_cast<const uint32_t*>(Vs + r * D + lane * DPL);
        }
        if (lane == 0) Pg[dst] = s_pos[r];
      }
      if (has_y) st_pairs<HP>(a.Y + (row0 + dst) * D + lane * DPL, y[i]);
    }
  }
  // ---- the moments back: this CTA's rows of C = S_tilde / n (each warp folded its own)
  const float nf1 = static_cast<float>(n);
  for (int j = warp; j < SR; j += kRW) {
    float s[DPL];
    ld_vec<DPL>(S + (size_t)j * D + lane * DPL, s);
#pragma unroll
    for (int d = 0; d < DPL; ++d) s[d] = n > 0 ? s[d] / nf1 : 0.f;
    st_vec<DPL>(a.C + (size_t)u * D * D + (size_t)(a0 + j) * D + lane * DPL, s);
  }
  if (rank == 0 && warp == 0) {
#pragma unroll
    for (int d = 0; d < DPL; ++d) {  // single elements: mu_k is only 8-byte aligned
      a.mu_k[(size_t)u * D + lane * DPL + d] = mk[d];
      a.mu_v[(size_t)u * D + lane * DPL + d] = mv[d];
    }
    if (lane == 0) {
      a.n[u] = n;
      a.len[u] = a.budget;
      a.seen[u] = seen_in + (has_new ? 1 : 0);
      if (has_y) a.y_len[u] = a.budget;  // ordered after the other CTAs' writes by the kernel end
    }
  }
}

// Clusters of `cl` CTAs of an instance that the device holds at once (0: none).
template <int D, int G, int RPW>
int active_clusters(int cl) {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static int known[kMaxDev][kMaxCL + 1] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (known[dev][cl] == 0) {
    int n = 0;
    const size_t smem = RegLayout<D, G, RPW>::total(2);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl, 1, 1);
    cfg.blockDim = dim3(kRT, 1, 1);
    cfg.dynamicSmemBytes = RegLayout<D, G, RPW>::total(cl);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(evict_reg_kernel<D, G, RPW>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(smem)) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, evict_reg_kernel<D, G, RPW>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    known[dev][cl] = n > 0 ? n : -1;
  }
  return std::max(0, known[dev][cl]);
}

template <int D, int G, int RPW>
cudaError_t launch_reg(const EvictArgs& a, int cl, cudaStream_t stream) {
  if (active_clusters<D, G, RPW>(cl) < 1) return cudaErrorLaunchOutOfResources;  // and the instance's attributes
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>((long)a.batch * a.n_kv * cl), 1, 1);
  cfg.blockDim = dim3(kRT, 1, 1);
  cfg.dynamicSmemBytes = RegLayout<D, G, RPW>::total(cl);
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cl;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, evict_reg_kernel<D, G, RPW>, a);
}

template <int D, int G>
cudaError_t launch_rows(const EvictArgs& a, int cl, cudaStream_t stream) {
  const int slice = (a.cap + cl - 1) / cl;  // rows of one CTA's slice at most
  if (slice <= kRW * 2) return launch_reg<D, G, 2>(a, cl, stream);
  if (slice <= kRW * 5) return launch_reg<D, G, 5>(a, cl, stream);
  if (slice <= kRW * 9) return launch_reg<D, G, 9>(a, cl, stream);
  return launch_reg<D, G, 16>(a, cl, stream);
}
template <int D, int G>
int active_rows(int slice, int cl) {
  if (slice <= kRW * 2) return active_clusters<D, G, 2>(cl);
  if (slice <= kRW * 5) return active_clusters<D, G, 5>(cl);
  if (slice <= kRW * 9) return active_clusters<D, G, 9>(cl);
  return active_clusters<D, G, 16>(cl);
}

// Of 8, 4 and 2 CTAs per unit (slices of at most 256 rows) the one that takes
// the fewest waves, at a tie the larger: a second wave doubles the time, while
// an eviction's chain of barriers grows by half from 2 to 9 rows per warp and
// by a third again to 16, whose instances spill at d = 128 (412 to 468 bytes).
// us of a call with 8 / 4 / 2 CTAs, 64 evictions: 24 units of 192 rows
// 233/143/185, of 364 rows 284/173/251; 32 units of 764 rows 510/231/-; 40 of
// 264 rows 425/282/195; 64 of 192 rows 576/284/186, of 464 rows 706/341/250;
// one eviction with y, 16 and 128 units of 513 rows: 19/12/- and 96/56/-.
template <int D, int G>
cudaError_t launch_dg(const EvictArgs& a, cudaStream_t stream) {
  if (a.cap > kRegCap) return launch_evict_large(a, D, G, stream);
  const long units = (long)a.batch * a.n_kv;
  int cl = kMaxCL;
  long best = -1;
  for (int c = kMaxCL; c >= 2; c /= 2) {
    const int slice = (a.cap + c - 1) / c;
    if (slice > kRW * 16) break;
    const int act = active_rows<D, G>(slice, c);
    if (act < 1) continue;
    const long waves = (units + act - 1) / act;
    if (best < 0 || waves < best) {
      best = waves;
      cl = c;
    }
  }
  return launch_rows<D, G>(a, cl, stream);
}

}  // namespace

size_t evict_workspace_bytes(const mkv_geom& g, int32_t capacity) {
  const size_t units = (size_t)g.batch * g.n_kv_heads;
  return kHeaderBytes + align_up(units * g.group * (size_t)capacity * sizeof(float), 256) +
         units * stage_stride(capacity, g.head_dim) + evict_large_y_bytes(g, capacity);
}

void evict_carve(EvictArgs& a, const mkv_geom& g, int32_t capacity, void* ws) {
  const size_t units = (size_t)g.batch * g.n_kv_heads;
  uint8_t* p = static_cast<uint8_t*>(ws);
  a.ws = ws;
  a.scratch = reinterpret_cast<float*>(p + kHeaderBytes);
  a.stage = p + kHeaderBytes + align_up(units * g.group * (size_t)capacity * sizeof(float), 256);
  a.Yw = reinterpret_cast<float*>(static_cast<uint8_t*>(a.stage) + units * stage_stride(capacity, g.head_dim));
}

cudaError_t launch_evict(const EvictArgs& a, int head_dim, int group, cudaStream_t stream) {
#define MKV_EVICT_CASE(D, G) \
  if (head_dim == D && group == G) return launch_dg<D, G>(a, stream);
  MKV_EVICT_CASE(128, 1)
  MKV_EVICT_CASE(128, 2)
  MKV_EVICT_CASE(128, 4)
  MKV_EVICT_CASE(128, 8)
  MKV_EVICT_CASE(64, 1)
  MKV_EVICT_CASE(64, 2)
  MKV_EVICT_CASE(64, 4)
  MKV_EVICT_CASE(64, 8)
#undef MKV_EVICT_CASE
  return cudaErrorInvalidValue;
}

}  // namespace mkv
