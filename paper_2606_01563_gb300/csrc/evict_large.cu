// Moment-informed eviction (Algorithm 1: append step and Phase 1) for caches
// whose row slices do not fit the register kernel (evict.cu): capacities
// above 1152 rows, up to 65536.
//
// One cluster of 8, 12 or 16 CTAs per unit; CTA r owns a contiguous slice of
// the unit's rows, warp w of it the slice rows w, w + 16, ..., and lane l the
// dims [l*DPL, (l+1)*DPL) of each row.  The loop is the register kernel's: the
// raw co-moment S_tilde = n C shared out over the CTAs by rows (a warp holds at
// most one), a list of the clamped entries exchanged when there are any, one
// block barrier and one cluster barrier per eviction.
// What differs is where the rows' state lives: y_j = S_tilde k_j (512 bytes a
// row at d = 128), the softmax terms and the K/V rows are in shared memory as
// far as they fit (y first: it is read and written at every eviction), else in
// the workspace and the cache, where L2 holds them.
//
// What bounds it: per eviction a CTA streams its slice once, 1.5 KB a row, so
// at 4160 rows (8 units of 12 CTAs, 347 rows per CTA) the row pass is about 4 us
// beside the 2 of the serial chain (fold, block barrier, mailboxes, cluster
// barrier): 64 evictions 430 us, the first of them 55 with the set-up, where one
// CTA per unit that recomputed C' k of every row took 73.5 ms.  The pass
// runs over 8 rows a warp at a time with all their loads in flight; the
// update of y and the residual norm share it.  The set-up products C k_j run
// on the tensor cores (keys exact in bf16, C split into three bf16 parts).
#include <cooperative_groups.h>

#include <algorithm>
#include <mutex>
#include <type_traits>

#include "evict_common.cuh"
#include "warp_mma.cuh"

namespace cg = cooperative_groups;

namespace mkv {

namespace {

constexpr int kLT = 512;       // threads per CTA
constexpr int kLW = kLT / 32;  // warps per CTA
constexpr int kMaxCL = 16;     // CTAs per cluster at most (above 8: non-portable sizes)
constexpr int kRB = 8;         // rows of a warp scored together
constexpr int kBlk = 32;       // rows per block of the set-up products
constexpr int kMaxSlice = 65536 / 8;
constexpr int kWords = kMaxSlice / kLW / 32;  // alive words per warp
// dynamic shared memory next to the static arrays (about 31 KB at d = 128, G = 8)
constexpr size_t kLargeSmem = 192 * 1024;

// Byte offsets of a slice's arrays in dynamic shared memory; those that do
// not fit stay in global memory (flags).
struct LargeLayout {
  size_t E, Y, K, V, total;
  bool e_smem, y_smem, kv_smem;
  __host__ __device__ LargeLayout(int R, int D, int G) {
    size_t off = 0;
    const size_t eb = align_up((size_t)G * R * 4, 16), yb = (size_t)R * D * 4, kb = (size_t)R * D * 2;
    E = Y = K = V = 0;
    e_smem = off + eb <= kLargeSmem / 4;
    if (e_smem) off += eb;
    y_smem = off + yb <= kLargeSmem;
    if (y_smem) {
      Y = off;
      off += yb;
    }
    kv_smem = off + 2 * kb <= kLargeSmem;
    if (kv_smem) {
      K = off;
      V = off + kb;
      off += 2 * kb;
    }
    total = off;
  }
};

template <int DPL>
__device__ __forceinline__ void unpack_bf16(const uint2& w, float (&o)[DPL]) {
  const float2 lo = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.x));
  o[0] = lo.x;
  o[1] = lo.y;
  if constexpr (DPL == 4) {
    const float2 hi = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w.y));
    o[2] = hi.x;
    o[3] = hi.y;
  }
}
template <int D, int G>
__global__ void __launch_bounds__(kLT, 1) evict_large_kernel(const EvictArgs a) {
  constexpr int NC = D / 32;   // float4 chunks per row for 8-lane row groups (logits)
  constexpr int DPL = D / 32;  // dims per lane
  constexpr int kRP = kLW * 4; // rows per pass of 8-lane groups
  constexpr int KS = D / 16, NT = D / 8;
  constexpr int P = kRB, SH = 2;  // transposing sums: lane l holds row l >> SH
  extern __shared__ __align__(16) uint8_t dsmem[];
  __shared__ __align__(16) float s_q[G][D];
  __shared__ float s_red[kLW][G];
  __shared__ double s_zpart[kLW][G];
  __shared__ float s_M[G], s_Mg[G];  // this CTA's largest logit per head (read remotely), the unit's
  __shared__ double s_Z[G], s_Zg[G];
  __shared__ float mail_e[2][kMaxCL][G];  // e_h of each CTA's candidate row
  __shared__ uint2 s_key[kLW];  // each warp's minimum key: (row, score bits)
  __shared__ unsigned long long mail_key[2][kMaxCL];
  // the mailboxes of candidate rows, and before the loop two K blocks of the set-up products
  constexpr int kMailBytes = 2 * kMaxCL * 2 * D * 2, kBlkBytes = 2 * kBlk * (D + 8) * 2;
  __shared__ __align__(16) uint8_t s_rows[kMailBytes > kBlkBytes ? kMailBytes : kBlkBytes];
  __shared__ int mail_nz[2][kMaxCL];
  __shared__ uint32_t s_zidx[kMaxClamp], s_gidx[kMaxClamp];  // this CTA's clamped entries, the unit's
  __shared__ float s_zval[kMaxClamp], s_gval[kMaxClamp];
  __shared__ int s_nz;
  __shared__ uint32_t s_alive[kLW][kWords];  // bit i of warp w: slice row w + 16 i
  __shared__ uint32_t s_bits[kMaxSlice / 32];
  __shared__ int s_pre[kMaxSlice / 32 + 1];  // survivors before each word of s_bits
  __shared__ int ex_cnt;
  auto mail_row = [&](int par, int r) -> __nv_bfloat16* {
    return reinterpret_cast<__nv_bfloat16*>(s_rows) + ((size_t)par * kMaxCL + r) * 2 * D;
  };

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
  const int len_in = a.len[u];
  const int seen_in = a.seen[u];
  const bool has_new = a.k_new != nullptr;
  if (len_in < 0 || len_in > a.cap || (has_new && len_in + 1 > a.cap)) {
    if (rank == 0 && tid == 0) record_error(a.ws, MKV_ERR_CAPACITY, u);
    return;  // uniform over the cluster
  }
  const int len = len_in + (has_new ? 1 : 0);
  const int rows_per = (len + CL - 1) / CL;
  const int j0 = min(len, rank * rows_per), j1 = min(len, j0 + rows_per);
  const int nr = j1 - j0;
  if (has_new && len_in >= j0 && len_in < j1) {  // the owning CTA appends the token
    const __nv_bfloat16* kn = reinterpret_cast<const __nv_bfloat16*>(a.k_new) + (size_t)u * D;
    const __nv_bfloat16* vn = reinterpret_cast<const __nv_bfloat16*>(a.v_new) + (size_t)u * D;
    for (int i = tid; i < D; i += kLT) {
      Kg[(size_t)len_in * D + i] = kn[i];
      Vg[(size_t)len_in * D + i] = vn[i];
    }
    if (tid == 0) Pg[len_in] = seen_in;
    __threadfence();
  }
  if (len <= a.budget) {
    cluster.sync();  // every CTA has read the length
    if (rank == 0 && tid == 0) {
      a.len[u] = len;
      a.seen[u] = seen_in + (has_new ? 1 : 0);
    }
    return;
  }

  // ---- where this slice's state lives (a CTA reads its own rows only)
  const int R = a.rows_max;
  const LargeLayout lay(R, D, G);
  float* eb = lay.e_smem ? reinterpret_cast<float*>(dsmem + lay.E) : a.scratch + ((size_t)u * a.cap + j0) * G;
  const int es = lay.e_smem ? R : nr;  // stride of a head's terms
  float* Y = lay.y_smem ? reinterpret_cast<float*>(dsmem + lay.Y) : a.Yw + (row0 + j0) * D;
  const __nv_bfloat16* Kr = Kg + (size_t)j0 * D;
  const __nv_bfloat16* Vr = Vg + (size_t)j0 * D;
  const float scale = rsqrtf(static_cast<float>(D));
  const __nv_bfloat16* qg = reinterpret_cast<const __nv_bfloat16*>(a.q) + (size_t)u * G * D;
  for (int i = tid; i < G * D; i += kLT) s_q[i / D][i % D] = __bfloat162float(qg[i]) * scale;
  __syncthreads();  // the appended row is this CTA's own
  if (lay.kv_smem) {
    __nv_bfloat16* Ks = reinterpret_cast<__nv_bfloat16*>(dsmem + lay.K);
    __nv_bfloat16* Vs = reinterpret_cast<__nv_bfloat16*>(dsmem + lay.V);
    for (int idx = tid; idx < nr * (D / 8); idx += kLT) {
      reinterpret_cast<uint4*>(Ks)[idx] = reinterpret_cast<const uint4*>(Kr)[idx];
      reinterpret_cast<uint4*>(Vs)[idx] = reinterpret_cast<const uint4*>(Vr)[idx];
    }
    Kr = Ks;
    Vr = Vs;
  }
  if (tid == 0) s_nz = 0;
  for (int i = tid; i < kLW * kWords; i += kLT) {
    const int w = i / kWords, b0 = (i % kWords) * 32;  // rows w + 16 (b0 ..)
    const int have = w < nr ? (nr - w + kLW - 1) / kLW : 0;
    s_alive[w][i % kWords] = have <= b0 ? 0u : (have - b0 >= 32 ? 0xffffffffu : (1u << (have - b0)) - 1u);
  }
  __syncthreads();

  // ---- logits of this CTA's rows (8 lanes per row), then e_hj relative to its largest
  {
    const int q = lane & 7, rsub = warp * 4 + (lane >> 3);
    float mx[G];
#pragma unroll
    for (int h = 0; h < G; ++h) mx[h] = -INFINITY;
    for (int base = 0; base < nr; base += kRP) {
      const int j = base + rsub;
      const bool ok = j < nr;
      float kf[NC][4];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (ok) load4_bf16<D>(Kr + (size_t)j * D + chunk_dim<D>(q, c), kf[c]);
        else kf[c][0] = kf[c][1] = kf[c][2] = kf[c][3] = 0.f;
      }
#pragma unroll
      for (int h = 0; h < G; ++h) {
        float acc = 0.f;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float4 q4 = *reinterpret_cast<const float4*>(&s_q[h][chunk_dim<D>(q, c)]);
          acc = fmaf(q4.x, kf[c][0], fmaf(q4.y, kf[c][1], fmaf(q4.z, kf[c][2], fmaf(q4.w, kf[c][3], acc))));
        }
        acc = group_sum(acc);
        if (ok) {
          mx[h] = fmaxf(mx[h], acc);
          if (q == 0) eb[(size_t)h * es + j] = acc;
        }
      }
    }
#pragma unroll
    for (int h = 0; h < G; ++h) {
      mx[h] = warp_max(mx[h]);
      if (lane == 0) s_red[warp][h] = mx[h];
    }
    __syncthreads();
    if (tid < G) {
      float m = -INFINITY;
      for (int w = 0; w < kLW; ++w) m = fmaxf(m, s_red[w][tid]);
      s_M[tid] = m;
    }
    __syncthreads();
    double zs[G];
#pragma unroll
    for (int h = 0; h < G; ++h) zs[h] = 0.0;
    for (int jj = tid; jj < nr; jj += kLT)
#pragma unroll
      for (int h = 0; h < G; ++h) {
        const float ev = expf(eb[(size_t)h * es + jj] - s_M[h]);
        eb[(size_t)h * es + jj] = ev;
        zs[h] += static_cast<double>(ev);
      }
#pragma unroll
    for (int h = 0; h < G; ++h) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) zs[h] += __shfl_xor_sync(kFull, zs[h], o);
      if (lane == 0) s_zpart[warp][h] = zs[h];
    }
    __syncthreads();
    if (tid < G) {
      double z = 0.0;
      for (int w = 0; w < kLW; ++w) z += s_zpart[w][tid];
      s_Z[tid] = z;
    }
  }
  cluster_arrive_release();  // (max, sum) published; awaited after the set-up products

  // ---- y_j = S_tilde k_j = n (C k_j) of the slice on the tensor cores: warp w
  // takes 8 value dims (its part of C as three bf16 parts in registers, exact
  // to 24 bits) over blocks of 32 keys staged through shared memory
  int n = a.n[u];
  const float nf0 = static_cast<float>(n);
  const float* Cg = a.C + (size_t)u * D * D;
  if (n > 0) {
    constexpr int kHalves = kLW / NT;  // warps sharing an n-tile: 1 at D = 128 (both row halves each), 2 at D = 64
    const int g = lane >> 2, t = lane & 3, nt = warp % NT, half = warp / NT;
    uint32_t b3[3][KS][2];
#pragma unroll
    for (int kk = 0; kk < KS; ++kk)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const float2 c2 = *reinterpret_cast<const float2*>(Cg + (size_t)(nt * 8 + g) * D + kk * 16 + hf * 8 + 2 * t);
        float x = c2.x, y = c2.y;
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          b3[part][kk][hf] = pack_bf16x2(x, y);
          x = bf16_residual(x);
          y = bf16_residual(y);
        }
      }
    __nv_bfloat16* kb = reinterpret_cast<__nv_bfloat16*>(s_rows);
    constexpr int LD = D + 8, CH = D / 8;
    const int pr = tid / CH, pc = tid % CH;
    const bool act = pr < kBlk;
    const int nblk = (nr + kBlk - 1) / kBlk;
    auto fetch = [&](int blk) -> uint4 {
      const int r = blk * kBlk + pr;
      if (act && r < nr) return reinterpret_cast<const uint4*>(Kr + (size_t)r * D)[pc];
      return make_uint4(0u, 0u, 0u, 0u);
    };
    uint4 pre = fetch(0);
    for (int blk = 0; blk < nblk; ++blk) {
      __nv_bfloat16* buf = kb + (blk & 1) * kBlk * LD;
      if (act) *reinterpret_cast<uint4*>(buf + pr * LD + pc * 8) = pre;
      if (blk + 1 < nblk) pre = fetch(blk + 1);
      __syncthreads();  // a block's buffer is written again two blocks on, past the next barrier
#pragma unroll
      for (int hh = 0; hh < 2 / kHalves; ++hh) {
        const int rt = kHalves == 1 ? hh : half;  // 16-row half of the block
        float d0[4] = {0.f, 0.f, 0.f, 0.f}, d1[4] = {0.f, 0.f, 0.f, 0.f}, d2[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int kk = 0; kk < KS; ++kk) {
          uint32_t k4[4];
          ldsm_x4(k4, buf + (rt * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * LD + kk * 16 + (lane >> 4) * 8);
          mma_m16n8k16(d0, k4[0], k4[1], k4[2], k4[3], b3[0][kk][0], b3[0][kk][1]);
          mma_m16n8k16(d1, k4[0], k4[1], k4[2], k4[3], b3[1][kk][0], b3[1][kk][1]);
          mma_m16n8k16(d2, k4[0], k4[1], k4[2], k4[3], b3[2][kk][0], b3[2][kk][1]);
        }
        const int ra = blk * kBlk + rt * 16 + g, col = nt * 8 + 2 * t;
        if (ra < nr)
          *reinterpret_cast<float2*>(Y + (size_t)ra * D + col) =
              make_float2((d0[0] + (d1[0] + d2[0])) * nf0, (d0[1] + (d1[1] + d2[1])) * nf0);
        if (ra + 8 < nr)
          *reinterpret_cast<float2*>(Y + (size_t)(ra + 8) * D + col) =
              make_float2((d0[2] + (d1[2] + d2[2])) * nf0, (d0[3] + (d1[3] + d2[3])) * nf0);
      }
    }
  } else {
    for (int i = tid; i < nr * (D / 4); i += kLT) reinterpret_cast<float4*>(Y)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }

  // ---- registers: warp w < SR holds row a0 + w of S_tilde (the CTAs share out
  // its rows), lane l columns l*DPL..; the means
  const int a0 = rank * D / CL, SR = (rank + 1) * D / CL - a0, arow = a0 + warp;
  const bool holds = warp < SR;
  float creg[DPL], mk[DPL], mv[DPL], sdk[DPL], sdv[DPL];
#pragma unroll
  for (int d = 0; d < DPL; ++d) creg[d] = 0.f;
  if (holds && n > 0) ld_vec<DPL>(Cg + (size_t)arow * D + lane * DPL, creg);
#pragma unroll
  for (int d = 0; d < DPL; ++d) {
    creg[d] *= nf0;
    mk[d] = n > 0 ? a.mu_k[(size_t)u * D + lane * DPL + d] : 0.f;
    mv[d] = n > 0 ? a.mu_v[(size_t)u * D + lane * DPL + d] : 0.f;
    sdk[d] = sdv[d] = 0.f;
  }
  const float tau = a.tau;
  auto scan_row = [&]() {  // this CTA's entries with 0 < |S_tilde_ab| < tau
#pragma unroll
    for (int d = 0; d < DPL; ++d)
      if (creg[d] != 0.f && fabsf(creg[d]) < tau) {
        const int slot = atomicAdd(&s_nz, 1);
        if (slot < kMaxClamp) {
          s_zidx[slot] = static_cast<uint32_t>(arow * D + lane * DPL + d);
          s_zval[slot] = creg[d];
        }
      }
  };
  if (holds && n > 0) scan_row();

  // ---- the unit's maximum and normaliser per head; this CTA's e_hj rescaled to it
  cluster_wait_acquire();
  if (tid < G) {
    float m = -INFINITY;
    for (int r = 0; r < CL; ++r) m = fmaxf(m, cluster.map_shared_rank(s_M, r)[tid]);
    double z = 0.0;
    for (int r = 0; r < CL; ++r) {
      const float mr = cluster.map_shared_rank(s_M, r)[tid];
      if (mr != -INFINITY) z += cluster.map_shared_rank(s_Z, r)[tid] * static_cast<double>(expf(mr - m));
    }
    s_Mg[tid] = m;
    s_Zg[tid] = z;
  }
  __syncthreads();
  {
    float f[G];
#pragma unroll
    for (int h = 0; h < G; ++h) f[h] = s_M[h] != -INFINITY ? expf(s_M[h] - s_Mg[h]) : 0.f;
    for (int jj = tid; jj < nr; jj += kLT)
#pragma unroll
      for (int h = 0; h < G; ++h) eb[(size_t)h * es + jj] *= f[h];
  }
  // Z_h lives in lane h < G of every warp as a compensated (Kahan) float,
  // decremented per eviction: value zf - zc; identical in every CTA
  float zf = 1.f, zc = 0.f, zinv = 1.f;
  if (lane < G) {
    zf = static_cast<float>(s_Zg[lane]);
    zc = static_cast<float>(static_cast<double>(zf) - s_Zg[lane]);
    zinv = 1.f / zf;
  }
  // no CTA starts the loop (whose mailboxes reuse the set-up's blocks, and
  // whose clamped products reuse C's memory) before all are done here
  cluster.sync();

  const int nri = warp < nr ? (nr - warp + kLW - 1) / kLW : 0;  // rows of this warp
  const int n_evict = len - a.budget;
  for (int e = 0;; ++e) {
    const int par = e & 1;
    // ---- fold the previous eviction into this CTA's rows of S_tilde and list
    // its clamped entries: S_tilde' = S_tilde + dv dk^T
    if (e > 0 && holds) {
      const float vd = __shfl_sync(kFull, select_n<DPL>(sdv, arow % DPL), arow / DPL);  // dv[arow]
#pragma unroll
      for (int d = 0; d < DPL; ++d) creg[d] = fmaf(vd, sdk[d], creg[d]);
      scan_row();
    }
    if (e == n_evict) break;  // uniform over the cluster

    const float rs = (n > 0) ? scale / static_cast<float>(n) : 0.f;
    float invz[G];
#pragma unroll
    for (int h = 0; h < G; ++h) invz[h] = __shfl_sync(kFull, zinv, h);
    // the residual norms ss of rows i0.. of this warp (alive mask m): lane l's row scored
    unsigned long long key = ~0ull;
    auto score_batch = [&](int i0, unsigned m, const float (&ss)[P]) {
      float pv[P];
#pragma unroll
      for (int i = 0; i < P; ++i) pv[i] = ss[i];
      const float sum = transpose_sum<P>(pv, lane);
      const int i = lane >> SH;
      if ((lane & ((1 << SH) - 1)) == 0 && ((m >> i) & 1u)) {
        const int r = warp + kLW * (i0 + i);
        float alpha = 0.f;
#pragma unroll
        for (int h = 0; h < G; ++h) alpha = fmaf(eb[(size_t)h * es + r], invz[h], alpha);
        const float score = alpha * sqrtf(sum);
        const unsigned long long k2 =
            (static_cast<unsigned long long>(__float_as_uint(score)) << 32) | static_cast<unsigned>(j0 + r);
        key = k2 < key ? k2 : key;
      }
    };
    auto post_key = [&]() {
      unsigned hi = static_cast<unsigned>(key >> 32), lo = static_cast<unsigned>(key);
      min_key(hi, lo);
      if (lane == 0) s_key[warp] = make_uint2(lo, hi);
    };
    // warp w < CL posts this CTA's key, candidate row and clamp count into rank w's mailbox
    auto post_mail = [&](int nz) {
      if (warp < CL) {
        const uint2 wk = s_key[lane % kLW];
        unsigned hi = wk.y, lo = wk.x;
        min_key(hi, lo);
        const int jb = (hi & lo) == ~0u ? -1 : static_cast<int>(lo) - j0;
        if (lane == 0) {
          *cluster.map_shared_rank(&mail_key[par][rank], warp) = (static_cast<unsigned long long>(hi) << 32) | lo;
          *cluster.map_shared_rank(&mail_nz[par][rank], warp) = nz;
        }
        if (jb >= 0 && lane < G) *cluster.map_shared_rank(&mail_e[par][rank][lane], warp) = eb[(size_t)lane * es + jb];
        if (jb >= 0 && lane < D / 4) {  // lanes 0..D/8-1 carry k, the next D/8 carry v
          const bool is_v = lane >= D / 8;
          const int i = is_v ? lane - D / 8 : lane;
          const uint4 w4 = reinterpret_cast<const uint4*>((is_v ? Vr : Kr) + (size_t)jb * D)[i];
          reinterpret_cast<uint4*>(cluster.map_shared_rank(mail_row(par, rank) + (is_v ? D : 0), warp))[i] = w4;
        }
      }
    };
    // ---- y_j' = y_j + (dk . k_j) dv, then ||v_j - mu_v - (scale / n) y_j||, 8
    // rows at a time with all their loads in flight.  Rows evicted before are
    // carried along; their scores are not posted.
    constexpr int HP = DPL / 2;
    uint64_t dk2[HP], dv2[HP], nmv2[HP];
#pragma unroll
    for (int d = 0; d < HP; ++d) {
      dk2[d] = pair(sdk[2 * d], sdk[2 * d + 1]);
      dv2[d] = pair(sdv[2 * d], sdv[2 * d + 1]);
      nmv2[d] = pair(-mv[2 * d], -mv[2 * d + 1]);
    }
    const uint64_t nrs2 = pair(-rs, -rs);
    auto batch = [&](int i0, auto full) {  // full: all 8 rows exist
      constexpr bool F = decltype(full)::value;
      const size_t off = (size_t)(warp + kLW * i0) * D + lane * DPL;
      const __nv_bfloat16 *kp = Kr + off, *vp = Vr + off;
      float* yp = Y + off;
      uint2 kw[P], vw[P];
      uint64_t y[P][HP];
#pragma unroll
      for (int i = 0; i < P; ++i) {
        kw[i] = vw[i] = make_uint2(0u, 0u);
#pragma unroll
        for (int d = 0; d < HP; ++d) y[i][d] = 0ull;
        if (F || i0 + i < nri) {
          if (e > 0) kw[i] = load_raw<DPL>(kp + i * kLW * D);
          vw[i] = load_raw<DPL>(vp + i * kLW * D);
          ld_pairs<HP>(yp + i * kLW * D, y[i]);
        }
      }
      if (e > 0) {
        float pv[P];
#pragma unroll
        for (int i = 0; i < P; ++i) {
          uint64_t a2 = fma2(dk2[0], unpack2(kw[i].x), 0ull);
          if constexpr (HP == 2) a2 = fma2(dk2[HP - 1], unpack2(kw[i].y), a2);
          pv[i] = pair_sum(a2);
        }
        const float dsum = transpose_sum<P>(pv, lane);
#pragma unroll
        for (int i = 0; i < P; ++i) {
          const float dot = __shfl_sync(kFull, dsum, i << SH);
#pragma unroll
          for (int d = 0; d < HP; ++d) y[i][d] = fma2(pair(dot, dot), dv2[d], y[i][d]);
          if (F || i0 + i < nri) st_pairs<HP>(yp + i * kLW * D, y[i]);
        }
      }
      float ss[P];
#pragma unroll
      for (int i = 0; i < P; ++i) {
        uint64_t s2 = 0ull;
#pragma unroll
        for (int d = 0; d < HP; ++d) {
          const uint64_t rr = fma2(nrs2, y[i][d], add2(unpack2(d == 0 ? vw[i].x : vw[i].y), nmv2[d]));
          s2 = fma2(rr, rr, s2);
        }
        ss[i] = pair_sum(s2);
      }
      score_batch(i0, (s_alive[warp][i0 >> 5] >> (i0 & 31)) & 0xffu, ss);
    };
    int i0 = 0;
#pragma unroll 1
    for (; i0 + kRB <= nri; i0 += kRB) batch(i0, std::true_type{});
    if (i0 < nri) batch(i0, std::false_type{});
    post_key();
    __syncthreads();
    post_mail(s_nz);
    cluster.sync();
    const int my_nz = lane < CL ? mail_nz[par][lane] : 0;
    if (__any_sync(kFull, my_nz > 0)) {  // uniform over the cluster: clamped entries of C' change y; score again
      const int nz = __reduce_add_sync(kFull, min(my_nz, kMaxClamp + 1));
      const bool direct = nz > kMaxClamp;
      float* St = a.C + (size_t)u * D * D;  // direct: S_tilde transposed, in C's memory (C is written at the end)
      if (direct) {
        if (holds)
#pragma unroll
          for (int d = 0; d < DPL; ++d) St[(size_t)(lane * DPL + d) * D + arow] = creg[d];
        __threadfence();
      } else if (tid < nz) {  // the unit's list: rank by rank
        int z = tid, r = 0;
        while (z >= mail_nz[par][r]) z -= mail_nz[par][r++];
        s_gidx[tid] = cluster.map_shared_rank(s_zidx, r)[z];
        s_gval[tid] = cluster.map_shared_rank(s_zval, r)[z];
      }
      key = ~0ull;
      cluster.sync();  // lists and mailboxes read, S_tilde written
      for (int i0 = 0; i0 < nri; i0 += kRB) {
        const unsigned m = (s_alive[warp][i0 >> 5] >> (i0 & 31)) & 0xffu;
        if (m == 0u) continue;
        float ss[P];
#pragma unroll
        for (int i = 0; i < P; ++i) {
          ss[i] = 0.f;
          if ((m >> i) & 1u) {
            const int r = warp + kLW * (i0 + i);
            float yc[DPL];
            if (!direct) {
              ld_vec<DPL>(Y + (size_t)r * D + lane * DPL, yc);
              for (int z = 0; z < nz; ++z) {  // y'_a -= S_tilde_ab k_b for clamped (a, b)
                const int va = static_cast<int>(s_gidx[z] / D), kb = static_cast<int>(s_gidx[z] % D);
                if (va / DPL == lane) {
                  const float corr = s_gval[z] * __bfloat162float(Kr[(size_t)r * D + kb]);
#pragma unroll
                  for (int d = 0; d < DPL; ++d)
                    if (va % DPL == d) yc[d] -= corr;
                }
              }
            } else {
#pragma unroll
              for (int d = 0; d < DPL; ++d) yc[d] = 0.f;
              for (int c = 0; c < D; ++c) {
                const float kv = __bfloat162float(Kr[(size_t)r * D + c]);
#pragma unroll
                for (int d = 0; d < DPL; ++d) {
                  const float cv = __ldcg(St + (size_t)c * D + lane * DPL + d);
                  yc[d] = fmaf((fabsf(cv) < tau) ? 0.f : cv, kv, yc[d]);
                }
              }
            }
            float vf[DPL];
            unpack_bf16<DPL>(load_raw<DPL>(Vr + (size_t)r * D + lane * DPL), vf);
#pragma unroll
            for (int d = 0; d < DPL; ++d) {
              const float rr = vf[d] - mv[d] - rs * yc[d];
              ss[i] = fmaf(rr, rr, ss[i]);
            }
          }
        }
        score_batch(i0, m, ss);
      }
      post_key();
      __syncthreads();
      if (tid == 0) s_nz = 0;  // the next entries are listed after the cluster barrier below
      post_mail(0);
      cluster.sync();
    }

    // ---- every warp: the cluster's minimum key (rows differ, so no ties), by
    // two warp-wide minimum reductions (score bits, then row)
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
      load_bf16<DPL>(mail_row(par, src) + lane * DPL, kx);
      load_bf16<DPL>(mail_row(par, src) + D + lane * DPL, vx);
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
    if (jr >= 0 && jr < nr && jr % kLW == warp) {  // the row's warp alone reads its alive words in the loop
      if (lane == 0) s_alive[warp][(jr / kLW) >> 5] &= ~(1u << ((jr / kLW) & 31));
      __syncwarp();
    }
    if (lane < G) {  // compensated Z_h -= e_h,js
      const float yk = -mail_e[par][src][lane] - zc;
      const float tk = zf + yk;
      zc = (tk - zf) - yk;
      zf = tk;
      zinv = 1.f / zf;
    }
  }

  // ---- survivors of the slice as a bitmap in row order, with running counts
  __syncthreads();
  const int nw = (nr + 31) / 32;
  for (int i = tid; i < nw; i += kLT) {
    uint32_t bits = 0u;
    for (int b = 0; b < 32; ++b) {  // row 32 i + b: warp b % 16, its row 2 i + b / 16
      const int w = b % kLW, k = i * (32 / kLW) + b / kLW;
      bits |= ((s_alive[w][k >> 5] >> (k & 31)) & 1u) << b;
    }
    s_bits[i] = bits;
  }
  __syncthreads();
  if (warp == 0) {
    int run = 0;
    for (int i0 = 0; i0 < nw; i0 += 32) {
      const int c = i0 + lane < nw ? __popc(s_bits[i0 + lane]) : 0;
      int x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
      }
      if (i0 + lane < nw) s_pre[i0 + lane] = run + x - c;
      run += __shfl_sync(kFull, x, 31);
    }
    if (lane == 0) ex_cnt = run;
  }
  cluster.sync();
  // ---- ordered compaction: rows that move go through the staging buffer
  int base = 0;
  for (int r = 0; r < rank; ++r) base += *cluster.map_shared_rank(&ex_cnt, r);
  uint8_t* st = static_cast<uint8_t*>(a.stage) + (size_t)u * stage_stride(a.cap, D);
  __nv_bfloat16* SK = reinterpret_cast<__nv_bfloat16*>(st);
  __nv_bfloat16* SV = SK + (size_t)a.cap * D;
  int32_t* SP = reinterpret_cast<int32_t*>(SV + (size_t)a.cap * D);
  auto dest = [&](int r) -> int {  // the row's place after compaction, -1 if evicted or unmoved
    const uint32_t bits = s_bits[r >> 5];
    if (!((bits >> (r & 31)) & 1u)) return -1;
    const int d = base + s_pre[r >> 5] + __popc(bits & ((1u << (r & 31)) - 1u));
    return d == j0 + r ? -1 : d;
  };
  constexpr int CH = D / 8;
  for (int idx = tid; idx < nr * CH; idx += kLT) {
    const int r = idx / CH, i = idx % CH, d = dest(r);
    if (d >= 0) {
      reinterpret_cast<uint4*>(SK + (size_t)d * D)[i] = reinterpret_cast<const uint4*>(Kr + (size_t)r * D)[i];
      reinterpret_cast<uint4*>(SV + (size_t)d * D)[i] = reinterpret_cast<const uint4*>(Vr + (size_t)r * D)[i];
      if (i == 0) SP[d] = Pg[j0 + r];
    }
  }
  __threadfence();
  cluster.sync();
  for (int idx = tid; idx < nr * CH; idx += kLT) {
    const int r = idx / CH, i = idx % CH, d = dest(r);
    if (d >= 0) {
      reinterpret_cast<uint4*>(Kg + (size_t)d * D)[i] = reinterpret_cast<const uint4*>(SK + (size_t)d * D)[i];
      reinterpret_cast<uint4*>(Vg + (size_t)d * D)[i] = reinterpret_cast<const uint4*>(SV + (size_t)d * D)[i];
      if (i == 0) Pg[d] = SP[d];
    }
  }
  // ---- the moments back: this CTA's rows of C = S_tilde / n
  if (holds) {
#pragma unroll
    for (int d = 0; d < DPL; ++d) creg[d] = n > 0 ? creg[d] / static_cast<float>(n) : 0.f;
    st_vec<DPL>(a.C + (size_t)u * D * D + (size_t)arow * D + lane * DPL, creg);
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
      if (a.y_len != nullptr) a.y_len[u] = 0;  // rows moved and the moments changed: no y row is current
    }
  }
}

// Clusters of `cl` CTAs that the device holds at once (0: none).
template <int D, int G>
int active_clusters(int cl) {
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static int known[kMaxDev][kMaxCL + 1] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
  std::lock_guard<std::mutex> lock(mu);
  if (known[dev][cl] == 0) {
    int n = 0;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(cl, 1, 1);
    cfg.blockDim = dim3(kLT, 1, 1);
    cfg.dynamicSmemBytes = kLargeSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const void* f = reinterpret_cast<const void*>(&evict_large_kernel<D, G>);
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kLargeSmem)) !=
            cudaSuccess ||
        cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, evict_large_kernel<D, G>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    known[dev][cl] = n > 0 ? n : -1;
  }
  return std::max(0, known[dev][cl]);
}

// More CTAs per unit shorten the row pass of every eviction, as long as all
// units' clusters are resident at once: of 16, 12 and 8 the largest such.
template <int D, int G>
cudaError_t launch_large(EvictArgs a, cudaStream_t stream) {
  const long units = (long)a.batch * a.n_kv;
  int cl = 8;
  for (int c : {16, 12})
    if (active_clusters<D, G>(c) >= units) {
      cl = c;
      break;
    }
  if (active_clusters<D, G>(cl) < 1) return cudaErrorLaunchOutOfResources;
  a.rows_max = (a.cap + cl - 1) / cl;
  const LargeLayout lay(a.rows_max, D, G);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(units * cl), 1, 1);
  cfg.blockDim = dim3(kLT, 1, 1);
  cfg.dynamicSmemBytes = lay.total;
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
  return cudaLaunchKernelEx(&cfg, evict_large_kernel<D, G>, a);
}

}  // namespace

// Workspace for the y rows of slices that shared memory does not hold (the
// slices of 8-CTA clusters, the largest that run).
size_t evict_large_y_bytes(const mkv_geom& g, int32_t capacity) {
  const LargeLayout lay((capacity + 7) / 8, g.head_dim, g.group);
  return lay.y_smem ? 0 : align_up((size_t)g.batch * g.n_kv_heads * capacity * g.head_dim * sizeof(float), 256);
}

cudaError_t launch_evict_large(const EvictArgs& a, int head_dim, int group, cudaStream_t stream) {
#define MKV_EVICT_CASE(D, G) \
  if (head_dim == D && group == G) return launch_large<D, G>(a, stream);
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
