// Prefill compression (Sec. 5.1 SnapKV protocol with the moment filter of
// Sec. 4.2, read as two data-parallel selection stages).
//
// Launch sequence per call (one stream):
//   stats_tc  (chunk, unit)  window logits Q_obs K^T on the tensor cores ->
//                            online (max, sum) of each causal window row; the
//                            covariance V^T K accumulated in TMEM and the column
//                            sums -> the chunk's centred moments
//   scores_tc (chunk, unit)  logits again (token-major) -> s_t = sum over rows
//                            of exp(l - m_row) / l_row, pooled
//   select    (8-CTA cluster per unit) R0 = protected + top-k(s): radix select
//                            with 8-bit digits, histograms summed through
//                            distributed shared memory, ties to the lower
//                            position
//   rset      (cluster, unit) M0 = moments(all) - moments(R0): the chunk records
//                            merged, R0's rows gathered and their co-moment
//                            removed; C0' written as three bf16 operand parts
//   residual_tc (chunk, unit) Y = K C0'^T on the tensor cores -> score2 =
//                            s_t ||v - mu_v0 - scale y||
//   select    (cluster, unit) R = protected + top-k(score2)
//   rset      (cluster, unit) R's rows into the cache, moments of E = all \ R
//                            into the caller's mkv_moments
// Every launch is a programmatic dependent of the one before it: a kernel's
// set-up, and what it reads of the prompt or of launches further back, run
// while its predecessor drains.
//
// With the budget shared by the KV heads of a batch item (adaptive), each
// select ranks the (head, position) pairs of the batch item together: a
// per-unit select first keeps each head's own top k as candidates (the joint
// top k lies among them) when that prunes at least half the pairs, then one
// cluster per batch item ranks the candidates.
//
// The tensor-core kernels are warp-specialised: warp 0 issues the TMA copies
// (3-D tensor maps over per-unit slabs: rows past a unit's end read as zeros),
// warp 1 owns TMEM and issues tcgen05.mma, and the other warps run the
// epilogue (two groups of four in stats_tc, scores_tc and residual_tc);
// stages hand over through mbarriers whose waits are all bounded.  Head dims
// below 128 use the same 128-wide MMAs: the missing 64-column box is
// zero-filled.
#include <algorithm>
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.h"
#include "tc.cuh"
#include "warp_mma.cuh"

namespace cg = cooperative_groups;

namespace mkv {

namespace {

constexpr int kTok = 128;                   // tokens per tile
constexpr int kDP = 128;                    // padded head dim of every MMA
constexpr int kTileBytes = kTok * kDP * 2;  // one [128 x 128] bf16 tile: 2 boxes of 16 KB
constexpr int kBoxBytes = kTok * 128;
// stats_tc: two epilogue groups of 4 warps (2..5 and 6..9), each taking half
// of a tile's tokens, so that two warps per scheduler share the softmax work
constexpr int kStatsThreads = 320;
constexpr int kSelThreads = 1024;
constexpr int kPF = 0;  // tiles prefetched into L2 ahead of the one being loaded (0: none)
constexpr unsigned kFull = 0xffffffffu;

struct Layout {
  int D, G, W, RW, RWb;  // head dim, group, window, window rows = G*W, 128-row blocks of them
  int T, B;
  int hs;    // units per selection group: 1, or the KV heads of a batch item (adaptive budget)
  int Tc;    // joint selection entries per unit: T, or the length of its candidate list
  int units, n_chunks, chunk;
  size_t rec;         // floats per moment record: 4 + 2D + D*D (padded)
  float* rowpart;     // [units][n_chunks][RW][2]  (max in log2 units, sum)
  float* mpart;       // [units][n_chunks][rec]    all-token chunk moments
  float* s;           // [units][T]
  float* s2;          // [units][T]
  int32_t* idx;       // [units / hs][hs * B] selection lists (h * T + t), ascending
  int32_t* cnt;       // [units] rows each unit retains
  int32_t* cand;      // [units][Tc] per-unit candidates of a joint selection (when Tc < T)
  int32_t* hbeg;      // [units] first slot of each unit in idx
  uint8_t* cimg;      // [units][3][128 x 128] C0' as three bf16 parts, in the residual's operand layout
  float* mv0;         // [units][kDP] mu_v of E0
};

__host__ __device__ inline size_t rec_floats(int D) { return align_up(4 + 2 * (size_t)D + (size_t)D * D, 4); }

__host__ __device__ __forceinline__ int protected_count(int T, int W, int sink, int keep_window) {
  const int s = sink < T ? sink : T;
  const int w = keep_window ? (W < T ? W : T) : 0;
  const int overlap = s - (T - w) > 0 ? s - (T - w) : 0;
  return s + w - overlap;
}

Layout make_layout(const mkv_geom& g, int T, int B, int W, int sink, int keep_window, int adaptive,
                   int num_sms) {
  Layout L{};
  L.hs = 1;
  L.Tc = T;
  if (adaptive && T > B) {  // a unit keeps its protected rows plus up to every joint selection
    const long prot = protected_count(T, W, sink, keep_window);
    const long most = std::min<long>(T, (long)g.n_kv_heads * (B - prot) + prot);
    L.hs = g.n_kv_heads;
    // every pair of the joint top k is in its own head's top k, so a first
    // per-unit selection of those (`most` rows with the protected ones)
    // leaves the joint one fewer entries when they are well below T
    if (2 * most <= T) L.Tc = static_cast<int>(most);
  }
  L.D = g.head_dim;
  L.G = g.group;
  L.W = W;
  L.RW = g.group * W;
  L.RWb = (L.RW + 127) / 128;
  L.T = T;
  L.B = B;
  L.units = g.batch * g.n_kv_heads;
  long per = num_sms / L.units;  // one resident CTA per SM: fill the machine once
  const long tiles = (T + kTok - 1) / kTok;
  if (per < 1) per = 1;
  if (per > tiles) per = tiles;
  L.chunk = static_cast<int>(((tiles + per - 1) / per) * kTok);
  L.n_chunks = (T + L.chunk - 1) / L.chunk;
  L.rec = rec_floats(L.D);
  return L;
}

size_t carve(Layout& L, void* ws) {
  uint8_t* base = static_cast<uint8_t*>(ws);
  size_t off = kHeaderBytes;
  auto take = [&](size_t bytes) {
    uint8_t* p = base ? base + off : nullptr;
    off += align_up(bytes, 256);
    return p;
  };
  const size_t U = L.units;
  L.rowpart = reinterpret_cast<float*>(take(U * L.n_chunks * L.RW * 2 * sizeof(float)));
  L.mpart = reinterpret_cast<float*>(take(U * L.n_chunks * L.rec * sizeof(float)));
  L.s = reinterpret_cast<float*>(take(U * (size_t)L.T * sizeof(float)));
  L.s2 = reinterpret_cast<float*>(take(U * (size_t)L.T * sizeof(float)));
  L.idx = reinterpret_cast<int32_t*>(take(U * (size_t)L.B * sizeof(int32_t)));
  L.cnt = reinterpret_cast<int32_t*>(take(U * sizeof(int32_t)));
  L.cand = L.Tc < L.T ? reinterpret_cast<int32_t*>(take(U * (size_t)L.Tc * sizeof(int32_t))) : nullptr;
  L.hbeg = reinterpret_cast<int32_t*>(take(U * sizeof(int32_t)));
  L.cimg = take(U * (size_t)3 * kTileBytes);
  L.mv0 = reinterpret_cast<float*>(take(U * (size_t)kDP * sizeof(float)));
  return off;
}

__device__ __forceinline__ bool is_protected(int t, int T, int W, int sink, int keep_window) {
  return t < sink || (keep_window && t >= T - W);
}

// eight bf16 of a 16-byte chunk as floats
__device__ __forceinline__ void unpack8(const uint4& w, float (&f)[8]) {
  const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 v = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&x[i]));
    f[2 * i] = v.x;
    f[2 * i + 1] = v.y;
  }
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 128;" ::: "memory"); }
// whether v holds in all 128 threads of the first epilogue group (barrier 1)
__device__ __forceinline__ bool epi_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

// Pipeline wait that gives up after `polls` polls: records the timeout once
// and raises the CTA's abort flag so that no other role waits on.
__device__ __forceinline__ bool pwait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, void* ws, int u,
                                      uint32_t polls) {
  if (*abort_flag) return false;
  if (mbar_wait(bar, parity, polls)) return true;
  *abort_flag = 1;
  record_error(ws, MKV_ERR_TIMEOUT, u);
  return false;
}

// After an abort, before a CTA frees its tensor memory and exits: wait (with
// the full poll limit) for the last tile copy issued into each of the kS
// stages, for the window-query copy if one was issued, and for the MMA
// thread's final commit (every MMA it issued has completed, so none still
// reads shared memory or writes TMEM).  `issued` tiles went out in order,
// tile i into stage i % kS.
__device__ __forceinline__ void drain_after_abort(uint64_t* full, int kS, int issued, uint64_t* qfull,
                                                  uint64_t* mma_done) {
  for (int st = 0; st < kS; ++st) {
    const int last = issued - 1 - ((issued - 1 - st) % kS + kS) % kS;  // largest i < issued with i % kS == st
    if (last >= 0 && last % kS == st) (void)mbar_wait(&full[st], (last / kS) & 1);
  }
  if (qfull != nullptr) (void)mbar_wait(qfull, 0);
  (void)mbar_wait(mma_done, 0);
}

struct TcArgs {
  int n_rows;  // rows of each unit's slab that take part
  int chunk;   // rows per CTA (multiple of kTok)
  int n_chunks;
  int D, RW, RWb, W, T, causal, sink, keep_window, pool;
  float qscale;  // scale * log2(e)
  float tau;
  float* rowpart;
  float* mrec;  // moment records, [units][n_chunks][rec]
  const float* s_in;
  float* s_out;
  float* diag;
  const uint8_t* cimg;  // [units][3][128 x 128] operand image of C0'
  const float* mv0;     // [units][kDP]
  void* ws;
  uint32_t polls;  // poll limit of the pipeline waits
};

// --------------------------------------------------------------- stats_tc
// Window-row statistics and chunk moments of the prompt.
__global__ void __launch_bounds__(kStatsThreads, 1)
    stats_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
             const __grid_constant__ CUtensorMap tmQ) {
  constexpr int kS = 2;
  constexpr uint32_t kTmemCols = 512;
  constexpr int cS = 256, cSum = 384;  // TMEM columns of V^T K and the sums
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = sm;                        // [kS][128 x 128]
  uint8_t* sV = sm + kS * kTileBytes;      // [kS][128 x 128]
  uint8_t* sQ = sm + 2 * kS * kTileBytes;  // [2 boxes][RWb*128 rows][128 B]
  uint8_t* sOnes = sQ + 2 * 2 * kBoxBytes;  // [2 boxes][16 rows][128 B] of bf16 1.0
  __shared__ __align__(8) uint64_t full[kS], empty[kS], lfull, lempty, qfull, sdone;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued;
  __shared__ float sum_k[kDP], sum_v[kDP];
  __shared__ float s_m1[2][128], s_l1[2][128];  // the second epilogue group's row stats

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  const int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;
  const int RWb = p.RWb;
  volatile int* abrt = &abort_flag;
  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);  // the stage is free once its MMAs have completed
    }
    mbar_init(&lfull, 1);
    mbar_init(&lempty, 8);
    mbar_init(&qfull, 1);
    mbar_init(&sdone, 1);
    abort_flag = 0;
    s_issued = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, kTmemCols);
  if (warp >= 2 && warp < 6) {  // the ones operand of the column sums K^T 1 and V^T 1
    for (int i = tid - 64; i < 2 * 16 * 128 / 16; i += 128)
      reinterpret_cast<uint4*>(sOnes)[i] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {  // ---- producer
      mbar_arrive_expect_tx(&qfull, 2u * RWb * kBoxBytes);
      for (int bx = 0; bx < 2; ++bx) tma_load_3d(sQ + bx * RWb * kBoxBytes, &tmQ, bx * 64, 0, u, &qfull);
      for (int i = 0; i < min(kPF, n_tiles); ++i)
        for (int bx = 0; bx < 2; ++bx) {
          tma_prefetch_3d(&tmK, bx * 64, t_begin + i * kTok, u);
          tma_prefetch_3d(&tmV, bx * 64, t_begin + i * kTok, u);
        }
      for (int i = 0; i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS;
        if (kPF > 0 && i + kPF < n_tiles)
          for (int bx = 0; bx < 2; ++bx) {
            tma_prefetch_3d(&tmK, bx * 64, t_begin + (i + kPF) * kTok, u);
            tma_prefetch_3d(&tmV, bx * 64, t_begin + (i + kPF) * kTok, u);
          }
        if (j >= 1 && !pwait(&empty[s], (j - 1) & 1, abrt, p.ws, u, p.polls)) break;
        mbar_arrive_expect_tx(&full[s], 2u * kTileBytes);
        for (int bx = 0; bx < 2; ++bx) {
          tma_load_3d(sK + s * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[s]);
          tma_load_3d(sV + s * kTileBytes + bx * kBoxBytes, &tmV, bx * 64, t_begin + i * kTok, u, &full[s]);
        }
        s_issued = i + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---- MMA issuer
      const uint32_t idL = idesc_bf16(128, 128, 0, 0);  // logits: rows x tokens, both K-major
      const uint32_t idS = idesc_bf16(128, 128, 1, 1);  // V^T K: both MN-major (reduction over tokens)
      const uint32_t id1 = idesc_bf16(128, 16, 1, 0);   // X^T 1: X MN-major, ones K-major
      const uint32_t aQ = smem_addr(sQ), a1 = smem_addr(sOnes);
      const bool ok = pwait(&qfull, 0, abrt, p.ws, u, p.polls);
      for (int i = 0; ok && i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS;
        if (!pwait(&full[s], j & 1, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        const uint32_t aK = smem_addr(sK + s * kTileBytes), aV = smem_addr(sV + s * kTileBytes);
        if (i >= 1 && !pwait(&lempty, (i - 1) & 1, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        for (int rb = 0; rb < RWb; ++rb)
          for (int kk = 0; kk < 8; ++kk) {
            const uint64_t dq =
                sdesc_sw128(aQ + (kk >> 2) * RWb * kBoxBytes + rb * kBoxBytes + (kk & 3) * 32, 16, 1024);
            const uint64_t dk = sdesc_sw128(aK + (kk >> 2) * kBoxBytes + (kk & 3) * 32, 16, 1024);
            umma_bf16(tm + rb * 128, dq, dk, idL, kk > 0 ? 1u : 0u);
          }
        umma_commit(&lfull);
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t dv = sdesc_sw128(aV + kk * 2048, kBoxBytes, 1024);
          const uint64_t dk = sdesc_sw128(aK + kk * 2048, kBoxBytes, 1024);
          const uint64_t d1 = sdesc_sw128(a1 + (kk >> 2) * 2048 + (kk & 3) * 32, 16, 1024);
          const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
          umma_bf16(tm + cS, dv, dk, idS, acc);
          umma_bf16(tm + cSum, dk, d1, id1, acc);       // column sums of K (lane = key dim)
          umma_bf16(tm + cSum + 16, dv, d1, id1, acc);  // column sums of V (lane = value dim)
        }
        umma_commit(&empty[s]);
      }
      umma_commit(&sdone);
    }
  } else {
    // ---- epilogue: group 0 = warps 2..5 (tokens 0..63 of a tile), group 1 =
    // warps 6..9 (tokens 64..127); TMEM lane quarter qd = warp % 4
    const int grp = (warp - 2) >> 2;
    const int et = tid - 64 - grp * 128, qd = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    int tmax_vis[2];
    for (int rb = 0; rb < 2; ++rb) {
      const int r = rb * 128 + qd * 32 + lane;  // window row of this thread
      tmax_vis[rb] = p.causal ? p.T - p.W + r % p.W : 0x7fffffff;
    }
    const int t_safe = p.causal ? p.T - p.W : 0x7fffffff;  // tokens every window row sees
    for (int i = 0; i < n_tiles; ++i) {
      if (!pwait(&lfull, i & 1, abrt, p.ws, u, p.polls)) break;
      tc_fence_after();
      const int tt0 = t_begin + i * kTok;
      const bool fast = tt0 + kTok <= t_end && tt0 + kTok - 1 <= t_safe;  // no masking in this tile
      // rb runs over a constant range (guarded by RWb), so that m, l and
      // tmax_vis stay in registers
#pragma unroll
      for (int rb = 0; rb < 2; ++rb) {
        if (rb >= RWb) break;
        for (int c0 = grp * 64; c0 < grp * 64 + 64; c0 += 32) {
          float x[32];
          tmem_ld32(tm + lane_base + rb * 128 + c0, x);
          const int t0 = tt0 + c0;
          float mx = -INFINITY;
          if (fast) {
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) {
              x[jj] *= p.qscale;
              mx = fmaxf(mx, x[jj]);
            }
          } else {
#pragma unroll
            for (int jj = 0; jj < 32; ++jj) {
              const int t = t0 + jj;
              x[jj] = (t < t_end && t <= tmax_vis[rb]) ? x[jj] * p.qscale : -INFINITY;
              mx = fmaxf(mx, x[jj]);
            }
          }
          {
            const float mn = fmaxf(m[rb], mx);
            if (mn != -INFINITY) {
              float acc = 0.f;
#pragma unroll
              for (int jj = 0; jj < 32; ++jj) acc += fast_exp2(x[jj] - mn);
              l[rb] = l[rb] * fast_exp2(m[rb] - mn) + acc;
              m[rb] = mn;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&lempty);
    }
    {  // merge the two groups' (max, sum) of each row
      if (grp == 1)
#pragma unroll
        for (int rb = 0; rb < 2; ++rb) {
          if (rb < RWb) {
            s_m1[rb][qd * 32 + lane] = m[rb];
            s_l1[rb][qd * 32 + lane] = l[rb];
          }
        }
      asm volatile("bar.sync 2, 256;" ::: "memory");
      if (grp == 0)
#pragma unroll
        for (int rb = 0; rb < 2; ++rb) {
          if (rb >= RWb) break;
          const int r = rb * 128 + qd * 32 + lane;
          const float m1 = s_m1[rb][qd * 32 + lane], l1 = s_l1[rb][qd * 32 + lane];
          const float M = fmaxf(m[rb], m1);
          float L = 0.f;
          if (M != -INFINITY) {
            if (m[rb] != -INFINITY) L += l[rb] * fast_exp2(m[rb] - M);
            if (m1 != -INFINITY) L += l1 * fast_exp2(m1 - M);
          }
          if (r < p.RW) {
            float* rp = p.rowpart + (((size_t)u * p.n_chunks + chunk) * p.RW + r) * 2;
            rp[0] = M;
            rp[1] = L;
          }
        }
    }
    if (grp == 0) {
    // uniform over the group: after an abort the MMAs may still write TMEM,
    // so it is not read and the chunk's record is left empty
    const bool got = epi_all(pwait(&sdone, 0, abrt, p.ws, u, p.polls));
    float* rec = p.mrec + ((size_t)u * p.n_chunks + chunk) * rec_floats(p.D);
    const float nc = got ? static_cast<float>(max(0, t_end - t_begin)) : 0.f;
    if (got) {
    tc_fence_after();
    {
      float x[32];
      tmem_ld32(tm + lane_base + cSum, x);  // [0]: sum of K's column (this lane), [16]: of V's
      sum_k[qd * 32 + lane] = x[0];
      sum_v[qd * 32 + lane] = x[16];
    }
    epi_sync();
    const float inv_nc = nc > 0.f ? 1.f / nc : 0.f;
    const int a = qd * 32 + lane;  // value dim = TMEM lane
    // centred co-moment rows staged 32 columns at a time through the (now
    // free) K stage, so that the record is written in coalesced rows
    float* stg = reinterpret_cast<float*>(sK);  // [128][33]
    for (int c0 = 0; c0 < kDP; c0 += 32) {
      float srow[32];
      tmem_ld32(tm + lane_base + cS + c0, srow);
#pragma unroll
      for (int jj = 0; jj < 32; ++jj) stg[a * 33 + jj] = srow[jj] - sum_v[a] * sum_k[c0 + jj] * inv_nc;
      epi_sync();
      if (nc > 0.f)
        for (int idx = et; idx < 128 * 32; idx += 128) {
          const int r = idx >> 5, c = c0 + (idx & 31);
          if (r < p.D && c < p.D) rec[4 + 2 * p.D + (size_t)r * p.D + c] = stg[r * 33 + (idx & 31)];
        }
      epi_sync();
    }
    if (a < p.D) {
      rec[4 + a] = nc > 0.f ? sum_k[a] / nc : 0.f;
      rec[4 + p.D + a] = nc > 0.f ? sum_v[a] / nc : 0.f;
    }
    } else if (et < 4 + 2 * p.D) {
      rec[et] = 0.f;  // an empty record: n = 0, zero means
    }
    if (et == 0) rec[0] = nc;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (abort_flag) {  // uniform: every role has left its loop
    if (tid == 0) drain_after_abort(full, kS, s_issued, &qfull, &sdone);
    __syncthreads();
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, kTmemCols);
  }
}

// -------------------------------------------------------------- scores_tc
__global__ void __launch_bounds__(kStatsThreads, 1)
    scores_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ) {
  constexpr int kS = 3;
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = sm;                    // [kS][128 x 128]
  uint8_t* sQ = sm + kS * kTileBytes;  // [2 boxes][RWb*128][128 B]
  __shared__ __align__(8) uint64_t full[kS], empty[kS], lfull[2], lempty[2], qfull, mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued;
  __shared__ __align__(16) float s_b[256];  // log2(1 / l_r) - m_r (-inf for padding rows)
  __shared__ int s_wi[256];                   // window index of row r (r mod W)

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  const int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;
  const int RWb = p.RWb, RWp = RWb * 128;
  volatile int* abrt = &abort_flag;

  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&lfull[i], 1);
      mbar_init(&lempty[i], 4);
    }
    mbar_init(&qfull, 1);
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    s_issued = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;
  // The prompt and the queries were complete before stats_tc passed its own
  // wait, so the copies need not wait for stats_tc; its row statistics do.
  if (warp != 0) {
    grid_dependency_wait();
    grid_launch_dependents();
  }

  if (warp == 0) {
    if (lane == 0) {
      mbar_arrive_expect_tx(&qfull, 2u * RWb * kBoxBytes);
      for (int bx = 0; bx < 2; ++bx) tma_load_3d(sQ + bx * RWb * kBoxBytes, &tmQ, bx * 64, 0, u, &qfull);
      for (int i = kS; i < min(kS + kPF, n_tiles); ++i)
        for (int bx = 0; bx < 2; ++bx) tma_prefetch_3d(&tmK, bx * 64, t_begin + i * kTok, u);
      for (int i = 0; i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS;
        if (kPF > 0 && i + kS + kPF < n_tiles)
          for (int bx = 0; bx < 2; ++bx) tma_prefetch_3d(&tmK, bx * 64, t_begin + (i + kS + kPF) * kTok, u);
        if (j >= 1 && !pwait(&empty[s], (j - 1) & 1, abrt, p.ws, u, p.polls)) break;
        mbar_arrive_expect_tx(&full[s], kTileBytes);
        for (int bx = 0; bx < 2; ++bx)
          tma_load_3d(sK + s * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[s]);
        s_issued = i + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id = idesc_bf16(128, RWp, 0, 0);  // tokens x window rows, both K-major
      const uint32_t aQ = smem_addr(sQ);
      const bool ok = pwait(&qfull, 0, abrt, p.ws, u, p.polls);
      for (int i = 0; ok && i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS, b = i & 1;
        if (!pwait(&full[s], j & 1, abrt, p.ws, u, p.polls)) break;
        if (i >= 2 && !pwait(&lempty[b], ((i >> 1) - 1) & 1, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        const uint32_t aK = smem_addr(sK + s * kTileBytes);
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t dk = sdesc_sw128(aK + (kk >> 2) * kBoxBytes + (kk & 3) * 32, 16, 1024);
          const uint64_t dq = sdesc_sw128(aQ + (kk >> 2) * RWb * kBoxBytes + (kk & 3) * 32, 16, 1024);
          umma_bf16(tm + b * 256, dk, dq, id, kk > 0 ? 1u : 0u);
        }
        umma_commit(&lfull[b]);
        umma_commit(&empty[s]);
      }
      umma_commit(&mma_done);  // every MMA issued has completed
    }
  } else {
    // two epilogue groups (warps 2..5 and 6..9) take alternate tiles; group g
    // always reads TMEM buffer g
    const int grp = (warp - 2) >> 2, qd = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    // merged row statistics of every window row
    for (int r = tid - 64; r < RWp; r += 256) {
      float M = -INFINITY, Lsum = 0.f;
      if (r < p.RW) {
        for (int c = 0; c < p.n_chunks; ++c)
          M = fmaxf(M, p.rowpart[(((size_t)u * p.n_chunks + c) * p.RW + r) * 2]);
        if (M != -INFINITY)
          for (int c = 0; c < p.n_chunks; ++c) {
            const float* rp = p.rowpart + (((size_t)u * p.n_chunks + c) * p.RW + r) * 2;
            if (rp[0] != -INFINITY) Lsum += rp[1] * fast_exp2(rp[0] - M);
          }
      }
      s_b[r] = (Lsum > 0.f) ? -log2f(Lsum) - M : -INFINITY;
      s_wi[r] = r % p.W;
    }
    asm volatile("bar.sync 1, 256;" ::: "memory");
    const int t_safe = p.causal ? p.T - p.W : 0x7fffffff;  // tokens every window row sees
    for (int i = grp; i < n_tiles; i += 2) {
      const int b = i & 1;
      if (!pwait(&lfull[b], (i >> 1) & 1, abrt, p.ws, u, p.polls)) break;
      tc_fence_after();
      const int t = t_begin + i * kTok + qd * 32 + lane;  // token of this thread (TMEM lane)
      const bool fast = t <= t_safe;  // every window row sees this token
      float acc = 0.f;
      for (int c0 = 0; c0 < RWp; c0 += 32) {
        float x[32];
        tmem_ld32(tm + lane_base + b * 256 + c0, x);
        if (fast) {  // p = 2^(x qscale + b_r); padding rows have b_r = -inf
#pragma unroll
          for (int jj = 0; jj < 32; jj += 4) {
            const float4 b4 = *reinterpret_cast<const float4*>(s_b + c0 + jj);
            acc += fast_exp2(fmaf(x[jj], p.qscale, b4.x)) + fast_exp2(fmaf(x[jj + 1], p.qscale, b4.y)) +
                   fast_exp2(fmaf(x[jj + 2], p.qscale, b4.z)) + fast_exp2(fmaf(x[jj + 3], p.qscale, b4.w));
          }
        } else {
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) {
            const int r = c0 + jj;
            if (t <= p.T - p.W + s_wi[r]) acc += fast_exp2(fmaf(x[jj], p.qscale, s_b[r]));
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&lempty[b]);
      for (int o = 1; o < p.pool; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);  // aligned chunks
      if (t < t_end) {
        p.s_out[(size_t)u * p.T + t] = acc;
        if (p.diag) p.diag[(size_t)u * p.T + t] = acc;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // the MMA thread's final commit, and after an abort the copies in flight
  if (tid == 0) drain_after_abort(full, kS, abort_flag ? s_issued : 0, abort_flag ? &qfull : nullptr, &mma_done);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// ------------------------------------------------------------ residual_tc
__global__ void __launch_bounds__(kStatsThreads, 1)
    residual_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV) {
  constexpr int kS = 2;
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = sm;                        // [kS][128 x 128]
  uint8_t* sV = sm + kS * kTileBytes;      // [kS][128 x 128]
  uint8_t* sC = sm + 2 * kS * kTileBytes;  // [3 parts][128 x 128]: C0' = hi + mid + lo
  __shared__ __align__(8) uint64_t full[kS], empty[kS], yfull[2], yempty[2], cfull, mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued;
  __shared__ float s_mv[kDP];

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  const int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;
  volatile int* abrt = &abort_flag;
  const int D = p.D;

  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1 + 4);  // MMA commit + the 4 epilogue warps (value rows)
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&yfull[i], 1);
      mbar_init(&yempty[i], 4);
    }
    mbar_init(&cfull, 1);
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    mbar_fence_init();
    // the first stages' copies go out before the dependency wait: the prompt
    // was complete before the compression began
    for (int i = kS; i < min(kS + kPF, n_tiles); ++i)
      for (int bx = 0; bx < 2; ++bx) {
        tma_prefetch_3d(&tmK, bx * 64, t_begin + i * kTok, u);
        tma_prefetch_3d(&tmV, bx * 64, t_begin + i * kTok, u);
      }
    for (int i = 0; i < min(kS, n_tiles); ++i) {
      mbar_arrive_expect_tx(&full[i], 2u * kTileBytes);
      for (int bx = 0; bx < 2; ++bx) {
        tma_load_3d(sK + i * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[i]);
        tma_load_3d(sV + i * kTileBytes + bx * kBoxBytes, &tmV, bx * 64, t_begin + i * kTok, u, &full[i]);
      }
    }
    s_issued = min(kS, n_tiles);
  }
  if (warp == 1) tmem_alloc(&tmem_base, 256);
  if (D < kDP) {  // no second box of key dims: that part of the operand image is zero
    for (int i = tid; i < 3 * kBoxBytes / 16; i += kStatsThreads)
      reinterpret_cast<uint4*>(sC + (i / (kBoxBytes / 16)) * kTileBytes + kBoxBytes)[i % (kBoxBytes / 16)] =
          make_uint4(0u, 0u, 0u, 0u);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
  }
  grid_dependency_wait();
  grid_launch_dependents();
  if (tid == 0) {  // C0' as rset_kernel left it: three bf16 parts in the operand layout
    const uint32_t part_bytes = D < kDP ? kBoxBytes : kTileBytes;
    mbar_arrive_expect_tx(&cfull, 3 * part_bytes);
    for (int part = 0; part < 3; ++part)
      bulk_g2s(sC + part * kTileBytes, p.cimg + ((size_t)u * 3 + part) * kTileBytes, part_bytes, &cfull);
  }
  if (tid < kDP) s_mv[tid] = p.mv0[(size_t)u * kDP + tid];
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;
  const float scale = rsqrtf(static_cast<float>(D));

  if (warp == 0) {
    if (lane == 0) {
      for (int i = kS; i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS;
        if (kPF > 0 && i + kPF < n_tiles)
          for (int bx = 0; bx < 2; ++bx) {
            tma_prefetch_3d(&tmK, bx * 64, t_begin + (i + kPF) * kTok, u);
            tma_prefetch_3d(&tmV, bx * 64, t_begin + (i + kPF) * kTok, u);
          }
        if (!pwait(&empty[s], (j - 1) & 1, abrt, p.ws, u, p.polls)) break;
        mbar_arrive_expect_tx(&full[s], 2u * kTileBytes);
        for (int bx = 0; bx < 2; ++bx) {
          tma_load_3d(sK + s * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[s]);
          tma_load_3d(sV + s * kTileBytes + bx * kBoxBytes, &tmV, bx * 64, t_begin + i * kTok, u, &full[s]);
        }
        s_issued = i + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id = idesc_bf16(128, 128, 0, 0);
      const uint32_t aC = smem_addr(sC);
      const bool ok = pwait(&cfull, 0, abrt, p.ws, u, p.polls);
      for (int i = 0; ok && i < n_tiles; ++i) {
        const int s = i % kS, j = i / kS, b = i & 1;
        if (!pwait(&full[s], j & 1, abrt, p.ws, u, p.polls)) break;
        if (i >= 2 && !pwait(&yempty[b], ((i >> 1) - 1) & 1, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        const uint32_t aK = smem_addr(sK + s * kTileBytes);
        for (int part = 0; part < 3; ++part)
          for (int kk = 0; kk < 8; ++kk) {
            const uint64_t dk = sdesc_sw128(aK + (kk >> 2) * kBoxBytes + (kk & 3) * 32, 16, 1024);
            const uint64_t dc =
                sdesc_sw128(aC + part * kTileBytes + (kk >> 2) * kBoxBytes + (kk & 3) * 32, 16, 1024);
            umma_bf16(tm + b * 128, dk, dc, id, (part > 0 || kk > 0) ? 1u : 0u);
          }
        umma_commit(&yfull[b]);
        umma_commit(&empty[s]);
      }
      umma_commit(&mma_done);  // every MMA issued has completed
    }
  } else {
    // two epilogue groups (warps 2..5 and 6..9) take alternate tiles; group g
    // always reads TMEM buffer g
    const int grp = (warp - 2) >> 2, qd = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    const int row = qd * 32 + lane;  // token within the tile = TMEM lane
    for (int i = grp; i < n_tiles; i += 2) {
      const int s = i % kS, j = i / kS, b = i & 1;
      if (!pwait(&yfull[b], (i >> 1) & 1, abrt, p.ws, u, p.polls)) break;
      if (!pwait(&full[s], j & 1, abrt, p.ws, u, p.polls)) break;
      tc_fence_after();
      const uint8_t* tv = sV + s * kTileBytes;
      float ss = 0.f;
      for (int c0 = 0; c0 < kDP; c0 += 32) {
        float y[32];
        tmem_ld32(tm + lane_base + b * 128 + c0, y);
        if (c0 < D) {
#pragma unroll
          for (int jj = 0; jj < 32; jj += 8) {
            const uint4 raw = *reinterpret_cast<const uint4*>(tv + swz_off(row, c0 + jj, kTok));
            const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 vv = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w[e]));
              const int c = c0 + jj + 2 * e;
              const float r0 = vv.x - s_mv[c] - scale * y[jj + 2 * e];
              const float r1 = vv.y - s_mv[c + 1] - scale * y[jj + 2 * e + 1];
              ss = fmaf(r0, r0, fmaf(r1, r1, ss));
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&yempty[b]);
        mbar_arrive(&empty[s]);
      }
      const int t = t_begin + i * kTok + row;
      if (t < t_end) {
        const float v =
            is_protected(t, p.T, p.W, p.sink, p.keep_window) ? 0.f : p.s_in[(size_t)u * p.T + t] * sqrtf(ss);
        p.s_out[(size_t)u * p.T + t] = v;
        if (p.diag) p.diag[(size_t)u * p.T + t] = v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // the MMA thread's final commit, and after an abort the copies in flight
  if (tid == 0) drain_after_abort(full, kS, abort_flag ? s_issued : 0, &cfull, &mma_done);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 256);
  }
}

// ----------------------------------------------------------------- select
// One cluster of kSelCL CTAs per selection group -- a unit, or with the
// adaptive budget the hs KV heads of a batch item, whose (head, position)
// pairs f = h * T + t are ranked together.  R = protected + the k highest
// keys among the other pairs (ties to the lower f), written ascending, with
// each unit's count and first slot.
// Exclusive block-wide prefix sum of one int per thread; *total gets the sum.
__device__ __forceinline__ int block_excl_sum(int v, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
    int xw = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(kFull, xw, o);
      if (lane >= o) xw += y;
    }
    wsum[lane] = xw - w;
    if (lane == 31) *total = xw;
  }
  __syncthreads();
  const int r = wsum[warp] + x - v;
  __syncthreads();  // wsum is reused by the next call
  return r;
}

struct SelectArgs {
  const float* scores;  // [units][T]
  int T, W, B, sink, keep_window;
  int32_t* idx;          // [groups][hs * B] selection lists, h * T + position, ascending (workspace)
  int32_t* diag_idx;     // optional copy
  int smem_keys;  // keys of a CTA's range that the dynamic shared memory holds
  int hs;         // units per selection group (1: one unit; > 1: the KV heads of a batch item)
  const int32_t* cand;  // optional [units][Tc] ascending candidate positions per unit (null: all T)
  int Tc;               // entries per unit taking part: T, or the candidate lists' length
  int32_t* cnt;    // optional [units] rows retained per unit
  int32_t* hbeg;   // optional [units] the unit's first slot in idx
};

constexpr int kSelCL = 8;  // CTAs per selection group (one cluster), each over a contiguous range of pairs
constexpr int kSelSmemKeys = 49152;  // keys of a CTA's range cached in shared memory (192 KB)
constexpr int kMaxHs = 64;           // KV heads of a batch item with the adaptive budget

__global__ void __cluster_dims__(kSelCL, 1, 1) __launch_bounds__(kSelThreads, 2) select_kernel(const SelectArgs a) {
  __shared__ uint32_t hist[2][256];   // this CTA's histogram, double-buffered by pass parity (read remotely)
  __shared__ uint32_t whist[8][256];  // private histograms for groups of 4 warps (less atomic contention)
  __shared__ uint32_t ghist[256];     // the cluster's histogram
  __shared__ int wsum[32];
  __shared__ int tot;
  __shared__ uint32_t s_prefix;
  __shared__ int s_need;
  __shared__ int ex_cnt[2];  // this CTA's ties and certain selections (protected or above the threshold)
  __shared__ int s_before[2];
  __shared__ int s_hstart[kMaxHs + 1];  // first slot of each head in the group's selection list
  __shared__ int s_hcnt[kMaxHs];        // this CTA's selections per head (read remotely)
  grid_dependency_wait();
  grid_launch_dependents();
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int grp = blockIdx.x / kSelCL, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = a.T, W = a.W, hs = a.hs;
  // entries f = h * Tc + j of the group stand for (head h, position t), t = j
  // or the candidate cand[h][j]; either way f ascending is (h, t) ascending
  const int Tc = a.Tc;
  const int N = hs * Tc;
  const int per = (N + kSelCL - 1) / kSelCL;
  const int r0 = min(N, rank * per), r1 = min(N, r0 + per);
  const float* sc = a.scores + (size_t)grp * hs * T;  // the group's units are consecutive
  const int32_t* cand = a.cand ? a.cand + (size_t)grp * N : nullptr;
  auto pos_of = [&](int f, int& h) -> int {  // (head, position) of entry f
    h = hs == 1 ? 0 : f / Tc;
    const int j = f - h * Tc;
    return cand ? cand[f] : j;
  };
  // >= 0 (validated), < candidates
  const int k = hs * (a.B - protected_count(T, W, a.sink, a.keep_window));

  // The CTA's keys are cached in shared memory when they fit (protected
  // positions hold key 0; every other position's key is at least 1, whatever
  // the bits of its score, so at most k of them are ever selected); larger
  // ranges are read from global memory on every pass.
  extern __shared__ uint32_t ks[];
  const int nk = r1 - r0;
  const bool cached = nk <= a.smem_keys;
  auto key_of = [&](int f) -> uint32_t {
    int h;
    const int t = pos_of(f, h);
    return is_protected(t, T, W, a.sink, a.keep_window) ? 0u : max(1u, float_key(sc[(size_t)h * T + t]));
  };
  auto key_at = [&](int f) -> uint32_t {  // 0 for protected positions
    return cached ? ks[f - r0] : key_of(f);
  };
  for (int h = tid; h < hs; h += kSelThreads) s_hcnt[h] = 0;
  if (cached)
    for (int i = tid; i < nk; i += kSelThreads) ks[i] = key_of(r0 + i);
  __syncthreads();
  // thread tid owns the contiguous positions [t0, t1) in the ordered passes
  const int E = (nk + kSelThreads - 1) / kSelThreads;
  const int t0 = min(r1, r0 + tid * E), t1 = min(r1, t0 + E);

  uint32_t prefix = 0, pmask = 0;
  int need = k;
  if (k > 0) {
    for (int pass = 0; pass < 4; ++pass) {
      const int shift = 24 - 8 * pass;
      for (int i = tid; i < 8 * 256; i += kSelThreads) (&whist[0][0])[i] = 0;
      __syncthreads();
      uint32_t* wh = whist[warp & 7];
#pragma unroll 4
      for (int i = tid; i < nk; i += kSelThreads) {
        const uint32_t key = key_at(r0 + i);
        if (key != 0u && (key & pmask) == prefix) atomicAdd(&wh[(key >> shift) & 255u], 1u);
      }
      __syncthreads();
      for (int i = tid; i < 256; i += kSelThreads) {
        uint32_t c = 0;
#pragma unroll
        for (int g = 0; g < 8; ++g) c += whist[g][i];
        hist[pass & 1][i] = c;
      }
      cluster.sync();  // every CTA's histogram of this pass is complete
      for (int i = tid; i < 256; i += kSelThreads) {
        uint32_t c = 0;
#pragma unroll
        for (int r = 0; r < kSelCL; ++r) c += cluster.map_shared_rank(&hist[pass & 1][0], r)[i];
        ghist[i] = c;
      }
      __syncthreads();
      if (warp == 0) {  // the digit where the descending cumulative count reaches `need`
        int cnt[8], tot8 = 0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          cnt[e] = static_cast<int>(ghist[255 - (lane * 8 + e)]);
          tot8 += cnt[e];
        }
        int incl = tot8;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        const int excl = incl - tot8;
        if (excl < need && incl >= need) {
          int cum = excl, e = 0;
          for (; e < 7; ++e) {
            if (cum + cnt[e] >= need) break;
            cum += cnt[e];
          }
          s_need = need - cum;
          s_prefix = prefix | (static_cast<uint32_t>(255 - (lane * 8 + e)) << shift);
        }
      }
      __syncthreads();
      need = s_need;
      prefix = s_prefix;
      pmask |= 255u << shift;
    }
  }
  // per-thread counts: protected or above the threshold key (certain), and
  // ties with it; scanned over the block, then over the cluster's ranks
  int n_tie = 0, n_sure = 0;
  for (int t = t0; t < t1; ++t) {
    const uint32_t key = key_at(t);
    if (key == 0u) {
      ++n_sure;  // protected
    } else if (k > 0) {
      n_sure += key > prefix ? 1 : 0;
      n_tie += key == prefix ? 1 : 0;
    }
  }
  const int tie_excl = block_excl_sum(n_tie, wsum, &tot);
  if (tid == 0) ex_cnt[0] = tot;
  const int sure_excl = block_excl_sum(n_sure, wsum, &tot);
  if (tid == 0) ex_cnt[1] = tot;
  (void)sure_excl;
  cluster.sync();
  if (tid == 0) {
    int ties_before = 0, sel_before = 0;
    for (int r = 0; r < rank; ++r) {
      const int* rc = cluster.map_shared_rank(ex_cnt, r);
      const int nt = rc[0], ns = rc[1];
      const int take = min(max(need - ties_before, 0), nt);  // this rank's ties that are selected
      sel_before += ns + take;
      ties_before += nt;
    }
    s_before[0] = ties_before;
    s_before[1] = sel_before;
  }
  __syncthreads();
  const int cta_ties_before = s_before[0], cta_sel_before = s_before[1];
  // this thread's selections: its certain ones and the ties that still fit
  int tb = cta_ties_before + tie_excl;
  const int my_sel = n_sure + min(max(need - tb, 0), n_tie);
  const int sel_excl = block_excl_sum(my_sel, wsum, &tot);
  int o = cta_sel_before + sel_excl;
  const int n_sel = hs * a.B;  // the group's selections (protected included)
  int32_t* out = a.idx + (size_t)grp * n_sel;
  int cur_h = 0, cur_n = 0;  // this thread's run of selections in one head (ranges rarely span two)
  for (int t = t0; t < t1; ++t) {
    const uint32_t key = key_at(t);
    bool sel = true;  // protected
    if (key != 0u) {
      const bool tie = k > 0 && key == prefix;
      sel = (k > 0 && key > prefix) || (tie && tb < need);
      tb += tie ? 1 : 0;
    }
    if (sel) {
      if (o < n_sel) {  // stored as h * T + position
        int h;
        const int pt = pos_of(t, h);
        out[o] = h * T + pt;
        if (a.diag_idx) a.diag_idx[(size_t)grp * n_sel + o] = h * T + pt;
        if (h != cur_h) {
          if (cur_n) atomicAdd(&s_hcnt[cur_h], cur_n);
          cur_h = h;
          cur_n = 0;
        }
        ++cur_n;
      }
      ++o;
    }
  }
  if (hs > 1) {
    // each head's slots are a contiguous run of the ascending list, as long
    // as the head's selections in all CTAs of the cluster
    if (cur_n) atomicAdd(&s_hcnt[cur_h], cur_n);
    cluster.sync();
    if (tid < hs) {
      int c = 0;
#pragma unroll
      for (int r = 0; r < kSelCL; ++r) c += cluster.map_shared_rank(s_hcnt, r)[tid];
      s_hstart[tid + 1] = c;
    }
    __syncthreads();
    if (tid == 0) {
      s_hstart[0] = 0;
      for (int h = 0; h < hs; ++h) s_hstart[h + 1] += s_hstart[h];
    }
  } else if (tid == 0) {
    s_hstart[0] = 0;
    s_hstart[1] = a.B;
  }
  __syncthreads();
  if (rank == 0 && tid < hs) {
    const int u = grp * hs + tid, c = s_hstart[tid + 1] - s_hstart[tid];
    if (a.cnt) a.cnt[u] = c;
    if (a.hbeg) a.hbeg[u] = grp * n_sel + s_hstart[tid];
  }
  cluster.sync();  // no CTA leaves while another may still read its shared memory
}

// ------------------------------------------------------------------- rset
// Moments of E = all \ R for the rows R a selection kept, in one kernel per
// stage: the rows are gathered by their list straight into the tensor-core
// operand layout (no dense copy of them), V^T K of them accumulates in TMEM,
// and the epilogue takes their centred co-moment out of the all-token set's.
// The first stage writes C0' as the residual pass's operand image, the final
// one the caller's moments and, from the same tiles, the retained cache.
//
// Grid (CL * D/64, units), clusters of CL CTAs: CTA (rank, kh) takes the row
// tiles rank, rank + CL, ... and the key dims [64 kh, 64 kh + 64); the CL
// partial sums meet through distributed shared memory, each rank finishing
// 128 / CL value dims.  A set of 128..1024 rows is one tile per CTA: the kernel
// is a chain of round trips (list, rows, MMA, exchange), 5-7 us, where the
// dense gather, the per-tile records and their merge took 25-40.
//
// The all-token co-moment is the multi-way Chan merge of the chunk records,
// taken about the first chunk's means x0 so that no global mean is needed first:
//   M = sum_ch [M_ch + n_ch d_ch d_ch^T] - n dbar dbar^T,  d_ch = mu_ch - x0,
//   dbar = sum_ch n_ch d_ch / n,  mu = x0 + dbar.
// It is merged before the dependency wait, while the selection runs: the
// records are stats_tc's, complete before the selection's predecessor (which
// the selection has waited for when this kernel may start) began.
// R's centred record is then removed with the reverse pairwise formula.
constexpr int kRsThreads = 256;
constexpr int kFinCH = 32;              // chunk records staged per pass
constexpr int kRsRed = 64 + 4;          // row stride of a CTA's partial sums (floats)
constexpr size_t kRsSmem = 1024 + kBoxBytes + kTileBytes;  // one K half, one V tile

struct RsetArgs {
  Layout L;
  const __nv_bfloat16* K;  // prompt [units][T][D]
  const __nv_bfloat16* V;
  float tau;
  __nv_bfloat16* dst_K;  // final stage: the cache
  __nv_bfloat16* dst_V;
  int dst_cap;
  int32_t *dst_pos, *dst_len, *dst_seen;
  mkv_moments mom;
  void* ws;
  uint32_t polls;
};

__device__ __forceinline__ void cp_async16(void* dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}

template <int CL, bool FINAL>
__global__ void __launch_bounds__(kRsThreads, 2) rset_kernel(const RsetArgs a) {
  constexpr int NI = 8 / CL;       // value dims per thread in the merges (16 apart)
  constexpr int RW = kDP / CL;     // value dims a rank finishes
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = sm;              // [128 rows][64 key dims]
  uint8_t* sV = sm + kBoxBytes;  // [2 boxes][128 rows][64 value dims]
  float* red = reinterpret_cast<float*>(sm);  // [128][kRsRed] this CTA's V^T K (after the tiles)
  __shared__ __align__(8) uint64_t done;
  __shared__ uint32_t tmem_base;
  __shared__ int s_ok;
  __shared__ __align__(16) float s_pk[32][64], s_pv[16][kDP];  // column sums per row group
  __shared__ __align__(16) float s_sk[64], s_sv[kDP];          // this CTA's column sums (read remotely)
  const Layout& L = a.L;
  const int D = L.D, T = L.T;
  const int rank = blockIdx.x % CL, kh = blockIdx.x / CL, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cq = tid % 16, ar = tid / 16;  // merges: columns kh*64 + 4 cq.., value dims rank*RW + ar + 16 i

  if (tid == 0) {
    mbar_init(&done, 1);
    mbar_fence_init();
    s_ok = 1;
  }
  if (warp == 0) tmem_alloc(&tmem_base, 64);

  // ---- the all-token set: this thread's elements of M and its means
  const size_t rf = L.rec;
  const float* recs = L.mpart + (size_t)u * L.n_chunks * rf;
  float n = 0.f, sk[4] = {0.f, 0.f, 0.f, 0.f}, x0k[4] = {0.f, 0.f, 0.f, 0.f};
  float sv[NI], x0v[NI], M[NI][4];
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    sv[i] = x0v[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) M[i][j] = 0.f;
  }
  {
    float* s_n = reinterpret_cast<float*>(sm);  // [kFinCH]
    float* s_mk = s_n + kFinCH;                 // [kFinCH][64]
    float* s_mv = s_mk + kFinCH * 64;           // [kFinCH][RW]
    for (int g0 = 0; g0 < L.n_chunks; g0 += kFinCH) {
      const int nb = min(kFinCH, L.n_chunks - g0);
      if (g0 > 0) __syncthreads();
      constexpr int per = 1 + 16 + RW / 4;  // float4s per record: n, 64 key means, RW value means
#pragma unroll 4
      for (int i = tid; i < nb * per; i += kRsThreads) {
        const int ch = i / per, j = i % per;
        const float* r = recs + (size_t)(g0 + ch) * rf;
        if (j == 0) {
          s_n[ch] = r[0];
        } else if (j <= 16) {
          *reinterpret_cast<float4*>(s_mk + ch * 64 + (j - 1) * 4) =
              *reinterpret_cast<const float4*>(r + 4 + kh * 64 + (j - 1) * 4);
        } else {
          const int c = rank * RW + (j - 17) * 4;
          *reinterpret_cast<float4*>(s_mv + ch * RW + (j - 17) * 4) =
              c < D ? *reinterpret_cast<const float4*>(r + 4 + D + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      __syncthreads();
      if (g0 == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) x0k[j] = s_mk[cq * 4 + j];
#pragma unroll
        for (int i = 0; i < NI; ++i) x0v[i] = s_mv[ar + 16 * i];
      }
#pragma unroll(CL >= 4 ? 8 : 2)
      for (int ch = 0; ch < nb; ++ch) {
        const float* m = recs + (size_t)(g0 + ch) * rf + 4 + 2 * D + kh * 64 + cq * 4;
        float4 m4[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int row = rank * RW + ar + 16 * i;
          m4[i] = row < D ? *reinterpret_cast<const float4*>(m + (size_t)row * D) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const float nc = s_n[ch];
        if (nc > 0.f) {  // an empty record's co-moment is never written
          const float4 k4 = *reinterpret_cast<const float4*>(s_mk + ch * 64 + cq * 4);
          const float dk[4] = {k4.x - x0k[0], k4.y - x0k[1], k4.z - x0k[2], k4.w - x0k[3]};
          n += nc;
#pragma unroll
          for (int j = 0; j < 4; ++j) sk[j] = fmaf(nc, dk[j], sk[j]);
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const float dv = s_mv[ch * RW + ar + 16 * i] - x0v[i];
            sv[i] = fmaf(nc, dv, sv[i]);
            const float mm[4] = {m4[i].x, m4[i].y, m4[i].z, m4[i].w};
#pragma unroll
            for (int j = 0; j < 4; ++j) M[i][j] += mm[j] + nc * dv * dk[j];
          }
        }
      }
    }
  }
  __syncthreads();  // the staged records give way to the row tiles
  if (D < kDP)      // no second box of value dims
    for (int i = tid; i < kBoxBytes / 16; i += kRsThreads)
      reinterpret_cast<uint4*>(sV + kBoxBytes)[i] = make_uint4(0u, 0u, 0u, 0u);
  grid_dependency_wait();
  grid_launch_dependents();

  // ---- row tiles
  const int cnt = L.cnt[u];
  const int32_t* lst = L.idx + L.hbeg[u];
  const int hT = (u % L.hs) * T;  // list entries are h * T + position
  const int n_tiles = (cnt + kTok - 1) / kTok;
  const __nv_bfloat16* Ku = a.K + (size_t)u * T * D + kh * 64;
  const __nv_bfloat16* Vu = a.V + (size_t)u * T * D;
  const uint32_t id = idesc_bf16(128, 64, 1, 1);  // V^T K: both MN-major (reduction over rows)
  const uint32_t aK = smem_addr(sK), aV = smem_addr(sV);
  const int vch = D / 8;  // 16-byte chunks of a value row
  float ks[8], vs[8];     // this thread's column sums: key chunk tid % 8, value chunk tid % 16
#pragma unroll
  for (int j = 0; j < 8; ++j) ks[j] = vs[j] = 0.f;
  int it = 0;
  bool ok = true;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;
  for (int ti = rank; ti < n_tiles; ti += CL, ++it) {
    if (it > 0) {  // the operands are free once their MMAs have completed
      if (tid == 0 && !mbar_wait(&done, (it - 1) & 1, a.polls)) {
        s_ok = 0;
        record_error(a.ws, MKV_ERR_TIMEOUT, u);
      }
      __syncthreads();
      ok = s_ok != 0;
      if (!ok) break;  // uniform: s_ok changes only before a barrier
    }
    const int r0 = ti * kTok;
#pragma unroll
    for (int j = 0; j < 4; ++j) {  // 128 rows x 8 chunks of the key half
      const int r = tid / 8 + 32 * j, c = tid % 8;
      const int t = r0 + r < cnt ? min(max(lst[r0 + r] - hT, 0), T - 1) : 0;  // never outside the unit's slab
      cp_async16(sK + r * 128 + ((c ^ (r & 7)) << 4), Ku + (size_t)t * D + c * 8, r0 + r < cnt ? 16u : 0u);
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // 128 rows x 16 chunks of the value rows
      const int r = tid / 16 + 16 * j, c = tid % 16;
      const int t = r0 + r < cnt ? min(max(lst[r0 + r] - hT, 0), T - 1) : 0;
      if (c < vch)
        cp_async16(sV + (c >> 3) * kBoxBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4), Vu + (size_t)t * D + c * 8,
                   r0 + r < cnt ? 16u : 0u);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
    __syncthreads();
    if (tid == 0) {
      for (int kk = 0; kk < 8; ++kk)
        umma_bf16(tm, sdesc_sw128(aV + kk * 2048, kBoxBytes, 1024), sdesc_sw128(aK + kk * 2048, kBoxBytes, 1024), id,
                  (it > 0 || kk > 0) ? 1u : 0u);
      umma_commit(&done);
    }
    // column sums, and in the final stage the cache rows, from the same tile
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = tid / 8 + 32 * j, c = tid % 8, row = r0 + r;
      const uint4 w = *reinterpret_cast<const uint4*>(sK + r * 128 + ((c ^ (r & 7)) << 4));
      float f[8];
      unpack8(w, f);
#pragma unroll
      for (int e = 0; e < 8; ++e) ks[e] += f[e];
      // (a joint selection's cache is zero up to the next tile past a unit's rows)
      if (FINAL && (row < cnt || (L.hs > 1 && row < a.dst_cap)))
        *reinterpret_cast<uint4*>(a.dst_K + ((size_t)u * a.dst_cap + row) * D + kh * 64 + c * 8) = w;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int r = tid / 16 + 16 * j, c = tid % 16, row = r0 + r;
      if (c < vch) {
        const uint4 w = *reinterpret_cast<const uint4*>(sV + (c >> 3) * kBoxBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4));
        float f[8];
        unpack8(w, f);
#pragma unroll
        for (int e = 0; e < 8; ++e) vs[e] += f[e];
        if (FINAL && (c >> 3) == kh && (row < cnt || (L.hs > 1 && row < a.dst_cap)))
          *reinterpret_cast<uint4*>(a.dst_V + ((size_t)u * a.dst_cap + row) * D + c * 8) = w;
      }
    }
    if (FINAL && kh == 0 && tid < kTok && r0 + tid < cnt)
      a.dst_pos[(size_t)u * a.dst_cap + r0 + tid] = lst[r0 + tid] - hT;
  }
  // ---- this CTA's sums and V^T K into shared memory
  if (it > 0 && ok) {
    if (tid == 0 && !mbar_wait(&done, (it - 1) & 1, a.polls)) {
      s_ok = 0;
      record_error(a.ws, MKV_ERR_TIMEOUT, u);
    }
    __syncthreads();
    ok = s_ok != 0;
  }
  if (!ok && tid == 0) (void)mbar_wait(&done, (it - 1) & 1);  // drain: the MMAs still read shared memory
  __syncthreads();
  tc_fence_after();
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    s_pk[tid / 8][(tid % 8) * 8 + e] = ks[e];
    s_pv[tid / 16][(tid % 16) * 8 + e] = vs[e];
  }
  {
    float x[32];
    const int row = (warp & 3) * 32 + lane, c0 = (warp >> 2) * 32;
    if (it > 0 && ok) {
      tmem_ld32(tm + (static_cast<uint32_t>((warp & 3) * 32) << 16) + c0, x);
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) x[j] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 32; j += 4)
      *reinterpret_cast<float4*>(red + row * kRsRed + c0 + j) = make_float4(x[j], x[j + 1], x[j + 2], x[j + 3]);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tm, 64);
  }
  if (tid < 64) {
    float x = 0.f;
    for (int g = 0; g < 32; ++g) x += s_pk[g][tid];
    s_sk[tid] = x;
  } else if (tid < 64 + kDP) {
    float x = 0.f;
    for (int g = 0; g < 16; ++g) x += s_pv[g][tid - 64];
    s_sv[tid - 64] = x;
  }
  cg::cluster_group cluster = cg::this_cluster();
  if constexpr (CL > 1) cluster.sync();
  else __syncthreads();

  // ---- R's sums over the cluster, and E = all \ R
  const float nR = ok ? static_cast<float>(cnt) : 0.f;
  float SR[NI][4], rv[NI], rk[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    rv[i] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) SR[i][j] = 0.f;
  }
#pragma unroll
  for (int r = 0; r < CL; ++r) {
    const float* pr = CL > 1 ? cluster.map_shared_rank(red, r) : red;
    const float* pk = CL > 1 ? cluster.map_shared_rank(s_sk, r) : s_sk;
    const float* pv = CL > 1 ? cluster.map_shared_rank(s_sv, r) : s_sv;
    const float4 k4 = *reinterpret_cast<const float4*>(pk + cq * 4);
    rk[0] += k4.x;
    rk[1] += k4.y;
    rk[2] += k4.z;
    rk[3] += k4.w;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const int row = rank * RW + ar + 16 * i;
      const float4 s4 = *reinterpret_cast<const float4*>(pr + row * kRsRed + cq * 4);
      SR[i][0] += s4.x;
      SR[i][1] += s4.y;
      SR[i][2] += s4.z;
      SR[i][3] += s4.w;
      rv[i] += pv[row];
    }
  }
  const float nE = n - nR;
  float mk[4], mkR[4], mkE[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    mk[j] = x0k[j] + sk[j] / n;
    mkR[j] = nR > 0.f ? rk[j] / nR : 0.f;
    mkE[j] = nE > 0.f ? (n * mk[j] - nR * mkR[j]) / nE : 0.f;
  }
#pragma unroll
  for (int i = 0; i < NI; ++i) {
    const int row = rank * RW + ar + 16 * i;
    const float mv = x0v[i] + sv[i] / n;
    const float mvR = nR > 0.f ? rv[i] / nR : 0.f;
    const float mvE = nE > 0.f ? (n * mv - nR * mvR) / nE : 0.f;
    float CE[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      CE[j] = 0.f;
      if (nE > 0.f) {
        const float Mall = M[i][j] - sv[i] * sk[j] / n;
        const float MR = nR > 0.f ? SR[i][j] - rv[i] * rk[j] / nR : 0.f;
        const float ME = Mall - MR - (nE * nR / n) * (mvR - mvE) * (mkR[j] - mkE[j]);
        CE[j] = ME / nE;
      }
    }
    if constexpr (FINAL) {
      if (row < D) {
        *reinterpret_cast<float4*>(a.mom.C + ((size_t)u * D + row) * D + kh * 64 + cq * 4) =
            make_float4(CE[0], CE[1], CE[2], CE[3]);
        if (kh == 0 && cq == 0) a.mom.mu_v[(size_t)u * D + row] = mvE;
        if (row == 0)
#pragma unroll
          for (int j = 0; j < 4; ++j) a.mom.mu_k[(size_t)u * D + kh * 64 + cq * 4 + j] = mkE[j];
      }
    } else {
      // C0' (clamped where |n0 C0| < tau) as three bf16 parts, K-major operand
      // rows (value dims; zero past D) in the swizzled layout
      float r4[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) r4[j] = (row < D && !(fabsf(CE[j] * nE) < a.tau)) ? CE[j] : 0.f;
      uint8_t* img = L.cimg + (size_t)u * 3 * kTileBytes + swz_off(row, kh * 64 + cq * 4, kTok);
#pragma unroll
      for (int part = 0; part < 3; ++part) {
        uint2 w;
        w.x = pack_bf16x2(r4[0], r4[1]);
        w.y = pack_bf16x2(r4[2], r4[3]);
        *reinterpret_cast<uint2*>(img + (size_t)part * kTileBytes) = w;
#pragma unroll
        for (int j = 0; j < 4; ++j) r4[j] = bf16_residual(r4[j]);
      }
      if (kh == 0 && cq == 0) L.mv0[(size_t)u * kDP + row] = row < D ? mvE : 0.f;
    }
  }
  if (FINAL && kh == 0 && rank == 0 && tid == 0) {
    a.mom.n[u] = static_cast<int32_t>(nE);
    a.dst_len[u] = cnt;
    a.dst_seen[u] = T;
  }
  if constexpr (CL > 1) cluster.sync();  // no CTA leaves while another reads its shared memory
}

// ---------------------------------------------------------- keep-all path
template <int D>
__global__ void __launch_bounds__(256) keep_all_kernel(const CompressArgs a, int T) {
  const int u = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + warp;
  if (i < T) {
    const __nv_bfloat16* Ks = reinterpret_cast<const __nv_bfloat16*>(a.K) + ((size_t)u * T + i) * D;
    const __nv_bfloat16* Vs = reinterpret_cast<const __nv_bfloat16*>(a.V) + ((size_t)u * T + i) * D;
    __nv_bfloat16* Kd = reinterpret_cast<__nv_bfloat16*>(a.cache.K) + ((size_t)u * a.cache.capacity + i) * D;
    __nv_bfloat16* Vd = reinterpret_cast<__nv_bfloat16*>(a.cache.V) + ((size_t)u * a.cache.capacity + i) * D;
    for (int c = lane * 2; c < D; c += 64) {
      *reinterpret_cast<__nv_bfloat162*>(Kd + c) = *reinterpret_cast<const __nv_bfloat162*>(Ks + c);
      *reinterpret_cast<__nv_bfloat162*>(Vd + c) = *reinterpret_cast<const __nv_bfloat162*>(Vs + c);
    }
    if (lane == 0) a.cache.pos[(size_t)u * a.cache.capacity + i] = i;
  }
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0) {
      a.cache.len[u] = T;
      a.cache.seen[u] = T;
      a.mom.n[u] = 0;
    }
    for (int e = threadIdx.x; e < D * D; e += blockDim.x) a.mom.C[(size_t)u * D * D + e] = 0.f;
    for (int e = threadIdx.x; e < D; e += blockDim.x) {
      a.mom.mu_k[(size_t)u * D + e] = 0.f;
      a.mom.mu_v[(size_t)u * D + e] = 0.f;
    }
  }
}

// ------------------------------------------------------------------- host
constexpr size_t kStatsSmem = 1024 + 2 * 2 * kTileBytes + 2 * 2 * kBoxBytes + 4096;  // K, V stages, Q, ones
constexpr size_t kScoresSmem = 1024 + 3 * kTileBytes + 2 * 2 * kBoxBytes;
constexpr size_t kResidualSmem = 1024 + 2 * 2 * kTileBytes + 3 * kTileBytes;

// A launch that may begin while the kernel before it on the stream drains (it
// waits for that kernel's end by itself); cl > 0: in clusters of cl CTAs
// (select_kernel declares its own).
template <typename... P, typename... A>
cudaError_t launch_pdl(void (*f)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st, int cl, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = cl;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cl > 0 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, f, std::forward<A>(args)...);
}

cudaError_t smem_attr(const void* f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

// CTAs per unit and key half of rset_kernel: one row tile each, and no more
// chunk records to merge than about 300 KB, as long as all CTAs run at once
// (two per SM).
int rset_cluster(const Layout& L, int num_sms) {
  const long tiles = (L.B + kTok - 1) / kTok, nh = L.D / 64;
  const long want = std::max(tiles, (long)L.n_chunks / 9);
  int cl = 1;
  while (cl < 8 && cl < want && 2L * cl * nh * L.units <= 2L * num_sms) cl *= 2;
  return cl;
}

template <bool FINAL>
cudaError_t launch_rset(const RsetArgs& a, int cl, cudaStream_t st) {
  const dim3 grid(cl * (a.L.D / 64), a.L.units);
  auto go = [&](void (*f)(RsetArgs)) -> cudaError_t {
    const cudaError_t e = smem_attr(reinterpret_cast<const void*>(f), kRsSmem);
    return e != cudaSuccess ? e : launch_pdl(f, grid, kRsThreads, kRsSmem, st, cl, a);
  };
  switch (cl) {
    case 8: return go(rset_kernel<8, FINAL>);
    case 4: return go(rset_kernel<4, FINAL>);
    case 2: return go(rset_kernel<2, FINAL>);
    default: return go(rset_kernel<1, FINAL>);
  }
}

cudaError_t run(const CompressArgs& a, const mkv_geom& g, int num_sms, cudaStream_t st) {
  Layout L = make_layout(g, a.T, a.budget, a.window, a.sink, a.keep_window, a.adaptive, num_sms);
  carve(L, a.ws);
  const int D = g.head_dim, T = a.T, B = a.budget, U = L.units;
  const bool keep_all = T <= B;
  cudaError_t e = cudaSuccess;
  if ((e = smem_attr((const void*)stats_tc, kStatsSmem)) != cudaSuccess) return e;
  if ((e = smem_attr((const void*)scores_tc, kScoresSmem)) != cudaSuccess) return e;
  if ((e = smem_attr((const void*)residual_tc, kResidualSmem)) != cudaSuccess) return e;

  CUtensorMap tmK, tmV, tmQ;
  const uint64_t rs = (uint64_t)D * 2;
  if (!encode_tmap_bf16_3d(&tmK, a.K, D, T, U, rs, (uint64_t)T * rs, kTok) ||
      !encode_tmap_bf16_3d(&tmV, a.V, D, T, U, rs, (uint64_t)T * rs, kTok) ||
      !encode_tmap_bf16_3d(&tmQ, a.Q, D, L.RW, U, rs, (uint64_t)L.RW * rs, L.RWb * 128))
    return cudaErrorInvalidValue;

  TcArgs tp{};
  tp.n_rows = T;
  tp.chunk = L.chunk;
  tp.n_chunks = L.n_chunks;
  tp.D = D;
  tp.RW = L.RW;
  tp.RWb = L.RWb;
  tp.W = a.window;
  tp.T = T;
  tp.causal = a.causal;
  tp.sink = a.sink;
  tp.keep_window = a.keep_window;
  tp.pool = a.pool;
  tp.qscale = rsqrtf(static_cast<float>(D)) * kLog2e;
  tp.rowpart = L.rowpart;
  tp.mrec = L.mpart;
  tp.ws = a.ws;
  tp.polls = pipeline_poll_limit();
  const dim3 cg(L.n_chunks, U);

  if (!keep_all || a.diag_scores != nullptr) {
    if ((e = launch_pdl(stats_tc, cg, kStatsThreads, kStatsSmem, st, 0, tp, tmK, tmV, tmQ)) != cudaSuccess) return e;
    TcArgs p2 = tp;
    p2.s_out = L.s;
    p2.diag = a.diag_scores;
    if ((e = launch_pdl(scores_tc, cg, kStatsThreads, kScoresSmem, st, 0, p2, tmK, tmQ)) != cudaSuccess) return e;
  }
  if (keep_all) {
    if (D == 128) keep_all_kernel<128><<<dim3((T + 7) / 8, U), 256, 0, st>>>(a, T);
    else keep_all_kernel<64><<<dim3((T + 7) / 8, U), 256, 0, st>>>(a, T);
    return cudaGetLastError();
  }

  SelectArgs sa{};
  const int n_groups = U / L.hs;
  const bool prefilter = L.cand != nullptr;
  // keys a CTA caches when its range fits, for the joint (or per-unit) selection and the prefilter
  auto cached_keys = [](long per) { return per <= kSelSmemKeys ? static_cast<int>(per) : 0; };
  sa.smem_keys = cached_keys((L.hs * (long)L.Tc + kSelCL - 1) / kSelCL);
  const int pf_keys = cached_keys((T + kSelCL - 1) / kSelCL);
  const size_t sel_smem = (size_t)sa.smem_keys * sizeof(uint32_t), pf_smem = (size_t)pf_keys * sizeof(uint32_t);
  if ((e = smem_attr((const void*)select_kernel, std::max(sel_smem, pf_smem))) != cudaSuccess) return e;
  sa.T = T;
  sa.Tc = L.Tc;
  sa.cand = L.cand;
  sa.W = a.window;
  sa.B = B;
  sa.sink = a.sink;
  sa.keep_window = a.keep_window;
  sa.idx = L.idx;
  sa.hs = L.hs;
  sa.cnt = L.cnt;
  sa.hbeg = L.hbeg;
  // one selection over `scores`; a joint one first keeps each unit's protected
  // rows and its top Tc - |protected| as candidates (a per-unit selection)
  auto select = [&](const float* scores, int32_t* diag_idx) -> cudaError_t {
    if (prefilter) {
      SelectArgs pf = sa;
      pf.scores = scores;
      pf.hs = 1;
      pf.Tc = T;
      pf.cand = nullptr;
      pf.B = L.Tc;
      pf.idx = L.cand;
      pf.smem_keys = pf_keys;
      pf.cnt = nullptr;
      pf.hbeg = nullptr;
      const cudaError_t pe = launch_pdl(select_kernel, dim3(U * kSelCL), kSelThreads, pf_smem, st, 0, pf);
      if (pe != cudaSuccess) return pe;
    }
    SelectArgs s0 = sa;
    s0.scores = scores;
    s0.diag_idx = diag_idx;
    return launch_pdl(select_kernel, dim3(n_groups * kSelCL), kSelThreads, sel_smem, st, 0, s0);
  };
  RsetArgs ra{};
  ra.L = L;
  ra.K = static_cast<const __nv_bfloat16*>(a.K);
  ra.V = static_cast<const __nv_bfloat16*>(a.V);
  ra.tau = a.tau;
  ra.dst_K = static_cast<__nv_bfloat16*>(a.cache.K);
  ra.dst_V = static_cast<__nv_bfloat16*>(a.cache.V);
  ra.dst_cap = a.cache.capacity;
  ra.dst_pos = a.cache.pos;
  ra.dst_len = a.cache.len;
  ra.dst_seen = a.cache.seen;
  ra.mom = a.mom;
  ra.ws = a.ws;
  ra.polls = tp.polls;
  const int cl = rset_cluster(L, num_sms);

  if ((e = select(L.s, a.diag_idx1)) != cudaSuccess) return e;
  if (a.mi) {
    if ((e = launch_rset<false>(ra, cl, st)) != cudaSuccess) return e;
    TcArgs r = tp;
    r.cimg = L.cimg;
    r.mv0 = L.mv0;
    r.s_in = L.s;
    r.s_out = L.s2;
    r.diag = a.diag_score2;
    if ((e = launch_pdl(residual_tc, cg, kStatsThreads, kResidualSmem, st, 0, r, tmK, tmV)) != cudaSuccess) return e;
    if ((e = select(L.s2, nullptr)) != cudaSuccess) return e;
  }
  return launch_rset<true>(ra, cl, st);
}

}  // namespace

size_t compress_workspace_bytes(const mkv_geom& g, int32_t T, const mkv_compress_params& p, int num_sms) {
  Layout L = make_layout(g, T, p.budget, p.window, p.sink, p.keep_window, p.adaptive, num_sms);
  return carve(L, nullptr);
}

cudaError_t launch_compress(const CompressArgs& a, const mkv_geom& g, size_t ws_bytes, int num_sms,
                            cudaStream_t stream) {
  (void)ws_bytes;
  if (g.head_dim != 128 && g.head_dim != 64) return cudaErrorInvalidValue;
  return run(a, g, num_sms, stream);
}

}  // namespace mkv
