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
//   select    (8-CTA cluster per unit) R0 = protected + top-k(s): the bin of the
//                            k-th key from counts the score kernels keep, then
//                            the k-th among the bin's keys, ties to the lower
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
// while its predecessor drains.  The last releases no launch after the call.
//
// With the budget shared by the KV heads of a batch item (adaptive), each
// select ranks the (head, position) pairs of the batch item together.
//
// The tensor-core kernels are warp-specialised: warp 0 issues the TMA copies
// (3-D tensor maps over per-unit slabs: rows past a unit's end read as zeros),
// warp 1 owns TMEM and issues tcgen05.mma, and the other warps run the
// epilogue (two groups of four in stats_tc and residual_tc, four in scores_tc);
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
// residual_tc: two epilogue groups of 4 warps (2..5 and 6..9), so that two
// warps per scheduler share the work
constexpr int kResThreads = 320;
constexpr int kMaxHs = 64;  // KV heads of a batch item with the adaptive budget
constexpr int kHot = 249, kHotLo = (127 - 20) * 8;  // bins a CTA counts in shared memory (count_bin)
// scores_tc's K stages, and its shared memory
__host__ __device__ constexpr int score_stages(int RWb) { return RWb == 1 ? 6 : 4; }
__host__ __device__ constexpr size_t score_smem(int RWb) {
  return (size_t)score_stages(RWb) * kTileBytes + (size_t)RWb * 2 * kBoxBytes + 256 * 4 + kHot * 4 +
         (RWb - 1) * 2 * 128 * 4;
}
// stats_tc's K/V stages: shared memory holds a third beside one block of window rows
__host__ __device__ constexpr int stats_stages(int RWb) { return RWb == 1 ? 3 : 2; }
__host__ __device__ constexpr size_t stats_smem(int RWb) {
  return 1024 + (size_t)stats_stages(RWb) * 2 * kTileBytes + (size_t)RWb * 2 * kBoxBytes;
}
constexpr int kBins = 2048;  // bins of the scores' keys (select_kernel)
constexpr int kGroupCont = 2048;  // contested pairs a joint selection's list holds
constexpr unsigned kFull = 0xffffffffu;

struct Layout {
  int D, G, W, RW, RWb;  // head dim, group, window, window rows = G*W, 128-row blocks of them
  int T, B;
  int hs;    // units per selection group: 1, or the KV heads of a batch item (adaptive budget)
  int units, n_chunks, chunk;
  size_t rec;         // floats per moment record: 4 + 2D + D*D (padded)
  float* rowpart;     // [units][n_chunks][RW][2]  (max in log2 units, sum)
  float* mpart;       // [units][n_chunks][rec]    all-token chunk moments
  float* s;           // [units][T]
  float* s2;          // [units][T]
  int lsel;           // most rows a unit keeps: B, or its share of a group's at most
  int32_t* idx;       // [units][lsel] selected positions, ascending
  int32_t* cnt;       // [units] rows each unit retains
  uint32_t* hist;     // [2][units][kBins] keys of the unprotected scores per bin (s, s2)
  unsigned long long* glist;  // [units / hs][kGroupCont] contested pairs of a joint selection
  int32_t* gcnt;              // [2][units] their counts by group (s, s2)
  uint32_t* sub;              // [2][units / hs][kBins] and their keys per second-level bin (sub_bin)
  uint8_t* cimg;      // [units][3][128 x 128] C0' as three bf16 parts, in the residual's operand layout
  float* mv0;         // [units][kDP] mu_v of E0
  float* fro;         // [units][kDP] parts of ||C0'||_F^2
  float* norms;       // [units][T][2] ||k_t||^2, ||v_t||^2
  int32_t* cand;      // [units][T] positions residual_tc has left to compute
};

__host__ __device__ inline size_t rec_floats(int D) { return align_up(4 + 2 * (size_t)D + (size_t)D * D, 4); }

__host__ __device__ __forceinline__ int protected_count(int T, int W, int sink, int keep_window) {
  const int s = sink < T ? sink : T;
  const int w = keep_window ? (W < T ? W : T) : 0;
  const int overlap = s - (T - w) > 0 ? s - (T - w) : 0;
  return s + w - overlap;
}

Layout make_layout(const mkv_geom& g, int T, int B, int W, int sink, int keep_window, int adaptive, int num_sms) {
  Layout L{};
  L.hs = 1;
  L.lsel = B;
  if (adaptive && T > B) {  // a unit keeps its protected rows plus up to every joint selection
    const long prot = protected_count(T, W, sink, keep_window);
    L.hs = g.n_kv_heads;
    L.lsel = static_cast<int>(std::min<long>(T, (long)g.n_kv_heads * (B - prot) + prot));
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
  L.idx = reinterpret_cast<int32_t*>(take(U * (size_t)L.lsel * sizeof(int32_t)));
  L.cnt = reinterpret_cast<int32_t*>(take(U * sizeof(int32_t)));
  L.hist = reinterpret_cast<uint32_t*>(take(2 * U * (size_t)kBins * sizeof(uint32_t)));
  L.glist = reinterpret_cast<unsigned long long*>(
      take(L.hs > 1 ? U / L.hs * (size_t)kGroupCont * sizeof(unsigned long long) : 0));
  L.gcnt = reinterpret_cast<int32_t*>(take(2 * U * sizeof(int32_t)));
  L.sub = reinterpret_cast<uint32_t*>(take(L.hs > 1 ? 2 * (U / L.hs) * (size_t)kBins * sizeof(uint32_t) : 0));
  L.cimg = take(U * (size_t)3 * kTileBytes);
  L.mv0 = reinterpret_cast<float*>(take(U * (size_t)kDP * sizeof(float)));
  L.fro = reinterpret_cast<float*>(take(U * (size_t)kDP * sizeof(float)));
  L.norms = reinterpret_cast<float*>(take(U * (size_t)L.T * 2 * sizeof(float)));
  L.cand = reinterpret_cast<int32_t*>(take(U * (size_t)L.T * sizeof(int32_t)));
  return off;
}

__device__ __forceinline__ bool is_protected(int t, int T, int W, int sink, int keep_window) {
  return t < sink || (keep_window && t >= T - W);
}

// Order-preserving key of a score, at least 1, and its bin: exponent and three
// mantissa bits of a score that is not negative (all others: bin 0).
__device__ __forceinline__ uint32_t score_key(float s) { return max(1u, float_key(s)); }
__device__ __forceinline__ int key_bin(uint32_t key) {
  return (key & 0x80000000u) ? static_cast<int>((key >> 20) & (kBins - 1)) : 0;
}

// A CTA's counts of its scores' bins, one addition to the table in global memory
// per bin and CTA: 31 octaves from 2^-20 up and bin 0 (zeros).  Others, rare or
// far apart, are counted there at once.  (All of a unit's scores lie in a few
// tens of bins: counting each in global memory, 1M positions of 2 units took
// scores_tc 185 us where the pass alone takes 90.)
__device__ __forceinline__ void count_bin(int bin, uint32_t* s_hot, uint32_t* table) {
  const unsigned i = bin == 0 ? kHot - 1u : static_cast<unsigned>(bin - kHotLo);
  atomicAdd(i < kHot - (bin != 0) ? s_hot + i : table + bin, 1u);
}
__device__ __forceinline__ void flush_bins(const uint32_t* s_hot, uint32_t* table) {
  for (int i = threadIdx.x; i < kHot; i += blockDim.x)
    if (s_hot[i] != 0u) atomicAdd(table + (i == kHot - 1 ? 0 : kHotLo + i), s_hot[i]);
}

// The keys of one bin in second-level bins, in order: eleven of the 20 bits
// below those that the bin fixes; bin 0's by the sign and ten bits below.
__device__ __forceinline__ int sub_bin(int bin, uint32_t key) {
  if (bin > 0) return static_cast<int>((key >> 9) & (kBins - 1));
  return static_cast<int>((key & 0x80000000u) ? 1024u | ((key >> 10) & 1023u) : key >> 21);
}

// 16 bytes global -> shared, asynchronously (src_bytes 0: zeros)
__device__ __forceinline__ void cp_async16(void* dst, const void* src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src), "r"(src_bytes)
               : "memory");
}

// Eight bf16 of a 16-byte chunk added to `acc` (pairs of floats), and the sum
// of their squares returned: two elements per instruction.
__device__ __forceinline__ float sum_chunk(const uint4& w, uint64_t (&acc)[4]) {
  const uint32_t x[4] = {w.x, w.y, w.z, w.w};
  uint64_t sq = 0ull;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    uint64_t v;
    asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(x[i] << 16), "r"(x[i] & 0xffff0000u));
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(acc[i]) : "l"(acc[i]), "l"(v));
    asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(sq) : "l"(v), "l"(sq));
  }
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(sq));
  return a + b;
}

// Sums over each half warp of eight values per lane: lanes 2x and 2x + 1 of a
// half get the sum of v[x] (x < 8).
__device__ __forceinline__ float half_warp_sums(float (&v)[8], int lane) {
#pragma unroll
  for (int w = 4; w >= 1; w >>= 1) {
    const bool hi = (lane & (2 * w)) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = hi ? v[i] : v[i + w], keep = hi ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(kFull, send, 2 * w);
    }
  }
  return v[0] + __shfl_xor_sync(kFull, v[0], 1);
}

__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, 384;" ::: "memory"); }
// whether v holds in all 384 threads of stats_tc's epilogue and summing warps (barrier 1)
__device__ __forceinline__ bool epi_all(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.and.pred q, 1, 384, p;\n\t"
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

// pwait by a whole warp: all its lanes go on or none.
__device__ __forceinline__ bool pwait_warp(uint64_t* bar, uint32_t parity, volatile int* abort_flag, void* ws, int u,
                                           uint32_t polls) {
  return __all_sync(kFull, pwait(bar, parity, abort_flag, ws, u, polls)) != 0;
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
  uint32_t* hist;  // stats_tc: both tables, zeroed; scores_tc, residual_tc: the table their scores are counted in
  int32_t* gcnt;   // [2][units] counts of joint selections, zeroed by stats_tc
  uint32_t* sub;   // [2][units / hs][kBins] second-level counts of joint selections (or null), zeroed by stats_tc
  int units;
  float* diag;
  const uint8_t* cimg;  // [units][3][128 x 128] operand image of C0'
  const float* mv0;     // [units][kDP]
  float* norms;         // [units][T][2] ||k_t||^2, ||v_t||^2
  int hs;  // units per selection group
  // residual_tc's pruning
  int prune, B;
  const int32_t* idx;   // [units][lsel] the first stage's selections
  const int32_t* cnt;   // [units] their numbers (joint; B otherwise)
  int lsel;
  const float* fro;     // [units][kDP] parts (n_fro of them) of ||C0'||_F^2
  int n_fro;
  int32_t* cand;        // [units][T] positions left to compute, per CTA from its first position on
  const void* K;
  const void* V;
  void* ws;
  uint32_t polls;  // poll limit of the pipeline waits
};

// --------------------------------------------------------------- stats_tc
// Window-row statistics, chunk moments and row norms of the prompt, in one
// pass over K and V.  Bounded by that read (64 KB a tile and SM): the tensor
// cores do the two products only, 1024 cycles a tile (column sums by products
// with ones cost as many again); eight warps turn the logits into row
// statistics, four others take the column sums and row norms from shared
// memory (in the same warps the two cost 32 us of 125 at 32K, batch 4); with
// up to 128 window rows three stages are in flight and the logits
// double-buffered.  V streams through L2, so that more of K is still there for
// the scores, which start from the end of the chunk.  Alone at 32K, 32 units:
// 115 us, 4.7 TB/s on 128 CTAs, one per SM; at 8K 17 us (21 before).
constexpr int kStatThreads = 64 + 256 + 128;
__global__ void __launch_bounds__(kStatThreads, 1)
    stats_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
             const __grid_constant__ CUtensorMap tmQ) {
  constexpr int kMaxS = 3;
  constexpr uint32_t kTmemCols = 512;
  constexpr int cS = 256;  // TMEM columns: the logits [0, 256), V^T K
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  const int RWb = p.RWb, kS = stats_stages(RWb), NB = RWb == 1 ? 2 : 1;  // stages, logits buffers
  uint8_t* sKV = sm;                           // [kS][K tile, V tile]
  uint8_t* sQ = sm + (size_t)kS * 2 * kTileBytes;  // [2 boxes][RWb*128 rows][128 B]
  // after the last tile the first stage holds the epilogue's staging
  float* stg = reinterpret_cast<float*>(sm);                  // [2 groups][128][36]
  float* s_pk = stg + 2 * 128 * 36;                           // [8][128] column sums of K per row group
  float* s_pv = s_pk + 8 * 128;                               // the same of V
  float* s_m1 = s_pv + 8 * 128;                              // [2][128] the second group's row maxima
  float* s_l1 = s_m1 + 2 * 128;                               // and sums
  float* sum_k = s_l1 + 2 * 128;                              // [128]
  float* sum_v = sum_k + kDP;                                 // [128]
  __shared__ __align__(8) uint64_t full[kMaxS], empty[kMaxS], lfull[2], lempty[2], qfull, sdone;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued;

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  const int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;
  volatile int* abrt = &abort_flag;

  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1 + 4);  // the stage's MMAs and the summing warps' reads
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&lfull[i], 1);
      mbar_init(&lempty[i], 8);
    }
    mbar_init(&qfull, 1);
    mbar_init(&sdone, 1);
    abort_flag = 0;
    s_issued = 0;
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_base, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;
  grid_dependency_wait();
  grid_launch_dependents();

  if (warp == 0) {
    if (lane == 0) {  // ---- producer
      const uint64_t pol_v = l2_evict_first();
      mbar_arrive_expect_tx(&qfull, 2u * RWb * kBoxBytes);
      for (int bx = 0; bx < 2; ++bx) tma_load_3d(sQ + bx * RWb * kBoxBytes, &tmQ, bx * 64, 0, u, &qfull);
      int s = 0;
      uint32_t ph = 1;
      for (int i = 0; i < n_tiles; ++i) {
        if (i >= kS && !pwait(&empty[s], ph, abrt, p.ws, u, p.polls)) break;
        uint8_t* dst = sKV + (size_t)s * 2 * kTileBytes;
        mbar_arrive_expect_tx(&full[s], 2u * kTileBytes);
        for (int bx = 0; bx < 2; ++bx) tma_load_3d(dst + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[s]);
        for (int bx = 0; bx < 2; ++bx)
          tma_load_3d_hint(dst + kTileBytes + bx * kBoxBytes, &tmV, bx * 64, t_begin + i * kTok, u, &full[s], pol_v);
        s_issued = i + 1;
        if (++s == kS) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {  // ---- MMA issuer
      const uint32_t idL = idesc_bf16(128, 128, 0, 0);  // logits: rows x tokens, both K-major
      const uint32_t idS = idesc_bf16(128, 128, 1, 1);  // V^T K: both MN-major (reduction over tokens)
      const uint64_t dq = sdesc_sw128(smem_addr(sQ), 16, 1024), dk0 = sdesc_sw128(smem_addr(sKV), 16, 1024);
      const uint64_t ds0 = sdesc_sw128(smem_addr(sKV), kBoxBytes, 1024);
      const bool ok = pwait(&qfull, 0, abrt, p.ws, u, p.polls);
      int s = 0, b = 0;               // stage and logits buffer of tile i, and their phases
      uint32_t ph = 0, bph = 1;
      for (int i = 0; ok && i < n_tiles; ++i) {
        if (!pwait(&full[s], ph, abrt, p.ws, u, p.polls)) break;
        if (i >= NB && !pwait(&lempty[b], bph, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        const uint32_t st = s * (2 * kTileBytes >> 4);  // in descriptor units
        for (int rb = 0; rb < RWb; ++rb)
          umma_k128(tm + (b + rb) * 128, dq + rb * (kBoxBytes >> 4), dk0 + st, RWb * kBoxBytes, kBoxBytes, idL, 0u);
        umma_commit(&lfull[b]);
        umma_mn128(tm + cS, ds0 + st + (kTileBytes >> 4), ds0 + st, idS, i > 0 ? 1u : 0u);
        umma_commit(&empty[s]);
        if (++s == kS) {
          s = 0;
          ph ^= 1u;
        }
        if (++b == NB) {
          b = 0;
          bph ^= 1u;
        }
      }
      umma_commit(&sdone);
    }
  } else if (warp >= 10) {
    // ---- column sums and row norms: warp w takes rows 32 w .. 32 w + 31, this
    // lane the 8 dims of chunk lane % 16 in the rows lane / 16 + 2 j of them
    const int sw = warp - 10, ch = lane & 15, rh = lane >> 4;
    uint64_t ksum[4] = {0ull, 0ull, 0ull, 0ull}, vsum[4] = {0ull, 0ull, 0ull, 0ull};
    for (int i = 0; i < n_tiles; ++i) {
      const int s = i % kS;
      if (!pwait_warp(&full[s], (i / kS) & 1, abrt, p.ws, u, p.polls)) break;
#pragma unroll 1
      for (int r16 = 0; r16 < 32; r16 += 16) {
        const uint8_t* tk = sKV + (size_t)s * 2 * kTileBytes + (ch >> 3) * kBoxBytes + (sw * 32 + r16 + rh) * 128;
        float kn[8], vn[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const uint32_t off = 2 * j * 128 + (((ch & 7) ^ ((rh + 2 * j) & 7)) << 4);
          kn[j] = sum_chunk(*reinterpret_cast<const uint4*>(tk + off), ksum);
          vn[j] = sum_chunk(*reinterpret_cast<const uint4*>(tk + kTileBytes + off), vsum);
        }
        // squared norms over the 16 lanes of each row: lanes 2 x, 2 x + 1 of a half hold its row 2 x
        const float kq = half_warp_sums(kn, lane), vq = half_warp_sums(vn, lane);
        const int t = t_begin + i * kTok + sw * 32 + r16 + rh + 2 * ((lane >> 1) & 7);
        if (t < t_end) p.norms[((size_t)u * p.T + t) * 2 + (lane & 1)] = (lane & 1) ? vq : kq;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
    }
    // the first stage is free once every MMA is done and every summing warp is
    // past its tiles: then the sums go there (after an abort they are not read)
    const bool got = epi_all(pwait_warp(&sdone, 0, abrt, p.ws, u, p.polls));
    if (got) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        reinterpret_cast<uint64_t*>(s_pk + (sw * 2 + rh) * 128 + ch * 8)[e] = ksum[e];
        reinterpret_cast<uint64_t*>(s_pv + (sw * 2 + rh) * 128 + ch * 8)[e] = vsum[e];
      }
      epi_sync();
    }
  } else {
    // ---- epilogue: group 0 = warps 2..5 (tokens 0..63 of a tile's logits),
    // group 1 = warps 6..9 (tokens 64..127); TMEM lane quarter qd = warp % 4
    const int ew = warp - 2, grp = ew >> 2;
    const int et = tid - 64 - grp * 128, qd = warp & 3;
    if (chunk == 0 && tid - 64 < 2) p.gcnt[(size_t)(tid - 64) * p.units + u] = 0;
    if (chunk == 0)  // the unit's two tables of key counts
      for (int i = tid - 64; i < 2 * kBins / 4; i += 256) {
        const int tab = i / (kBins / 4), b4 = i % (kBins / 4);
        reinterpret_cast<uint4*>(p.hist + ((size_t)tab * p.units + u) * kBins)[b4] = make_uint4(0u, 0u, 0u, 0u);
        if (p.sub != nullptr && u % p.hs == 0)
          reinterpret_cast<uint4*>(p.sub + ((size_t)tab * p.units + u) / p.hs * kBins)[b4] = make_uint4(0u, 0u, 0u, 0u);
      }
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    float m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
    int tmax_vis[2];
    for (int rb = 0; rb < 2; ++rb) {
      const int r = rb * 128 + qd * 32 + lane;  // window row of this thread
      tmax_vis[rb] = p.causal ? p.T - p.W + r % p.W : 0x7fffffff;
    }
    const int t_safe = p.causal ? p.T - p.W : 0x7fffffff;  // tokens every window row sees
    for (int i = 0; i < n_tiles; ++i) {
      const int b = i % NB, tt0 = t_begin + i * kTok;
      if (!pwait_warp(&lfull[b], (i / NB) & 1, abrt, p.ws, u, p.polls)) break;
      tc_fence_after();
      const bool fast = tt0 + kTok <= t_end && tt0 + kTok - 1 <= t_safe;  // no masking in this tile
      // rb runs over a constant range (guarded by RWb), so that m, l and
      // tmax_vis stay in registers
#pragma unroll
      for (int rb = 0; rb < 2; ++rb) {
        if (rb >= RWb) break;
        for (int c0 = grp * 64; c0 < grp * 64 + 64; c0 += 32) {
          float x[32];
          tmem_ld32(tm + lane_base + (b + rb) * 128 + c0, x);
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
      if (lane == 0) mbar_arrive(&lempty[b]);
    }
    // uniform over the epilogue and summing warps: after an abort the MMAs may still write
    // TMEM and read the stages, so neither is touched and the chunk's record
    // is left empty
    const bool got = epi_all(pwait_warp(&sdone, 0, abrt, p.ws, u, p.polls));
    float* rec = p.mrec + ((size_t)u * p.n_chunks + chunk) * rec_floats(p.D);
    if (got) {
      tc_fence_after();
      // the second group's row statistics
      if (grp == 1)
#pragma unroll
        for (int rb = 0; rb < 2; ++rb) {
          s_m1[rb * 128 + qd * 32 + lane] = m[rb];
          s_l1[rb * 128 + qd * 32 + lane] = l[rb];
        }
      epi_sync();
      {
        const float* part = grp == 0 ? s_pk : s_pv;
        float x = 0.f;
#pragma unroll
        for (int g = 0; g < 8; ++g) x += part[g * 128 + et];
        (grp == 0 ? sum_k : sum_v)[et] = x;
      }
      if (grp == 0)
#pragma unroll
        for (int rb = 0; rb < 2; ++rb) {
          if (rb >= RWb) break;
          const int r = rb * 128 + qd * 32 + lane;
          const float m1 = s_m1[r], l1 = s_l1[r];
          const float Mx = fmaxf(m[rb], m1);
          float Ls = 0.f;
          if (Mx != -INFINITY) {
            if (m[rb] != -INFINITY) Ls += l[rb] * fast_exp2(m[rb] - Mx);
            if (m1 != -INFINITY) Ls += l1 * fast_exp2(m1 - Mx);
          }
          if (r < p.RW)
            *reinterpret_cast<float2*>(p.rowpart + (((size_t)u * p.n_chunks + chunk) * p.RW + r) * 2) =
                make_float2(Mx, Ls);
        }
      named_sync(4, 256);
      const float nc = static_cast<float>(max(0, t_end - t_begin)), inv_nc = nc > 0.f ? 1.f / nc : 0.f;
      const int a = qd * 32 + lane;  // value dim = TMEM lane
      const float sva = sum_v[a] * inv_nc;
      // centred co-moment rows, 32 columns at a time and group, through shared
      // memory so that the record is written in whole 128-byte lines
      float* sg = stg + grp * 128 * 36;
#pragma unroll 1
      for (int c0 = grp * 64; c0 < grp * 64 + 64; c0 += 32) {
        float x[32];
        tmem_ld32(tm + lane_base + cS + c0, x);
#pragma unroll
        for (int jj = 0; jj < 32; jj += 4) {
          const float4 k4 = *reinterpret_cast<const float4*>(sum_k + c0 + jj);
          *reinterpret_cast<float4*>(sg + a * 36 + jj) =
              make_float4(x[jj] - sva * k4.x, x[jj + 1] - sva * k4.y, x[jj + 2] - sva * k4.z, x[jj + 3] - sva * k4.w);
        }
        named_sync(2 + grp, 128);
        if (c0 < p.D)
#pragma unroll 4
          for (int r = et / 8; r < p.D; r += 16)
            *reinterpret_cast<float4*>(rec + 4 + 2 * p.D + (size_t)r * p.D + c0 + (et % 8) * 4) =
                *reinterpret_cast<const float4*>(sg + r * 36 + (et % 8) * 4);
        named_sync(2 + grp, 128);
      }
      if (et < p.D) rec[4 + grp * p.D + et] = (grp == 0 ? sum_k : sum_v)[et] * inv_nc;
      if (tid == 64) rec[0] = nc;
    } else if (tid - 64 < 4 + 2 * p.D) {  // an empty record: n = 0, zero means
      for (int i = tid - 64; i < 4 + 2 * p.D; i += 256) rec[i] = 0.f;
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
// Token scores: the logits again, token-major.  Four epilogue groups of four
// warps, each on a TMEM buffer of 128 logits columns: with up to 128 window
// rows they take every fourth tile, with more each tile is shared by two
// groups (rows 0..127 and the others).  Bounded by the read of K, whose rate
// follows the bytes in flight (four stages: 4.5 TB/s with no epilogue at all),
// so shared memory goes to stages; from the chunk's end, where L2 still holds
// what stats_tc read last.  Alone from a cold L2: 62 us at 32K, 32 units (4.4
// TB/s); 74 us at 128K with 256 window rows, where the exponentials bound it.
constexpr int kScoreThreads = 64 + 4 * 128;
__global__ void __launch_bounds__(kScoreThreads, 1)
    scores_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmQ) {
  constexpr int kMaxS = 6;
  extern __shared__ __align__(1024) uint8_t sm[];  // a multiple of 1024 bytes from the block's base
  const int RWb = p.RWb, RWp = RWb * 128, NB = 4 / RWb;  // TMEM buffers of RWp columns
  const int kS = score_stages(RWb);
  uint8_t* sK = sm;                            // [kS][128 x 128]
  uint8_t* sQ = sm + (size_t)kS * kTileBytes;  // [2 boxes][RWb*128][128 B]
  float* s_b = reinterpret_cast<float*>(sQ + (size_t)RWb * 2 * kBoxBytes);  // [256] log2(1 / l_r) - m_r (-inf: padding)
  uint32_t* s_hot = reinterpret_cast<uint32_t*>(s_b + 256);                 // [kHot] counts of the scores' bins
  float(*s_part)[128] = reinterpret_cast<float(*)[128]>(s_hot + kHot);      // [2] the upper rows' sums (RWb = 2)
  __shared__ uint8_t s_wi[256];                                             // window index of row r (r mod W)
  __shared__ __align__(8) uint64_t full[kMaxS], empty[kMaxS], lfull[4], lempty[4], pfull[2], qfull, mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued;

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  const int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;
  volatile int* abrt = &abort_flag;

  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 4; ++i) {
      mbar_init(&lfull[i], 1);
      mbar_init(&lempty[i], 4 * RWb);
    }
    for (int i = 0; i < 2; ++i) mbar_init(&pfull[i], 4);
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
  // wait, so the copies and products need not wait for stats_tc; its row
  // statistics do.
  if (warp == 0) {
    if (lane == 0) {
      mbar_arrive_expect_tx(&qfull, 2u * RWb * kBoxBytes);
      for (int bx = 0; bx < 2; ++bx) tma_load_3d(sQ + bx * RWb * kBoxBytes, &tmQ, bx * 64, 0, u, &qfull);
      int s = 0;
      uint32_t ph = 1;
      for (int i = 0; i < n_tiles; ++i) {
        if (i >= kS && !pwait(&empty[s], ph, abrt, p.ws, u, p.polls)) break;
        mbar_arrive_expect_tx(&full[s], kTileBytes);
        for (int bx = 0; bx < 2; ++bx)
          tma_load_3d(sK + s * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + (n_tiles - 1 - i) * kTok, u,
                      &full[s]);
        s_issued = i + 1;
        if (++s == kS) {
          s = 0;
          ph ^= 1u;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id = idesc_bf16(128, RWp, 0, 0);  // tokens x window rows, both K-major
      const uint64_t dq = sdesc_sw128(smem_addr(sQ), 16, 1024), dk0 = sdesc_sw128(smem_addr(sK), 16, 1024);
      const bool ok = pwait(&qfull, 0, abrt, p.ws, u, p.polls);
      int s = 0, b = 0;  // stage and buffer of tile i, and their phases
      uint32_t ph = 0, bph = 1;
      for (int i = 0; ok && i < n_tiles; ++i) {
        if (!pwait(&full[s], ph, abrt, p.ws, u, p.polls)) break;
        if (i >= NB && !pwait(&lempty[b], bph, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
        umma_k128(tm + b * RWp, dk0 + s * (kTileBytes >> 4), dq, kBoxBytes, RWb * kBoxBytes, id, 0u);
        umma_commit(&lfull[b]);
        umma_commit(&empty[s]);
        if (++s == kS) {
          s = 0;
          ph ^= 1u;
        }
        if (++b == NB) {
          b = 0;
          bph ^= 1u;
        }
      }
      umma_commit(&mma_done);  // every MMA issued has completed
    }
  } else {
    const int grp = (warp - 2) >> 2, qd = warp & 3;
    const int b = grp % NB, half = grp / NB;  // this group's buffer, and its 128 columns of it
    const uint32_t cols = tm + (static_cast<uint32_t>(qd * 32) << 16) + b * RWp + half * 128;
    grid_dependency_wait();
    grid_launch_dependents();
    // merged row statistics of every window row
    for (int r = tid - 64; r < RWp; r += 512) {
      float M = -INFINITY, Lsum = 0.f;
      if (r < p.RW) {
        const float2* rp = reinterpret_cast<const float2*>(p.rowpart) + (size_t)u * p.n_chunks * p.RW + r;
#pragma unroll 8
        for (int c = 0; c < p.n_chunks; ++c) M = fmaxf(M, rp[(size_t)c * p.RW].x);
        if (M != -INFINITY)
#pragma unroll 8
          for (int c = 0; c < p.n_chunks; ++c) {
            const float2 v = rp[(size_t)c * p.RW];
            if (v.x != -INFINITY) Lsum += v.y * fast_exp2(v.x - M);
          }
      }
      s_b[r] = (Lsum > 0.f) ? -log2f(Lsum) - M : -INFINITY;
      s_wi[r] = static_cast<uint8_t>(r % p.W);
    }
    for (int i = tid - 64; i < kHot; i += 512) s_hot[i] = 0u;
    named_sync(1, 512);
    const int t_safe = p.causal ? p.T - p.W : 0x7fffffff;  // tokens every window row sees
    const float* sb = s_b + half * 128;
    for (int i = b; i < n_tiles; i += NB) {
      if (!pwait_warp(&lfull[b], (i / NB) & 1, abrt, p.ws, u, p.polls)) break;
      tc_fence_after();
      const int t = t_begin + (n_tiles - 1 - i) * kTok + qd * 32 + lane;  // token of this thread (TMEM lane)
      const bool fast = t <= t_safe;  // every window row sees this token
      float acc = 0.f;
#pragma unroll 2
      for (int c0 = 0; c0 < 128; c0 += 32) {
        float x[32];
        tmem_ld32(cols + c0, x);
        if (fast) {  // p = 2^(x qscale + b_r); padding rows have b_r = -inf
#pragma unroll
          for (int jj = 0; jj < 32; jj += 4) {
            const float4 b4 = *reinterpret_cast<const float4*>(sb + c0 + jj);
            acc += fast_exp2(fmaf(x[jj], p.qscale, b4.x)) + fast_exp2(fmaf(x[jj + 1], p.qscale, b4.y)) +
                   fast_exp2(fmaf(x[jj + 2], p.qscale, b4.z)) + fast_exp2(fmaf(x[jj + 3], p.qscale, b4.w));
          }
        } else {
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) {
            const int r = half * 128 + c0 + jj;
            if (t <= p.T - p.W + s_wi[r]) acc += fast_exp2(fmaf(x[jj], p.qscale, s_b[r]));
          }
        }
      }
      if (half == 1) {  // the upper rows' sums go to the group of the lower ones
        s_part[b][qd * 32 + lane] = acc;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&pfull[b]);
          mbar_arrive(&lempty[b]);
        }
        continue;
      }
      if (RWb == 2) {
        if (!pwait_warp(&pfull[b], (i / NB) & 1, abrt, p.ws, u, p.polls)) break;
        acc += s_part[b][qd * 32 + lane];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&lempty[b]);
      // rows past the unit's end hold zeros: without the causal mask their
      // logits of 0 would add to the last chunk
      if (t >= t_end) acc = 0.f;
      for (int o = 1; o < p.pool; o <<= 1) acc += __shfl_xor_sync(kFull, acc, o);  // aligned chunks
      if (t < t_end) {
        p.s_out[(size_t)u * p.T + t] = acc;
        if (!is_protected(t, p.T, p.W, p.sink, p.keep_window))
          count_bin(key_bin(score_key(acc)), s_hot, p.hist + (size_t)u * kBins);
        if (p.diag) p.diag[(size_t)u * p.T + t] = acc;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // the MMA thread's final commit, and after an abort the copies in flight
  if (tid == 0) drain_after_abort(full, kS, abort_flag ? s_issued : 0, abort_flag ? &qfull : nullptr, &mma_done);
  flush_bins(s_hot, p.hist + (size_t)u * kBins);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 512);
  }
}

// ------------------------------------------------------------ residual_tc
// score2 = s_t ||v_t - mu_v0 - scale C0' k_t||.  Only the top k of it matter,
// and ||r_t|| lies within c_t = ||mu_v0|| + scale ||C0'||_F ||k_t|| of ||v_t||:
// with theta the smallest s_t (||v_t|| - c_t) over the first stage's k free
// rows, at least k positions reach theta, so a position with
// s_t (||v_t|| + c_t) < theta is not among the top k.  With `prune` a CTA
// compares its positions' scores and norms against theta, gathers the rows
// that remain (a few times the budget where C0' is small beside the values)
// and computes score2 of those; the others get 0, which the k higher ones keep
// out.  Reading K and V a second time is what the full pass costs: alone at
// 32K, batch 4 (32 units) it takes 143 us, the bounded one 23.  When more than half
// of a CTA's positions remain, or the caller wants score2 itself, the full
// pass runs; a position's score2 is the same bits either way.
//
// Roundings: each norm is a chain of at most 18 fp32 additions (1e-6 of it),
// Y's elements come from 24 sums on the tensor core, which may drop a unit in
// the last place each (3e-6 of ||C0'||_F ||k||), so a bound and the score2 it
// stands for differ by less than 1e-5 (||v|| + c).  Relative to ||v|| + c that
// is within theta's factor; ||v|| - c may be much smaller and gives it up.
constexpr float kBoundSlack = 1e-5f;
__global__ void __launch_bounds__(kResThreads, 1)
    residual_tc(const TcArgs p, const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV) {
  constexpr int kS = 2;  // tile i is in stage and TMEM buffer i % 2
  extern __shared__ __align__(1024) uint8_t sm[];  // a multiple of 1024 bytes from the block's base
  uint8_t* sK = sm;                        // [kS][128 x 128]
  uint8_t* sV = sm + kS * kTileBytes;      // [kS][128 x 128]
  uint8_t* sC = sm + 2 * kS * kTileBytes;  // [3 parts][128 x 128]: C0' = hi + mid + lo
  __shared__ __align__(8) uint64_t full[kS], empty[kS], yfull[2], yempty[2], cfull, mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag, s_issued, s_cnt;
  __shared__ uint32_t s_theta;              // bits of a float >= 0
  __shared__ float s_mv[kDP];
  __shared__ float s_mvn[kMaxHs], s_fro[kMaxHs];  // per head of the selection group: ||mu_v0||, scale ||C0'||_F
  __shared__ int s_sel[kMaxHs];                   // and the positions its first selection holds
  __shared__ uint32_t s_hot[kHot];                // counts of the scores' bins

  const int chunk = blockIdx.x, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t_begin = chunk * p.chunk;
  const int t_end = min(p.n_rows, t_begin + p.chunk);
  volatile int* abrt = &abort_flag;
  const int D = p.D;
  const float scale = rsqrtf(static_cast<float>(D));
  auto load_tile = [&](int i) {  // whole tile i of the chunk into stage i % kS
    const int s = i % kS;
    mbar_arrive_expect_tx(&full[s], 2u * kTileBytes);
    for (int bx = 0; bx < 2; ++bx) {
      tma_load_3d(sK + s * kTileBytes + bx * kBoxBytes, &tmK, bx * 64, t_begin + i * kTok, u, &full[s]);
      tma_load_3d(sV + s * kTileBytes + bx * kBoxBytes, &tmV, bx * 64, t_begin + i * kTok, u, &full[s]);
    }
    s_issued = i + 1;
  };
  int n_tiles = (max(0, t_end - t_begin) + kTok - 1) / kTok;

  if (tid == 0) {
    for (int i = 0; i < kS; ++i) {
      mbar_init(&full[i], p.prune ? 4 : 1);  // (set again when a pruning CTA turns to the full pass)
      mbar_init(&empty[i], 1 + 4);           // MMA commit + the 4 epilogue warps (value rows)
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&yfull[i], 1);
      mbar_init(&yempty[i], 4);
    }
    mbar_init(&cfull, 1);
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    s_issued = 0;
    s_cnt = 0;
    s_theta = 0x7f800000u;
    mbar_fence_init();
    // the first stages' copies go out before the dependency wait: the prompt
    // was complete before the compression began
    if (!p.prune)
      for (int i = 0; i < min(kS, n_tiles); ++i) load_tile(i);
  }
  if (warp == 1) tmem_alloc(&tmem_base, 256);
  if (D < kDP) {  // no second box of key dims: that part of the operand image is zero
    for (int i = tid; i < 3 * kBoxBytes / 16; i += kResThreads)
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
  for (int i = tid; i < kHot; i += kResThreads) s_hot[i] = 0u;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tmem_base;

  bool gather = false;
  int32_t* list = p.cand + (size_t)u * p.T + t_begin;  // this CTA's remaining positions, in any order
  if (p.prune) {
    const int g0 = u / p.hs * p.hs;  // the selection group's first unit
    for (int h = warp; h < p.hs; h += kResThreads / 32) {
      float a2 = 0.f, f2 = 0.f;
#pragma unroll
      for (int j = 0; j < kDP; j += 32) {
        const float x = p.mv0[(size_t)(g0 + h) * kDP + j + lane];
        a2 = fmaf(x, x, a2);
        if (j < p.n_fro) f2 += p.fro[(size_t)(g0 + h) * kDP + j + lane];
      }
      a2 = warp_sum(a2);
      f2 = warp_sum(f2);
      if (lane == 0) {
        s_mvn[h] = sqrtf(a2);
        s_fro[h] = scale * sqrtf(f2);
        s_sel[h] = p.hs == 1 ? p.B : min(max(p.cnt[g0 + h], 0), p.lsel);
      }
    }
    __syncthreads();
    // theta: the smallest lower bound over the first stage's free rows (0 where
    // a bound says nothing).  All threads walk the group's lists end to end: a
    // warp per head waited for the longest list (adaptive, 16 units of 20K: 6 us
    // of the call).
    float lowest = INFINITY;
    int total = 0;
    for (int h = 0; h < p.hs; ++h) total += s_sel[h];
    constexpr int kRows = 4;  // rows of a thread whose loads are in flight together
    int hd = 0, first = 0;    // head of the row, and the index of the head's first row
    for (int f0 = tid; f0 < total; f0 += kRows * kResThreads) {
      int t[kRows], hs[kRows];
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        const int f = min(f0 + i * kResThreads, total - 1);
        while (f - first >= s_sel[hd]) first += s_sel[hd++];
        hs[i] = hd;
        t[i] = p.idx[(size_t)(g0 + hd) * p.lsel + f - first];
      }
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        t[i] = min(max(t[i], 0), p.T - 1);
        const size_t at = (size_t)(g0 + hs[i]) * p.T + t[i];
        const float2 nn = reinterpret_cast<const float2*>(p.norms)[at];
        const float vn = sqrtf(nn.y), off = s_mvn[hs[i]] + s_fro[hs[i]] * sqrtf(nn.x);
        const float lb = (vn - off) - kBoundSlack * (vn + off);
        const float b = p.s_in[at] * (lb > 0.f ? lb : 0.f);
        if (!is_protected(t[i], p.T, p.W, p.sink, p.keep_window))
          lowest = fminf(lowest, b > 0.f ? b : 0.f);  // a NaN counts as 0
      }
    }
    const uint32_t wmin = __reduce_min_sync(kFull, __float_as_uint(lowest));
    if (lane == 0) atomicMin(&s_theta, wmin);
    __syncthreads();
    const float theta = __uint_as_float(s_theta) * 0.9999f;  // relative roundings: theta's, ub's and score2's
    const int h = u - g0;
    const float mvn = s_mvn[h], fro = s_fro[h];
    constexpr int kBatch = 8;  // positions per lane whose loads are in flight together
#pragma unroll 1
    for (int t0 = t_begin + warp * 32; t0 < t_end; t0 += kResThreads * kBatch) {
      float2 nn[kBatch];
      float sc[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const int t = min(t0 + i * kResThreads + lane, t_end - 1);
        nn[i] = reinterpret_cast<const float2*>(p.norms)[(size_t)u * p.T + t];
        sc[i] = p.s_in[(size_t)u * p.T + t];
      }
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        const int t = t0 + i * kResThreads + lane;
        const float ub = sc[i] * (sqrtf(nn[i].y) + mvn + fro * sqrtf(nn[i].x));
        const bool cand = t < t_end && !(ub < theta) &&  // a NaN remains
                          !is_protected(t, p.T, p.W, p.sink, p.keep_window);
        if (t < t_end && !cand) p.s_out[(size_t)u * p.T + t] = 0.f;
        const unsigned mask = __ballot_sync(kFull, cand);
        if (mask != 0u) {
          int at = 0;
          if (lane == 0) at = atomicAdd(&s_cnt, __popc(mask));
          at = __shfl_sync(kFull, at, 0) + __popc(mask & ((1u << lane) - 1u));
          if (cand) list[at] = t;
        }
      }
    }
    __syncthreads();
    gather = 2 * s_cnt <= t_end - t_begin;
    if (gather) {
      n_tiles = (s_cnt + kTok - 1) / kTok;
    } else {
      if (tid == 0) {
        for (int i = 0; i < kS; ++i) {
          asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(smem_addr(&full[i])) : "memory");
          mbar_init(&full[i], 1);
        }
        mbar_fence_init();
      }
      __syncthreads();
    }
  }

  if (warp == 0) {
    if (lane == 0 && !gather) {
      for (int i = s_issued; i < n_tiles; ++i) {
        if (i >= kS && !pwait(&empty[i % kS], (i / kS - 1) & 1, abrt, p.ws, u, p.polls)) break;
        load_tile(i);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t id = idesc_bf16(128, 128, 0, 0);
      const uint64_t dk0 = sdesc_sw128(smem_addr(sK), 16, 1024), dc0 = sdesc_sw128(smem_addr(sC), 16, 1024);
      const bool ok = pwait(&cfull, 0, abrt, p.ws, u, p.polls);
      for (int i = 0; ok && i < n_tiles; ++i) {
        const int s = i & 1;
        if (!pwait(&full[s], (i >> 1) & 1, abrt, p.ws, u, p.polls)) break;
        if (i >= 2 && !pwait(&yempty[s], ((i >> 1) - 1) & 1, abrt, p.ws, u, p.polls)) break;
        tc_fence_after();
#pragma unroll
        for (int part = 0; part < 3; ++part)
          umma_k128(tm + s * 128, dk0 + s * (kTileBytes >> 4), dc0 + part * (kTileBytes >> 4), kBoxBytes, kBoxBytes, id,
                    part > 0 ? 1u : 0u);
        umma_commit(&yfull[s]);
        umma_commit(&empty[s]);
      }
      umma_commit(&mma_done);  // every MMA issued has completed
    }
  } else {
    // two epilogue groups (warps 2..5 and 6..9) take alternate tiles; group g
    // always reads stage g and TMEM buffer g
    const int grp = (warp - 2) >> 2, qd = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(qd * 32) << 16;
    const int row = qd * 32 + lane;  // row within the tile = TMEM lane
    for (int i = grp; i < n_tiles; i += 2) {
      const int s = i % kS, j = i / kS, b = i & 1;
      int t = t_begin + i * kTok + row;
      bool live = t < t_end;
      if (gather) {
        // this warp's 32 rows of the list into the stage (free: the group is
        // done with its tile i - 2, whose MMAs it waited for): 16 chunks of k
        // and 16 of v a row, a row per step
        live = i * kTok + row < s_cnt;
        t = live ? list[i * kTok + row] : -1;
#pragma unroll 4
        for (int r = 0; r < 32; ++r) {
          const int tr = __shfl_sync(kFull, t, r), c = lane & 15, rr = qd * 32 + r;
          const uint8_t* src = reinterpret_cast<const uint8_t*>(lane < 16 ? p.K : p.V) +
                               (((size_t)u * p.T + max(tr, 0)) * D + (c < D / 8 ? c * 8 : 0)) * 2;
          uint8_t* dst = (lane < 16 ? sK : sV) + s * kTileBytes + (c >> 3) * kBoxBytes + rr * 128 +
                         (((c & 7) ^ (rr & 7)) << 4);
          cp_async16(dst, src, tr >= 0 && c < D / 8 ? 16u : 0u);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[s]);
      }
      if (!pwait_warp(&yfull[b], (i >> 1) & 1, abrt, p.ws, u, p.polls)) break;
      if (!pwait_warp(&full[s], j & 1, abrt, p.ws, u, p.polls)) break;
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
      if (live) {
        const bool prot = is_protected(t, p.T, p.W, p.sink, p.keep_window);
        const float v = prot ? 0.f : p.s_in[(size_t)u * p.T + t] * sqrtf(ss);
        p.s_out[(size_t)u * p.T + t] = v;
        if (!prot) count_bin(key_bin(score_key(v)), s_hot, p.hist + (size_t)u * kBins);
        if (p.diag) p.diag[(size_t)u * p.T + t] = v;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // the MMA thread's final commit, and after an abort the copies in flight
  if (tid == 0) drain_after_abort(full, kS, abort_flag ? s_issued : 0, &cfull, &mma_done);
  flush_bins(s_hot, p.hist + (size_t)u * kBins);
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 256);
  }
}

// ----------------------------------------------------------------- select
// One cluster of kSelCL CTAs per unit.  R = protected + the k highest keys
// among the unit's other positions (ties to the lower position), or with the
// adaptive budget the unit's share of the highest keys among the (head,
// position) pairs f = h * T + t of its batch item's KV heads (ties to the lower
// f); its positions are written ascending, with their count.
//
// The kernel that computed the scores has counted their keys into kBins bins
// (exponent and three mantissa bits), so the bin of the k-th highest is known
// from one scan.  The keys of that bin (about a sixth of k) are exchanged and
// the last selected pair found among them (list_select); one more pass counts
// and one writes.  Two cluster barriers, where a radix select over the keys
// took four passes of three barriers each: alone at 32K, 32 units, 14 us
// against 24.5 (with the rows' gather, now rset's), at 128K 22.6 against 35.
// A unit's contested keys are exchanged over its cluster; the pairs of a batch
// item through global memory (contest_kernel lists them), so that a joint
// selection too has kSelCL CTAs per unit.
// When there are more contested keys than the lists hold (k above about
// 12000, or many equal scores), counts of their next eleven bits, taken as they
// were listed, narrow them down and the scan is repeated; equal keys that
// still do not fit are counted by position.
struct SelectArgs {
  const float* scores;   // [units][T]
  const uint32_t* hist;  // [units][kBins] counts of the unprotected scores' keys
  int T, W, B, sink, keep_window;
  int32_t* idx;       // [units][lsel] selected positions, ascending (workspace)
  int32_t* diag_idx;  // optional copy (one unit per group)
  int lsel;
  int hs;             // units per selection group (1, or the KV heads of a batch item)
  int32_t* cnt;       // [units] rows each unit retains (joint)
  unsigned long long* glist;  // [groups][kGroupCont] contested pairs of a group (joint)
  int32_t* gcnt;              // [groups] their count
  uint32_t* sub;              // [groups][kBins] their second-level counts
};

constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelCL = 8;         // CTAs per unit (one cluster), each over a contiguous range of positions
constexpr int kMaxCont = 256;     // keys of the contested bin a CTA may hold
static_assert(kGroupCont == kSelCL * kMaxCont, "one list serves both");
constexpr int kSelBatch = 8;      // positions per lane loaded together

// pairs are ordered by (key, ~f): a higher key first, at equal keys the lower f
__device__ __forceinline__ unsigned long long select_pair(float s, int f) {
  return (static_cast<unsigned long long>(score_key(s)) << 32) | (0xffffffffu - static_cast<unsigned>(f));
}

// Exclusive sum over the block of one count per warp; the total in *total.
__device__ __forceinline__ int block_counts(int mine, int* s_w, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) s_w[warp] = mine;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll 4
  for (int w = 0; w < kSelWarps; ++w) {
    before += w < warp ? s_w[w] : 0;
    all += s_w[w];
  }
  *total = all;
  return before;
}

// Of kBins counts, thread t holding the four bins 4 (kSelThreads - 1 - t) ..,
// the bin where their descending sum reaches k > 0, how many of its keys are
// selected, and (if s_left) how many it has, into *s_bin, *s_need and *s_left.
__device__ __forceinline__ void threshold_of(const uint4& c, int k, int* s_w, int* s_bin, int* s_need,
                                             int* s_left = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31;
  static_assert(kBins == 4 * kSelThreads, "four bins per thread");
  const int b[4] = {(int)c.w, (int)c.z, (int)c.y, (int)c.x};
  int incl = b[0] + b[1] + b[2] + b[3];
  const int mine = incl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  int total;
  int above = block_counts(__shfl_sync(kFull, incl, 31), s_w, &total) + incl - mine;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if (above < k && above + b[e] >= k) {  // one bin of the block
      *s_bin = kBins - 1 - (tid * 4 + e);
      *s_need = k - above;
      if (s_left != nullptr) *s_left = b[e];
    }
    above += b[e];
  }
  __syncthreads();
}

// The bin of the group's k-th highest key.
__device__ __forceinline__ void threshold_bin(const SelectArgs& a, int grp, int k, int* s_w, int* s_bin, int* s_need) {
  uint4 c = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 4
  for (int h = 0; h < a.hs; ++h) {
    const uint4 x =
        reinterpret_cast<const uint4*>(a.hist + ((size_t)grp * a.hs + h) * kBins)[kBins / 4 - 1 - threadIdx.x];
    c.x += x.x;
    c.y += x.y;
    c.z += x.z;
    c.w += x.w;
  }
  threshold_of(c, k, s_w, s_bin, s_need);
}

// fn(position, in range, pair) for the positions [w0, w1) of one unit, a warp's
// share, kSelBatch x 32 loads in flight; f0 = the unit's first pair.  A
// protected position's pair stands above all.
template <typename F>
__device__ __forceinline__ void each_pair(const SelectArgs& a, const float* sc, int w0, int w1, int f0, F&& fn) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int t0 = w0; t0 < w1; t0 += 32 * kSelBatch) {
    float s[kSelBatch];
#pragma unroll
    for (int i = 0; i < kSelBatch; ++i) {
      const int t = t0 + i * 32 + lane;
      s[i] = t < w1 ? sc[t] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < kSelBatch; ++i) {
      if (t0 + i * 32 >= w1) break;  // warp-uniform
      const int t = t0 + i * 32 + lane;
      fn(t, t < w1, is_protected(t, a.T, a.W, a.sink, a.keep_window) ? ~0ull : select_pair(s[i], f0 + t));
    }
  }
}

// One addition to a slot counter and to a table of counts for the lanes of a
// warp with `is`: the counter once per warp, the table once where all agree on
// the bin (as equal scores do).  Returns the lane's slot.
__device__ __forceinline__ int warp_append(bool is, int d, int* n, uint32_t* counts) {
  const int lane = threadIdx.x & 31;
  const unsigned mask = __ballot_sync(kFull, is);
  if (mask == 0u) return 0;
  const int first = __ffs(mask) - 1, d0 = __shfl_sync(kFull, d, first);
  int slot = 0;
  if (lane == first) slot = atomicAdd(n, __popc(mask));
  slot = __shfl_sync(kFull, slot, first) + __popc(mask & ((1u << lane) - 1u));
  if (__all_sync(kFull, !is || d == d0)) {
    if (lane == first) atomicAdd(&counts[d0], static_cast<uint32_t>(__popc(mask)));
  } else if (is) {
    atomicAdd(&counts[d], 1u);
  }
  return slot;
}

// The need-th highest of the list's pairs (lists by CTA, s_cn[r] pairs at r *
// kMaxCont, all with p >> bits == pre), into *s_last; need is at most their
// number.  A pair's rank among
// kRankMax or fewer is counted by comparing; more are narrowed down before by
// counts of eleven of their bits at a time (32K, 8 units, budget 8192, about
// 1400 pairs: a selection 108 us with all compared, 15 narrowed).
constexpr int kRankMax = 64;
__device__ __forceinline__ void list_select(const unsigned long long* s_cont, const int* s_cn, int m, int need,
                                            unsigned long long pre, int bits, uint32_t* s_hist, unsigned long long* s_few, int* s_n, int* s_w, int* s_bin,
                                            int* s_need, unsigned long long* s_last) {
  const int tid = threadIdx.x;
  auto each = [&](auto&& fn) {
    for (int i = tid; i < m; i += kSelThreads) {
      int j = i, r = 0;
      while (j >= s_cn[r]) j -= s_cn[r++];
      fn(s_cont[r * kMaxCont + j]);
    }
  };
  int left = m;  // candidates: the pairs with p >> bits == pre
  while (left > kRankMax && bits > 0) {
    const int w = min(bits, 11), sh = bits - w;
    for (int i = tid; i < kBins; i += kSelThreads) s_hist[i] = 0u;
    __syncthreads();
    each([&](unsigned long long p) {
      if (bits > 63 || p >> bits == pre) atomicAdd(&s_hist[(p >> sh) & ((1u << w) - 1u)], 1u);
    });
    __syncthreads();
    threshold_of(reinterpret_cast<const uint4*>(s_hist)[kBins / 4 - 1 - tid], need, s_w, s_bin, s_need);
    pre = pre << w | static_cast<unsigned>(*s_bin);
    bits = sh;
    need = *s_need;
    left = static_cast<int>(s_hist[*s_bin]);
    __syncthreads();
  }
  if (tid == 0) *s_n = 0;
  __syncthreads();
  each([&](unsigned long long p) {
    if (bits > 63 || p >> bits == pre) {
      const int slot = atomicAdd(s_n, 1);
      if (slot < kRankMax) s_few[slot] = p;
    }
  });
  __syncthreads();
  const int few = min(*s_n, kRankMax);
  if (tid < few) {
    const unsigned long long p = s_few[tid];
    int before = 0;
#pragma unroll 4
    for (int j = 0; j < few; ++j) before += s_few[j] > p ? 1 : 0;
    if (before == need - 1) *s_last = p;
  }
  __syncthreads();
}

// The contested pairs of joint selections: grid (kSelCL, units), every CTA's
// part of its unit's positions, into the group's list.
__global__ void __launch_bounds__(kSelThreads) contest_kernel(const SelectArgs a) {
  __shared__ int s_w[kSelWarps];
  __shared__ int s_bin, s_need, s_n, s_at;
  __shared__ unsigned long long s_cont[kGroupCont];
  const int u = blockIdx.y, grp = u / a.hs, h = u % a.hs, tid = threadIdx.x, warp = tid >> 5;
  const int k = a.hs * (a.B - protected_count(a.T, a.W, a.sink, a.keep_window));
  if (tid == 0) {
    s_n = 0;
    s_bin = kBins;
  }
  grid_dependency_wait();
  grid_launch_dependents();
  if (k <= 0) return;
  __syncthreads();
  threshold_bin(a, grp, k, s_w, &s_bin, &s_need);
  const int bin = s_bin, per = (a.T + kSelCL * kSelWarps - 1) / (kSelCL * kSelWarps);
  const int w0 = min(a.T, (static_cast<int>(blockIdx.x) * kSelWarps + warp) * per), w1 = min(a.T, w0 + per);
  each_pair(a, a.scores + (size_t)u * a.T, w0, w1, h * a.T, [&](int, bool in, unsigned long long p) {
    const uint32_t key = static_cast<uint32_t>(p >> 32);
    const bool is = in && p != ~0ull && key_bin(key) == bin;
    const int slot = warp_append(is, sub_bin(bin, key), &s_n, a.sub + (size_t)grp * kBins);
    if (is && slot < kGroupCont) s_cont[slot] = p;
  });
  __syncthreads();
  if (tid == 0) s_at = atomicAdd(a.gcnt + grp, s_n);
  __syncthreads();
  for (int i = tid; i < min(s_n, kGroupCont); i += kSelThreads)
    if (s_at + i < kGroupCont) a.glist[(size_t)grp * kGroupCont + s_at + i] = s_cont[i];
}

template <bool JOINT>
__global__ void __cluster_dims__(kSelCL, 1, 1) __launch_bounds__(kSelThreads, 2) select_kernel(const SelectArgs a) {
  __shared__ int s_w[kSelWarps];
  __shared__ int s_bin, s_need, s_left;
  __shared__ int s_n;            // this CTA's contested keys
  __shared__ int s_cn[kSelCL];   // every CTA's (written remotely)
  // the unit's contested pairs by CTA (written remotely), or the group's list
  __shared__ unsigned long long s_cont[kSelCL * kMaxCont];
  __shared__ __align__(16) uint32_t s_hist[kBins];  // this CTA's counts of the contested keys' next bits (read remotely)
  __shared__ int s_tie[kMaxHs];                     // and of its equal keys per unit (read remotely)
  __shared__ unsigned long long s_few[kRankMax];
  __shared__ unsigned long long s_last;  // the last selected pair (written remotely when joint)
  __shared__ int s_tot[2][kSelCL];       // every CTA's counts (written remotely)
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = static_cast<int>(cluster.block_rank());
  const int u = blockIdx.x / kSelCL, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int T = a.T, hs = JOINT ? a.hs : 1, grp = u / hs, h = u % hs;
  const int prot = protected_count(T, a.W, a.sink, a.keep_window);
  const int k = hs * (a.B - prot);  // >= 0 (validated), < candidates
  const float* sc = a.scores + (size_t)u * T;
  const float* sc0 = a.scores + (size_t)grp * hs * T;  // the group's first unit
  // warp w of CTA r takes the contiguous positions [w0, w1)
  const int per = (T + kSelCL * kSelWarps - 1) / (kSelCL * kSelWarps);
  const int w0 = min(T, (rank * kSelWarps + warp) * per), w1 = min(T, w0 + per);
  if (tid == 0) {
    s_n = 0;
    s_bin = kBins;
    s_need = 0;
    s_last = ~0ull;
  }
  __syncthreads();
  // every CTA has started, with its initial values in place (release): awaited
  // before the first remote store
  cluster_arrive_release();
  grid_dependency_wait();
  grid_launch_dependents();

  if (k > 0) {
    threshold_bin(a, grp, k, s_w, &s_bin, &s_need);
    const int bin = s_bin;
    int need = s_need;  // of the contested keys, how many are selected
    // contested: the keys of the bin, or (bits >= 0) those with key >> bits == pre
    uint32_t pre = 0u;
    int bits = -1;
    auto contested = [&](uint32_t key) { return bits < 0 ? key_bin(key) == bin : key >> bits == pre; };
    int left = 0;  // keys contested, where known
    auto narrow = [&](int d) {  // to the digit d that the counts gave, of the next 11 bits
      need = s_need;
      left = s_left;
      if (bits >= 0) {
        const int w = min(bits, 11);
        pre = pre << w | static_cast<uint32_t>(d);
        bits -= w;
      } else if (bin > 0) {
        pre = (0x800u | static_cast<uint32_t>(bin)) << 11 | static_cast<uint32_t>(d);
        bits = 9;
      } else {
        pre = d >= 1024 ? 0x200000u | (d & 1023u) : static_cast<uint32_t>(d);
        bits = d >= 1024 ? 10 : 21;
      }
    };
    // the pair to find is in the lists, whose lengths are s_cn
    auto from_lists = [&](int m) {
      const unsigned long long p0 = bits >= 0 ? pre : bin > 0 ? 0x800u | static_cast<uint32_t>(bin) : 0u;
      list_select(s_cont, s_cn, m, need, p0, bits >= 0 ? bits + 32 : bin > 0 ? 52 : 64, s_hist, s_few, &s_n, s_w, &s_bin,
                  &s_need, &s_last);
    };
    // this CTA's list to every CTA, unless it overflowed; whether all fit, and their sum
    auto exchange = [&](int& m) -> bool {
      const int mn = s_n;
      if (tid < kSelCL) *cluster.map_shared_rank(&s_cn[rank], tid) = mn;
      if (mn <= kMaxCont)
        for (int i = tid; i < mn * kSelCL; i += kSelThreads) {
          const int r = i % kSelCL, e = rank * kMaxCont + i / kSelCL;
          if (r != rank) *cluster.map_shared_rank(&s_cont[e], r) = s_cont[e];
        }
      cluster.sync();
      bool fit = true;
      m = 0;
      for (int r = 0; r < kSelCL; ++r) {
        fit &= s_cn[r] <= kMaxCont;
        m += s_cn[r];
      }
      return fit;
    };
    // the cluster's counts of the contested keys' next digit
    auto narrow_by_counts = [&]() {
      uint4 c = make_uint4(0u, 0u, 0u, 0u);
      for (int r = 0; r < kSelCL; ++r) {
        const uint4 x = reinterpret_cast<const uint4*>(cluster.map_shared_rank(s_hist, r))[kBins / 4 - 1 - tid];
        c.x += x.x;
        c.y += x.y;
        c.z += x.z;
        c.w += x.w;
      }
      threshold_of(c, need, s_w, &s_bin, &s_need, &s_left);
      narrow(s_bin);
    };
    // ---- scan of the group's units: the contested keys into this CTA's list,
    // and their next digit counted
    auto scan = [&]() {
      for (int i = tid; i < kBins; i += kSelThreads) s_hist[i] = 0u;
      if (tid == 0) s_n = 0;
      __syncthreads();
      const int w = min(max(bits, 0), 11), sh = max(bits, 0) - w;
#pragma unroll 1
      for (int g = 0; g < hs; ++g)
        each_pair(a, sc0 + (size_t)g * T, w0, w1, g * T, [&](int, bool in, unsigned long long p) {
          const uint32_t key = static_cast<uint32_t>(p >> 32);
          const bool is = in && p != ~0ull && contested(key);
          const int d = bits < 0 ? sub_bin(bin, key) : static_cast<int>((key >> sh) & ((1u << w) - 1u));
          const int slot = warp_append(is, d, &s_n, s_hist);
          if (is && slot < kMaxCont) s_cont[rank * kMaxCont + slot] = p;
        });
      __syncthreads();
    };
    int m;
    bool found;
    if constexpr (JOINT) {
      cluster_wait_acquire();
      m = a.gcnt[grp];
      found = m <= kGroupCont;
      if (found) {  // contest_kernel's list, in parts as the clusters' lists are
        for (int i = tid; i < m; i += kSelThreads) s_cont[i] = a.glist[(size_t)grp * kGroupCont + i];
        if (tid < kSelCL) s_cn[tid] = min(max(m - tid * kMaxCont, 0), kMaxCont);
        __syncthreads();
        from_lists(m);
      } else {
        const uint4 c = reinterpret_cast<const uint4*>(a.sub + (size_t)grp * kBins)[kBins / 4 - 1 - tid];
        threshold_of(c, need, s_w, &s_bin, &s_need, &s_left);
        narrow(s_bin);
      }
    } else {
      // ---- the contested keys: this CTA's into every CTA's list
      each_pair(a, sc, w0, w1, 0, [&](int, bool in, unsigned long long p) {
        if (in && p != ~0ull && key_bin(static_cast<uint32_t>(p >> 32)) == bin) {
          const int slot = atomicAdd(&s_n, 1);
          if (slot < kMaxCont) s_cont[rank * kMaxCont + slot] = p;
        }
      });
      __syncthreads();
      cluster_wait_acquire();
      found = exchange(m);
      if (found) {
        from_lists(m);
      } else {
        cluster.sync();  // every CTA is done with s_cn
        scan();
        cluster.sync();
        narrow_by_counts();
      }
    }
#pragma unroll 1
    while (!found) {
      cluster.sync();  // the lists and counts of the scan before are read
      const bool equal = bits == 0 && left > kGroupCont;  // uniform over the cluster
      if (!equal) scan();
      if (!equal && exchange(m)) {
        from_lists(m);
        found = true;
      } else if (bits != 0) {
        narrow_by_counts();
      } else {
        // ---- equal keys: the need-th by unit and position, from the counts of every (unit, CTA)
        for (int g = tid; g < hs; g += kSelThreads) s_tie[g] = 0;
        __syncthreads();
        auto tied = [&](int g, auto&& fn) {
          each_pair(a, sc0 + (size_t)g * T, w0, w1, g * T, [&](int, bool in, unsigned long long p) {
            const bool is = in && p != ~0ull && static_cast<uint32_t>(p >> 32) == pre;
            fn(__ballot_sync(kFull, is), p);
          });
        };
#pragma unroll 1
        for (int g = 0; g < hs; ++g) {
          int c = 0;
          tied(g, [&](unsigned mask, unsigned long long) { c += __popc(mask); });
          if (lane == 0) atomicAdd(&s_tie[g], c);
        }
        cluster.sync();
        if (tid == 0) s_bin = -1;
        static_assert(kMaxHs * kSelCL <= kSelThreads, "one count per thread");
        const int mine = tid < hs * kSelCL ? cluster.map_shared_rank(s_tie, tid % kSelCL)[tid / kSelCL] : 0;
        int incl = mine, total;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += y;
        }
        incl += block_counts(__shfl_sync(kFull, incl, 31), s_w, &total);
        if (incl >= need && incl - mine < need) {  // one thread
          s_bin = tid;
          s_need = need - (incl - mine);
        }
        __syncthreads();
        if (s_bin % kSelCL == rank) {  // uniform over the CTA: it holds the pair
          const int g = s_bin / kSelCL, left = s_need;
          int c = 0;
          tied(g, [&](unsigned mask, unsigned long long) { c += __popc(mask); });
          int run = block_counts(c, s_w, &total);
          if (run < left && run + c >= left)  // one warp
            tied(g, [&](unsigned mask, unsigned long long p) {
              if (((mask >> lane) & 1u) && run + __popc(mask & ((1u << lane) - 1u)) == left - 1)
                for (int r = 0; r < kSelCL; ++r) *cluster.map_shared_rank(&s_last, r) = p;
              run += __popc(mask);
            });
        }
        found = true;
        cluster.sync();
      }
    }
  } else {
    cluster_wait_acquire();
  }

  // ---- this CTA's selections, then everybody's: protected positions and those not below the last
  const unsigned long long last = s_last;
  int c = 0;
  each_pair(a, sc, w0, w1, h * T,
            [&](int, bool in, unsigned long long p) { c += __popc(__ballot_sync(kFull, in && p >= last)); });
  int tot;
  int o = block_counts(c, s_w, &tot);
  if (tid < kSelCL) *cluster.map_shared_rank(&s_tot[0][rank], tid) = tot;
  cluster.sync();
  for (int r = 0; r < rank; ++r) o += s_tot[0][r];
  int32_t* out = a.idx + (size_t)u * a.lsel;
  each_pair(a, sc, w0, w1, h * T, [&](int t, bool in, unsigned long long p) {
    const bool sel = in && p >= last;
    const unsigned mask = __ballot_sync(kFull, sel);
    const int at = o + __popc(mask & ((1u << lane) - 1u));
    if (sel && at < a.lsel) {
      out[at] = t;
      if (!JOINT && a.diag_idx) a.diag_idx[(size_t)u * a.lsel + at] = t;
    }
    o += __popc(mask);
  });
  if (JOINT && rank == 0 && tid == 0) {
    int x = 0;
    for (int r = 0; r < kSelCL; ++r) x += s_tot[0][r];
    a.cnt[u] = min(x, a.lsel);
  }
  // no remote access follows the last cluster barrier
}

// The first stage's joint list for inspection, [groups][hs * B] of h * T + t,
// ascending: one CTA per group, from its units' lists.
__global__ void __launch_bounds__(256) diag_joint_kernel(const SelectArgs a) {
  int o = 0;
  for (int h = 0; h < a.hs; ++h) {
    const int u = blockIdx.x * a.hs + h, c = a.cnt[u];
    for (int i = threadIdx.x; i < c; i += 256)
      if (o + i < a.hs * a.B)
        a.diag_idx[(size_t)blockIdx.x * a.hs * a.B + o + i] = h * a.T + a.idx[(size_t)u * a.lsel + i];
    o += c;
  }
}

// ------------------------------------------------------------------- rset
// Moments of E = all \ R for the rows R a selection kept, in one kernel per
// stage: the rows are gathered by their list straight into the tensor-core
// operand layout (no dense copy of them), V^T K of a 128-row tile forms in
// TMEM, the tile's co-moment is centred as it is read from there and added to
// the CTA's earlier ones, and the epilogue takes the sum out of the all-token
// set's co-moment.
// The first stage writes C0' as the residual pass's operand image, the final
// one the caller's moments and, from the same tiles, the retained cache.
//
// Grid (CL * D/64, units), clusters of CL CTAs of 2048 / CL threads: CTA (rank,
// kh) takes the row tiles rank, rank + CL, ... and the key dims [64 kh,
// 64 kh + 64); the CL partial sums meet through distributed shared memory,
// each rank finishing 128 / CL value dims, four elements of C per thread.  A
// chain of round trips (list, rows, MMA, exchange) over code that runs once:
// its time is latency and instruction fetch, so the loops stay rolled.  Alone
// at 32K, 32 units, it takes 16 us, where a second pass of stats_tc over
// gathered rows (13.5) and a merge kernel (11.5) took 25; its merge runs while
// the selection does, and the gathered copies are gone.
//
// The all-token co-moment is the multi-way Chan merge of the chunk records,
// taken about the first chunk's means x0 so that no global mean is needed first:
//   M = sum_ch [M_ch + n_ch d_ch d_ch^T] - n dbar dbar^T,  d_ch = mu_ch - x0,
//   dbar = sum_ch n_ch d_ch / n,  mu = x0 + dbar.
// It is merged before the dependency wait, while the selection runs: the
// records are stats_tc's, complete before the selection's predecessor (which
// the selection has waited for when this kernel may start) began.
// R's tiles and ranks are merged about the same x0, and R's centred record is
// then removed with the reverse pairwise formula.  The centring tile by tile
// matters where channels have means of several standard deviations: taken out
// once over all of R (4096 of 8192 rows, means of 10 and 4), it left C 25 times
// as far from 64 bits as fp32 sums need.
constexpr int kFinCH = 32;      // chunk records staged per pass
constexpr int kRsRed = 64 + 4;  // row stride of a CTA's partial sums (floats)
constexpr int kRsOperands = kBoxBytes + kTileBytes + 2048;  // one K half, one V tile, ones
constexpr size_t rset_smem(bool several) {
  return 1024 + kRsOperands + (several ? (size_t)kDP * kRsRed * 4 : 0);
}

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
  int several;  // a CTA may have more than one row tile
};

// x0 + (s - r) / n, the roundings of the difference and the quotient put back:
// where the means are near zero they weigh as x0 (a chunk's mean) does.
__device__ __forceinline__ float mean_about(float x0, float s, float r, float n, float inv) {  // inv = 1 / n
  const float t = s - r, b = t - s, err = (s - (t - b)) - (r + b);
  const float q = t * inv;
  return (x0 + q) + (fmaf(-q, n, t) + err) * inv;
}

template <int CL, bool FINAL>
__global__ void __launch_bounds__(2048 / CL, CL == 2 ? 1 : 2) rset_kernel(const RsetArgs a) {
  constexpr int kThr = 2048 / CL;
  constexpr int RW = kDP / CL;  // value dims a rank finishes
  extern __shared__ __align__(1024) uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = sm;                               // [128 rows][64 key dims]
  uint8_t* sV = sm + kBoxBytes;                   // [2 boxes][128 rows][64 value dims]
  uint8_t* sOnes = sm + kBoxBytes + kTileBytes;   // [16 rows][128 B] of bf16 1.0
  // [128][kRsRed] this CTA's V^T K about x0: over the operands of its only tile, or past them
  float* red = reinterpret_cast<float*>(sm + (a.several ? kRsOperands : 0));
  __shared__ __align__(8) uint64_t done;
  __shared__ uint32_t tmem_base;
  __shared__ int s_ok;
  __shared__ int s_t[kTok];                              // positions of a tile's rows, -1 past the unit's rows
  __shared__ __align__(16) float s_sk[64], s_sv[kDP];  // this CTA's column sums about x0 (read remotely)
  __shared__ __align__(16) float s_x0k[64], s_tk[64];   // x0 of the key half, and a tile's sums of K
  const Layout& L = a.L;
  const int D = L.D, T = L.T;
  const int rank = blockIdx.x % CL, kh = blockIdx.x / CL, u = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cq = tid % 16, row = rank * RW + tid / 16;  // this thread's four elements: (row, kh*64 + 4 cq ..)

  if (tid == 0) {
    mbar_init(&done, 1);
    mbar_fence_init();
    s_ok = 1;
  }
  if (warp == 0) tmem_alloc(&tmem_base, 128);

  // ---- the all-token set: this thread's elements of M and its means
  const size_t rf = L.rec;
  const float* recs = L.mpart + (size_t)u * L.n_chunks * rf;
  float n = 0.f, sv = 0.f, x0v = 0.f, sk[4] = {0.f, 0.f, 0.f, 0.f}, x0k[4] = {0.f, 0.f, 0.f, 0.f};
  float M[4] = {0.f, 0.f, 0.f, 0.f};
  {
    float* s_n = reinterpret_cast<float*>(sm);  // [kFinCH]
    float* s_mk = s_n + kFinCH;                 // [kFinCH][64]
    float* s_mv = s_mk + kFinCH * 64;           // [kFinCH][RW]
#pragma unroll 1
    for (int g0 = 0; g0 < L.n_chunks; g0 += kFinCH) {
      const int nb = min(kFinCH, L.n_chunks - g0);
      if (g0 > 0) __syncthreads();
      constexpr int per = 1 + 16 + RW / 4;  // float4s per record: n, 64 key means, RW value means
#pragma unroll 2
      for (int i = tid; i < nb * per; i += kThr) {
        const int ch = i / per, j = i % per;
        const float* r = recs + (size_t)(g0 + ch) * rf;
        const int c = rank * RW + (j - 17) * 4;  // value dims past D are zero
        const float* src = j == 0 ? r : j <= 16 ? r + 4 + kh * 64 + (j - 1) * 4 : r + 4 + D + c;
        float* dst = j <= 16 ? s_mk + ch * 64 + (j - 1) * 4 : s_mv + ch * RW + (j - 17) * 4;
        const float4 v =
            j <= 16 || c < D ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (j == 0) s_n[ch] = v.x;
        else *reinterpret_cast<float4*>(dst) = v;
      }
      __syncthreads();
      if (g0 == 0) {
#pragma unroll
        for (int j = 0; j < 4; ++j) x0k[j] = s_mk[cq * 4 + j];
        x0v = s_mv[tid / 16];
        if (tid < 64) s_x0k[tid] = s_mk[tid];
      }
      const float* m = recs + (size_t)g0 * rf + 4 + 2 * D + (size_t)min(row, D - 1) * D + kh * 64 + cq * 4;
#pragma unroll 4
      for (int ch = 0; ch < nb; ++ch) {
        const float4 m4 = *reinterpret_cast<const float4*>(m + (size_t)ch * rf);
        const float nc = s_n[ch];
        if (nc > 0.f) {  // an empty record's co-moment is never written
          const float4 k4 = *reinterpret_cast<const float4*>(s_mk + ch * 64 + cq * 4);
          const float dk[4] = {k4.x - x0k[0], k4.y - x0k[1], k4.z - x0k[2], k4.w - x0k[3]};
          const float mm[4] = {m4.x, m4.y, m4.z, m4.w};
          const float dv = s_mv[ch * RW + tid / 16] - x0v;
          n += nc;
          sv = fmaf(nc, dv, sv);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            sk[j] = fmaf(nc, dk[j], sk[j]);
            M[j] += mm[j] + nc * dv * dk[j];
          }
        }
      }
    }
  }
  __syncthreads();  // the staged records give way to the row tiles
  if (D < kDP)      // no second box of value dims
    for (int i = tid; i < kBoxBytes / 16; i += kThr)
      reinterpret_cast<uint4*>(sV + kBoxBytes)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid < 2048 / 16)  // the ones operand of the column sums
    reinterpret_cast<uint4*>(sOnes)[tid] = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
  grid_dependency_wait();
  // The call's last kernel releases nothing early: a decode step with
  // early_load reads the cache and the moments before its own wait.
  if constexpr (!FINAL) grid_launch_dependents();

  // ---- row tiles
  const int cnt = L.hs == 1 ? L.B : L.cnt[u];
  const int32_t* lst = L.idx + (size_t)u * L.lsel;
  const int n_tiles = (cnt + kTok - 1) / kTok;
  const __nv_bfloat16* Ku = a.K + (size_t)u * T * D + kh * 64;
  const __nv_bfloat16* Vu = a.V + (size_t)u * T * D;
  const int vch = D / 8;  // 16-byte chunks of a value row
  // this thread's TMEM lane (a value dim) and its part of the 64 key columns
  constexpr int kCols = 64 * 128 / kThr;
  const int vrow = (warp & 3) * 32 + lane, c_lo = (warp >> 2) * kCols;
  const uint32_t tm_lane = static_cast<uint32_t>((warp & 3) * 32) << 16;
  const float x0row = vrow < D ? recs[4 + D + vrow] : 0.f;  // x0 of that dim
  float rv_lane = 0.f, rk_lane = 0.f;  // R's sums about x0: of value dim vrow, of key dim tid (tid < 64)
  float* my_red = red + vrow * kRsRed;
  int it = 0;
  bool ok = true;
#pragma unroll 1
  for (int ti = rank; ti < n_tiles; ti += CL, ++it) {
    const int r0 = ti * kTok;
    if (tid < kTok)  // never outside the unit's slab
      s_t[tid] = r0 + tid < cnt ? min(max(lst[r0 + tid], 0), T - 1) : -1;
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < kTok * 8; i += kThr) {  // the key half: 8 chunks a row
      const int r = i / 8, c = i % 8, t = s_t[r];
      cp_async16(sK + r * 128 + ((c ^ (r & 7)) << 4), Ku + (size_t)max(t, 0) * D + c * 8, t >= 0 ? 16u : 0u);
    }
#pragma unroll 1
    for (int i = tid; i < kTok * vch; i += kThr) {  // the value rows
      const int r = i / vch, c = i % vch, t = s_t[r];
      cp_async16(sV + (c >> 3) * kBoxBytes + r * 128 + (((c & 7) ^ (r & 7)) << 4), Vu + (size_t)max(t, 0) * D + c * 8,
                 t >= 0 ? 16u : 0u);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // generic writes -> tensor-core reads
    tc_fence_before();
    __syncthreads();
    if (tid == 0) {
      // V^T K, and the column sums of [K half | V's first box] and of V against
      // ones (the boxes lie one after another), all MN-major over the rows
      tc_fence_after();
      const uint32_t tm = tmem_base, aK = smem_addr(sK), aV = smem_addr(sV), a1 = smem_addr(sOnes);
      const uint32_t id = idesc_bf16(128, 64, 1, 1), id1 = idesc_bf16(128, 16, 1, 0);
#pragma unroll 1
      for (int kk = 0; kk < 8; ++kk) {
        const uint64_t dk = sdesc_sw128(aK + kk * 2048, kBoxBytes, 1024), dv = sdesc_sw128(aV + kk * 2048, kBoxBytes, 1024);
        const uint64_t d1 = sdesc_sw128(a1 + (kk & 3) * 32, 16, 1024);
        const uint32_t acc = kk > 0 ? 1u : 0u;
        umma_bf16(tm, dv, dk, id, acc);
        umma_bf16(tm + 64, dk, d1, id1, acc);
        umma_bf16(tm + 80, dv, d1, id1, acc);
      }
      umma_commit(&done);
    }
    if constexpr (FINAL) {
      // the cache rows from the same tile, this CTA's halves (a joint
      // selection's cache is zero up to the next tile past a unit's rows)
#pragma unroll 1
      for (int i = tid; i < kTok * 8; i += kThr) {
        const int r = i / 8, c = i % 8, to = r0 + r;
        if (to < cnt || (L.hs > 1 && to < a.dst_cap)) {
          const size_t o = ((size_t)u * a.dst_cap + to) * D + kh * 64 + c * 8;
          const uint32_t at = r * 128 + ((c ^ (r & 7)) << 4);
          *reinterpret_cast<uint4*>(a.dst_K + o) = *reinterpret_cast<const uint4*>(sK + at);
          *reinterpret_cast<uint4*>(a.dst_V + o) = *reinterpret_cast<const uint4*>(sV + kh * kBoxBytes + at);
        }
      }
      if (kh == 0 && tid < kTok && r0 + tid < cnt) a.dst_pos[(size_t)u * a.dst_cap + r0 + tid] = s_t[tid];
    }
    if (tid == 0 && !mbar_wait(&done, it & 1, a.polls)) {
      s_ok = 0;
      record_error(a.ws, MKV_ERR_TIMEOUT, u);
    }
    __syncthreads();
    ok = s_ok != 0;
    if (!ok) {  // uniform: s_ok changes only before a barrier
      if (tid == 0) (void)mbar_wait(&done, it & 1);  // drain: the MMAs still read shared memory
      break;
    }
    // ---- the tile's means, then its co-moment about x0 onto the tiles before
    tc_fence_after();
    const float nt = static_cast<float>(min(kTok, cnt - r0));
    if (warp < 2) {  // lanes 64.. hold sums of V's first box: not read
      const float tk = tmem_ld1(tmem_base + tm_lane + 64);
      s_tk[tid] = tk;
      rk_lane += fmaf(-nt, s_x0k[tid], tk);
    }
    const float tv = tmem_ld1(tmem_base + tm_lane + 80);
    rv_lane += fmaf(-nt, x0row, tv);
    float x[kCols];
    tmem_ld<kCols>(tmem_base + tm_lane + c_lo, x);
    __syncthreads();
    const float inv = 1.f / nt, mv = tv / nt, w = nt * (mv - x0row);
#pragma unroll
    for (int j = 0; j < kCols; j += 4) {
      const float4 tk = *reinterpret_cast<const float4*>(s_tk + c_lo + j);
      const float4 xk = *reinterpret_cast<const float4*>(s_x0k + c_lo + j);
      float4* to = reinterpret_cast<float4*>(my_red + c_lo + j);
      float4 y = it > 0 ? *to : make_float4(0.f, 0.f, 0.f, 0.f);
      y.x += fmaf(w, fmaf(tk.x, inv, -xk.x), fmaf(-mv, tk.x, x[j]));
      y.y += fmaf(w, fmaf(tk.y, inv, -xk.y), fmaf(-mv, tk.y, x[j + 1]));
      y.z += fmaf(w, fmaf(tk.z, inv, -xk.z), fmaf(-mv, tk.z, x[j + 2]));
      y.w += fmaf(w, fmaf(tk.w, inv, -xk.w), fmaf(-mv, tk.w, x[j + 3]));
      *to = y;
    }
    tc_fence_before();
  }
  if (it == 0 || !ok) {
    __syncthreads();  // what the operands' set-up wrote there
    for (int c = c_lo; c < c_lo + kCols; c += 4) *reinterpret_cast<float4*>(my_red + c) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (tid < 64) s_sk[tid] = ok ? rk_lane : 0.f;
  if (tid < kDP) s_sv[tid] = ok ? rv_lane : 0.f;
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 128);
  }

  // ---- R's sums over the cluster, and E = all \ R
  const float nR = ok ? static_cast<float>(cnt) : 0.f;
  float SR[4] = {0.f, 0.f, 0.f, 0.f}, rk[4] = {0.f, 0.f, 0.f, 0.f}, rv = 0.f;
#pragma unroll
  for (int r = 0; r < CL; ++r) {  // ranks past the tiles hold zeros; all loads in flight
    const float4 k4 = *reinterpret_cast<const float4*>(cluster.map_shared_rank(s_sk, r) + cq * 4);
    const float4 s4 = *reinterpret_cast<const float4*>(cluster.map_shared_rank(red, r) + row * kRsRed + cq * 4);
    rv += cluster.map_shared_rank(s_sv, r)[row];
    rk[0] += k4.x;
    rk[1] += k4.y;
    rk[2] += k4.z;
    rk[3] += k4.w;
    SR[0] += s4.x;
    SR[1] += s4.y;
    SR[2] += s4.z;
    SR[3] += s4.w;
  }
  const float nE = n - nR;
  // means of R and E about x0
  const float invE = nE > 0.f ? 1.f / nE : 0.f;
  const float dvR = nR > 0.f ? rv / nR : 0.f, dvE = (sv - rv) * invE;
  const float mvE = nE > 0.f ? mean_about(x0v, sv, rv, nE, invE) : 0.f;
  float CE[4], mkE[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float dkR = nR > 0.f ? rk[j] / nR : 0.f;
    CE[j] = mkE[j] = 0.f;
    if (nE > 0.f) {
      const float dkE = (sk[j] - rk[j]) * invE;
      mkE[j] = mean_about(x0k[j], sk[j], rk[j], nE, invE);
      const float Mall = M[j] - sv * sk[j] / n;
      const float MR = nR > 0.f ? SR[j] - rv * rk[j] / nR : 0.f;
      const float ME = Mall - MR - (nE * nR / n) * (dvR - dvE) * (dkR - dkE);
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
    if (kh == 0 && rank == 0 && tid == 0) {
      a.mom.n[u] = static_cast<int32_t>(nE);
      a.dst_len[u] = cnt;
      a.dst_seen[u] = T;
    }
  } else {
    // C0' (clamped where |n0 C0| < tau) as three bf16 parts, K-major operand
    // rows (value dims; zero past D) in the swizzled layout
    float r4[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) r4[j] = (row < D && !(fabsf(CE[j] * nE) < a.tau)) ? CE[j] : 0.f;
    const float fro = warp_sum(r4[0] * r4[0] + r4[1] * r4[1] + r4[2] * r4[2] + r4[3] * r4[3]);
    if (lane == 0) L.fro[(size_t)u * kDP + kh * 64 + rank * (RW / 2) + warp] = fro;  // two rows' part of ||C0'||_F^2
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
  cluster.sync();  // no CTA leaves while another reads its shared memory
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
constexpr size_t kResidualSmem = 2 * 2 * kTileBytes + 3 * kTileBytes;

// residual_tc compares scores and norms before it reads rows when its CTAs
// have at least this many tiles; below, the full pass takes no longer.
constexpr int kPruneTiles = 8;

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

// CTAs per unit and key half of rset_kernel (2048 threads of them in any case:
// the count decides into how many parts a unit's row tiles fall and how often
// its records' means are read).  Four, unless more would still find room and
// have tiles, or fewer do with as many parts.  us of a call with 8 / 4 / 2:
//   8 units, 8K, budgets 512, 1024, 4096: 69.5/63.8/70.3, 76.0/75.0/87.9, 142/156/208
//   16 units, 16K, budget 2048: 177/190/207; 24 units: 230/210/227
//   32 units, 32K, budgets 256, 1500, 4096: 274/246/239, 346/317/330, 530/510/549
//   512 units, 1K, budget 128: 1167/772/726
int rset_cluster(const Layout& L, int num_sms) {
  const long pairs = (long)L.units * (L.D / 64);
  if (L.B > 8 * kTok && 8 * pairs <= 2L * num_sms) return 8;
  return L.B <= 2 * kTok && 4 * pairs > num_sms ? 2 : 4;
}

template <bool FINAL>
cudaError_t launch_rset(RsetArgs a, int cl, cudaStream_t st) {
  const dim3 grid(cl * (a.L.D / 64), a.L.units);
  a.several = a.L.lsel > cl * kTok ? 1 : 0;
  auto go = [&](void (*f)(RsetArgs)) -> cudaError_t {
    const cudaError_t e = smem_attr(reinterpret_cast<const void*>(f), rset_smem(true));
    return e != cudaSuccess ? e : launch_pdl(f, grid, 2048 / cl, rset_smem(a.several != 0), st, cl, a);
  };
  switch (cl) {
    case 8: return go(rset_kernel<8, FINAL>);
    case 4: return go(rset_kernel<4, FINAL>);
    default: return go(rset_kernel<2, FINAL>);
  }
}

cudaError_t run(const CompressArgs& a, const mkv_geom& g, int num_sms, cudaStream_t st) {
  Layout L = make_layout(g, a.T, a.budget, a.window, a.sink, a.keep_window, a.adaptive, num_sms);
  carve(L, a.ws);
  const int D = g.head_dim, T = a.T, B = a.budget, U = L.units;
  const bool keep_all = T <= B;
  cudaError_t e = cudaSuccess;
  if ((e = smem_attr((const void*)stats_tc, std::max(stats_smem(1), stats_smem(2)))) != cudaSuccess) return e;
  if ((e = smem_attr((const void*)scores_tc, std::max(score_smem(1), score_smem(2)))) != cudaSuccess) return e;
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
  tp.hist = L.hist;
  tp.gcnt = L.gcnt;
  tp.sub = L.hs > 1 ? L.sub : nullptr;
  tp.hs = L.hs;
  tp.units = U;
  tp.norms = L.norms;
  tp.ws = a.ws;
  tp.polls = pipeline_poll_limit();
  const dim3 cg(L.n_chunks, U);

  if (!keep_all || a.diag_scores != nullptr) {
    if ((e = launch_pdl(stats_tc, cg, kStatThreads, stats_smem(L.RWb), st, 0, tp, tmK, tmV, tmQ)) != cudaSuccess) return e;
    TcArgs p2 = tp;
    p2.s_out = L.s;
    p2.diag = a.diag_scores;
    if ((e = launch_pdl(scores_tc, cg, kScoreThreads, score_smem(L.RWb), st, 0, p2, tmK, tmQ)) != cudaSuccess) return e;
  }
  if (keep_all) {
    if (D == 128) keep_all_kernel<128><<<dim3((T + 7) / 8, U), 256, 0, st>>>(a, T);
    else keep_all_kernel<64><<<dim3((T + 7) / 8, U), 256, 0, st>>>(a, T);
    return cudaGetLastError();
  }

  auto select = [&](int stage, const float* scores, int32_t* diag_idx) -> cudaError_t {
    SelectArgs sa{};
    sa.scores = scores;
    sa.hist = L.hist + (size_t)stage * U * kBins;
    sa.diag_idx = diag_idx;
    sa.T = T;
    sa.W = a.window;
    sa.B = B;
    sa.sink = a.sink;
    sa.keep_window = a.keep_window;
    sa.idx = L.idx;
    sa.lsel = L.lsel;
    sa.hs = L.hs;
    sa.cnt = L.cnt;
    sa.glist = L.glist;
    sa.gcnt = L.gcnt + (size_t)stage * U;
    sa.sub = L.sub + (size_t)stage * (U / L.hs) * kBins;
    if (L.hs == 1) return launch_pdl(select_kernel<false>, dim3(U * kSelCL), kSelThreads, 0, st, 0, sa);
    cudaError_t se = launch_pdl(contest_kernel, dim3(kSelCL, U), kSelThreads, 0, st, 0, sa);
    if (se == cudaSuccess) se = launch_pdl(select_kernel<true>, dim3(U * kSelCL), kSelThreads, 0, st, 0, sa);
    if (se == cudaSuccess && diag_idx != nullptr) {
      diag_joint_kernel<<<U / L.hs, 256, 0, st>>>(sa);
      se = cudaGetLastError();
    }
    return se;
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

  if ((e = select(0, L.s, a.diag_idx1)) != cudaSuccess) return e;
  if (a.mi) {
    if ((e = launch_rset<false>(ra, cl, st)) != cudaSuccess) return e;
    TcArgs r = tp;
    r.cimg = L.cimg;
    r.mv0 = L.mv0;
    r.s_in = L.s;
    r.s_out = L.s2;
    r.hist = L.hist + (size_t)U * kBins;
    r.diag = a.diag_score2;
    // a second pass over the prompt is worth avoiding from eight tiles a CTA on
    r.prune = a.diag_score2 == nullptr && L.chunk >= kPruneTiles * kTok ? 1 : 0;
    r.B = B;
    r.idx = L.idx;
    r.cnt = L.cnt;
    r.lsel = L.lsel;
    r.fro = L.fro;
    r.n_fro = D;
    r.cand = L.cand;
    r.K = a.K;
    r.V = a.V;
    if ((e = launch_pdl(residual_tc, cg, kResThreads, kResidualSmem, st, 0, r, tmK, tmV)) != cudaSuccess) return e;
    if ((e = select(1, L.s2, nullptr)) != cudaSuccess) return e;
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
