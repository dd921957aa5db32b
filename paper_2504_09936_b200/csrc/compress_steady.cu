// keepkv_compress with KEEPKV_FLAG_COMPRESS_STEADY: Algorithm 1 in one kernel for a cache that is only one
// period over its budget.  A unit qualifies when it evicts at most kStEv entries and has at most kStCand
// entries between the sinks and the recent window; the others are reported and left alone.  The R CTAs of
// a unit (grid (R, U)), eight warps and two that only copy, each
//   1. repeat the selection (Algorithm 1, selection step): keys of the candidates in shared memory, range_select,
//      one ordered pass -> the kept candidates and the evicted entries as lists in shared memory;
//   2. move their slice of the retained slots src -> dst (Algorithm 1, insertion step).  One of the copying warps moves the
//      values, 32 rows at a time, by bulk copies through shared memory, the other votes, score estimates and index outputs;
//      both begin with the recent window, which does not depend on the selection.  Keys go 64 slots at a time
//      global -> shared by cp.async into a ring of 128-byte-swizzled tiles, two tiles ahead of their use, and from there
//      to dst by a TMA store.  The key tiles are the
//      B operand of a tcgen05.mma (M = 128 evicted keys, staged once as A operand; N = 64; fp32 accumulators in tensor
//      memory, double-buffered) that one thread issues per tile (Algorithm 1, similarity step).  All eight
//      warps drain the accumulator of the previous tile with tcgen05.ld while the next product runs: a thread
//      owns one evicted row and half of the columns and keeps the row's two best cosines with their slots, of those
//      above the merge threshold (an entry whose best cosine does not exceed it is dropped whatever its best column was);
//   3. are a cluster: every evicted row has one of them that gets its candidates from all through shared memory, folds them and settles
//      arg-max and threshold (Algorithm 1, arg-max and threshold step) with the interface's exact fp32 chain wherever the tensor-core ranking is
//      closer than kRankEps, and tells all of them; each sorts the entries to merge into the same groups and its warps merge their
//      share of them (Eq. A.3; Algorithm 1, merge step).
// Decisions, and therefore all outputs, are the same bits as the general pipeline's (compress.cu).
// Bound: the chain selection (6 us) -> evicted keys and first tile (5 us) -> tiles (12 us) -> decisions and merges (5 us); the
// bytes of 64 units of 1766 entries, 112 MB, take 17 us at the copy rate.  Every warp copying, searching and selecting in
// turn took 69 us a layer; values through the registers of two copying warps 85 us (they ended at 60-70 us, the search at
// 24); values by bulk copies through shared memory 45 us; with the candidates in global memory and all decisions and merges the
// last CTA's, 29 groups on eight warps.  Shared out over the cluster: 40 us.
// Every wait on the tensor core and on a bulk copy is bounded; one that runs out raises KEEPKV_DEV_TIMEOUT and the CTA goes
// on without further products (its unit's result is then unspecified), frees its tensor memory and returns.
#include "compress.cuh"
#include "ptx.cuh"

namespace keepkv {

constexpr int kStThreads = 256;  // the warps that select, search and merge
constexpr int kStWarps = kStThreads / 32;
constexpr int kStAll = kStThreads + 64;
constexpr int kStCand = 2048;    // candidates (entries between sinks and recent window) a CTA holds keys for
constexpr int kStEv = 128;       // evicted entries per unit (rows of the product, lanes of tensor memory)
constexpr int kStRet = 16384;    // retained entries per unit
constexpr int kStN = 64;         // retained slots per tile (columns of the product)
constexpr int kStTmemCols = 128; // two accumulators of kStN columns
constexpr int kStRows = 32;      // rows of a block of values
constexpr int kStOneCtaSmem = 120 * 1024;   // more than half of an SM's shared memory
constexpr int kStMaxCtas = kNomChunksMax;   // CTAs per unit: a cluster

// Barriers of parts of the CTA.  (Not the aligned form: a warp may come to them from a branch of its lanes.)
struct StSync { __device__ __forceinline__ void operator()() const { asm volatile("barrier.sync 1, 256;" ::: "memory"); } };
__device__ __forceinline__ void st_sync_all(int id) { __syncwarp(); asm volatile("barrier.sync %0, 320;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void st_arrive_all(int id) { __syncwarp(); asm volatile("barrier.arrive %0, 320;" ::"r"(id) : "memory"); }

template <int D>
struct StSmem {
  static constexpr int kSub = D / 64;                            // 64-channel (128-byte) atoms per row
  static constexpr int kABytes = kSub * kStEv * 128;
  static constexpr int kBBytes = kSub * kStN * 128;
  static constexpr int kStages = 3;
  static constexpr int kStageBytes = kBBytes;                    // one stage: a key tile, swizzled
  static constexpr int kA = 0;                                   // evicted keys, swizzled
  static constexpr int kRing = kA + kABytes;
  static constexpr int kVal = kRing + kStages * kStageBytes;     // bf16 [2][kStRows][D]  values on their way
  static constexpr int kCinv = kVal + 2 * kStRows * D * 2;       // f32 [4][64]   1/|k| of the keys of four tiles
  static constexpr int kEinv = kCinv + 4 * kStN * 4;             // f32 [kStEv]   1/|k_e|
  static constexpr int kXchg = kEinv + kStEv * 4;                // u32 [kStEv][4] column-half exchange
  static constexpr int kHeavy = kXchg + kStEv * 16;              // i32 [kStCand] source index of kept candidates
  static constexpr int kEv = kHeavy + kStCand * 4;               // i32 [kStEv]   source index of evicted entries
  // what the CTAs of a unit tell one another: a row's candidates go to the CTA that settles it, its target to all
  static constexpr int kInbox = kEv + kStEv * 4;                 // uint4 [R][kStEv / R, rounded up]
  static constexpr int kDec = kInbox + (kStEv + kStMaxCtas) * 16; // i32 [kStEv]   slot to merge into, or -1
  static constexpr int kBytes = kDec + kStEv * 4;
  static constexpr int kKeys = kA;                               // u32 [kStCand] selection keys, gone before A is staged
  static constexpr int kHist = kRing + 2 * kStageBytes;          // i32 [kSelBins] in the stage that is filled last
  // scratch of the last CTA, laid over the operand tiles once the similarity search is over
  static constexpr int kKe = 0;                                  // f32 [kStWarps][D]
  static constexpr int kKc = kKe + kStWarps * D * 4;             // f32 [kStWarps][2][D]
  static constexpr int kQ = kKc + kStWarps * 2 * D * 4;          // i32 [7][kStEv]
  static constexpr int kSkey = kQ + 7 * kStEv * 4;               // u32 [kStEv]
  static constexpr int kGhead = kSkey + kStEv * 4;               // i32 [kStEv + 1]
  static_assert(kGhead + (kStEv + 1) * 4 <= kVal, "tail scratch must fit the operand tiles");
  static_assert(kStCand * 4 <= kABytes, "selection keys must fit the A tile");
  static_assert(kSelBins * 4 <= kStageBytes, "selection bins must fit a stage");
};

// kCluster: a unit's CTAs are a cluster, which settles the candidates and the merges together.  Otherwise they leave them in
// global memory (nom), and the unit's last CTA to arrive does all of it.
template <int D, bool kCluster>
__global__ void __launch_bounds__(kStAll, 2)
steady_compress_kernel(const __grid_constant__ CUtensorMap mapD, keepkv_params p, keepkv_cache src, keepkv_cache dst,
                       const int32_t *budget_dev, int budget_scalar,
                       const int32_t *n_recent_dev, int32_t *ret_idx, int32_t *target, uint4 *nom, int C_max, int *counters,
                       keepkv_stats *stats, int32_t *status_dev, const float *__restrict__ select_key, int spin_limit, int withhold) {
  using SL = StSmem<D>;
  constexpr int KSTEPS = D / 16;          // k-steps of the similarity product
  constexpr int CH = D / 8;               // 16-byte chunks of a row
  constexpr int RP = kStThreads / CH;     // rows the CTA requests per pass (one chunk per thread)
  constexpr int NP = kStN / RP;           // passes per 64-slot tile
  constexpr uint32_t IDESC = umma_idesc_bf16(kStEv, kStN);
  extern __shared__ __align__(1024) uint8_t st_smem_raw[];
  __shared__ int warp_tot[32];
  __shared__ uint32_t s_kmin[kStWarps], s_kmax[kStWarps];
  __shared__ int s_sel[4];
  __shared__ int s_last, s_nq;
  __shared__ __align__(8) uint64_t bars[5];   // t_full[2], drain, v_full[2]
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  uint8_t *st_smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(st_smem_raw) + 1023) & ~(uintptr_t)1023);
  float *cinv = reinterpret_cast<float *>(st_smem + SL::kCinv);
  float *einv = reinterpret_cast<float *>(st_smem + SL::kEinv);
  uint32_t *xchg = reinterpret_cast<uint32_t *>(st_smem + SL::kXchg);
  uint32_t *keys = reinterpret_cast<uint32_t *>(st_smem + SL::kKeys);
  int *heavy = reinterpret_cast<int *>(st_smem + SL::kHeavy);
  int *ev = reinterpret_cast<int *>(st_smem + SL::kEv);
  const uint32_t bar_t_full = smem_u32(&bars[0]), bar_drain = smem_u32(&bars[2]);
  const StSync sync;   // of the eight warps

  const int u = blockIdx.y, r = blockIdx.x, R = gridDim.x, b = u / p.H_kv, h = u % p.H_kv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Nobody writes to a CTA that has not started: waited for in front of the first such write, and of every return.  (What is written
  // is set up by nobody before, so the arrival orders no memory: as a release the launch took 0.8 us longer, 40 us.)
  if (kCluster) cluster_arrive_relaxed();
  if (tid == 0) prefetch_tensormap(&mapD);
  pdl_wait();
  pdl_trigger();
  // ---- the sets of Algorithm 1, selection step, exactly as the general selection defines them
  const int len = max(0, min(src.seq_len[b], p.N_cap));
  int budget = budget_dev ? budget_dev[b] : budget_scalar;
  budget = max(0, min(budget, p.N_cap));
  int n_sink = p.n_sink, n_recent = n_recent_dev ? max(0, n_recent_dev[b]) : p.n_recent;
  int lo, hi, n_heavy;
  if (budget >= len) {
    lo = hi = len;
    n_heavy = 0;
  } else {
    n_sink = min(n_sink, budget);
    n_recent = min(n_recent, budget - n_sink);
    lo = n_sink;
    hi = len - n_recent;
    n_heavy = budget - n_sink - n_recent;
  }
  const int m_cand = hi - lo, n_ret = min(len, budget), n_ev = len - n_ret;
  if (m_cand > kStCand || n_ev > kStEv || n_ret > kStRet) {
    if (r == 0 && tid == 0) atomicOr(status_dev, KEEPKV_DEV_NOT_STEADY);   // the promise does not hold here
    __syncwarp();
    if (kCluster) cluster_wait();
    return;
  }
  const size_t base = (size_t)u * p.N_cap;
  const uint8_t *kS = reinterpret_cast<const uint8_t *>(src.K) + base * (2 * D);
  const uint8_t *vS = reinterpret_cast<const uint8_t *>(src.V) + base * (2 * D);
  uint8_t *vD = reinterpret_cast<uint8_t *>(dst.V) + base * (2 * D);
  const uint32_t sbase = smem_u32(st_smem);
  // byte offset of 16-byte chunk c of row `row` inside a swizzled tile of `rows` rows
  auto swz = [](int rows, int row, int c) { return (c >> 3) * (rows * 128) + row * 128 + (((c & 7) ^ (row & 7)) << 4); };
  // source index of retained slot s: sinks, kept candidates (known once the selection is done), recent window
  auto ret = [&](int s) { return s < lo ? s : (s < lo + n_heavy ? heavy[s - lo] : hi + (s - lo - n_heavy)); };

  // ---- this CTA's slice of the retained slots, in 64-slot tiles
  constexpr int S = SL::kStages;
  const int n_tiles = (n_ret + kStN - 1) / kStN;
  const int t0 = (int)((long long)n_tiles * r / R), t1 = (int)((long long)n_tiles * (r + 1) / R);

  if (warp >= kStWarps) {
    const int s0 = t0 * kStN, s1 = min(t1 * kStN, n_ret), rec = min(s1, max(s0, lo + n_heavy));
    if (warp == kStWarps) {
      // ---- values: two blocks of rows, one on its way in while the other is on its way out
      const uint32_t bar_v = smem_u32(&bars[3]);
      constexpr uint32_t kRow = 2 * D;
      if (lane == 0) { mbar_init(bar_v, 1); mbar_init(bar_v + 8, 1); mbar_fence_init(); }
      __syncwarp();
      bool ok = true;
      int c = 0, asked = 0;   // blocks so far: of the ranges before this one, and whose rows have been asked for
      auto copy = [&](int from, int to, bool in_order) {
        const int n = max(0, to - from + kStRows - 1) / kStRows;
        auto load = [&](int k) {
          const int q = from + kStRows * k, rows = min(kStRows, to - q), at = (c + k) & 1;
          const uint32_t bar = bar_v + 8 * at, buf = sbase + SL::kVal + at * (kStRows * kRow);
          if (asked++ == withhold) return;   // (test hook: these rows are never asked for)
          if (lane == 0) {
            bulk_wait_read();   // the block before the last has left this half
            mbar_expect_tx(bar, rows * kRow);
            if (in_order) bulk_load_1d(buf, vS + (size_t)ret(q) * kRow, rows * kRow, bar);
          }
          __syncwarp();
          if (!in_order && lane < rows) bulk_load_1d(buf + lane * kRow, vS + (size_t)ret(q + lane) * kRow, kRow, bar);
          __syncwarp();
        };
        if (n > 0) load(0);
        for (int k = 0; ok && k < n; ++k) {
          if (k + 1 < n) load(k + 1);
          const int q = from + kStRows * k, at = (c + k) & 1;
          ok = __all_sync(0xffffffffu, mbar_wait_n(bar_v + 8 * at, ((c + k) >> 1) & 1, spin_limit));
          if (ok && lane == 0) {
            bulk_store_1d(vD + (size_t)q * kRow, sbase + SL::kVal + at * (kStRows * kRow), min(kStRows, to - q) * kRow);
            bulk_commit();
          }
          __syncwarp();
        }
        c += n;
      };
      copy(rec, s1, true);
      st_sync_all(2);   // the list of kept candidates is complete
      if (ok) copy(s0, rec, false);
      if (!ok)   // the CTA does not end before the rows it has asked for are here (bounded)
        for (int j = max(0, asked - 2); j < asked; ++j)
          if (j != withhold) mbar_wait_n(bar_v + 8 * (j & 1), (j >> 1) & 1, spin_limit);
      __syncwarp();
      if (lane == 0) {
        if (!ok) atomicOr(status_dev, KEEPKV_DEV_TIMEOUT);
        bulk_wait();
        fence_proxy_async_all();
      }
    } else {
      auto copy = [&](int from, int to) {
#pragma unroll 4
        for (int q = from + lane; q < to; q += 32) {
          const int i = ret(q);
          dst.votes[base + q] = src.votes[base + i];
          dst.lscore[base + q] = src.lscore[base + i];
          ret_idx[base + q] = i;
          target[base + i] = -2;
        }
      };
      copy(rec, s1);
      st_sync_all(2);
      copy(s0, rec);
    }
    __threadfence();
    st_arrive_all(3);   // these rows are in place
    __syncwarp();
    if (kCluster) cluster_wait();
    return;
  }

  if (tid == 0) {
    mbar_init(bar_t_full, 1);
    mbar_init(bar_t_full + 8, 1);
    mbar_init(bar_drain, 1);
    s_abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&s_tmem), kStTmemCols);
    tmem_relinquish();
  }
  const int crow = tid / CH, cch = tid % CH;   // the row (of every pass) and the 16-byte chunk this thread requests
  // The keys of tile t into their stage by cp.async, two tiles ahead of the product.  A commit per call, also for a tile
  // past the slice, keeps the group count uniform.
  auto issue_keys = [&](int t) {
    if (t < t1) {
      const uint32_t st = sbase + SL::kRing + ((t - t0) % S) * SL::kStageBytes;
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const int rw = j * RP + crow, s = t * kStN + rw;
        const bool ok = s < n_ret;
        cp_async_16(st + swz(kStN, rw, cch), kS + (ok ? (size_t)ret(s) * (2 * D) + cch * 16 : 0), ok);
      }
    }
    cp_async_commit();
  };
  // A slice that starts in the recent window does not depend on the selection: its first tiles are requested now.
  const bool early = t0 * kStN >= lo + n_heavy;
  if (early) { issue_keys(t0); issue_keys(t0 + 1); }

  // ---- selection (Algorithm 1, selection step)
  uint32_t k_lo = 0xffffffffu, k_hi = 0u;
  for (int i = tid; i < m_cand; i += kStThreads) {   // the caller's scores where given, else kappa = ln p + lscore
    const uint32_t k = select_key ? ordered_key(select_key[base + lo + i])
                                  : kappa_key(src.votes[base + lo + i], src.lscore[base + lo + i]);
    keys[i] = k;
    k_lo = min(k_lo, k);
    k_hi = max(k_hi, k);
  }
  __syncwarp();
  k_lo = __reduce_min_sync(0xffffffffu, k_lo);
  k_hi = __reduce_max_sync(0xffffffffu, k_hi);
  if (lane == 0) { s_kmin[warp] = k_lo; s_kmax[warp] = k_hi; }
  tc_fence_before();
  sync();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  uint32_t kth = 0u;
  int n_tie = 0, tot_ties = 0;
  if (n_heavy > 0) {
#pragma unroll
    for (int w = 0; w < kStWarps; ++w) { k_lo = min(k_lo, s_kmin[w]); k_hi = max(k_hi, s_kmax[w]); }
    range_select(keys, 0, m_cand, k_lo, k_hi, n_heavy, kStThreads, reinterpret_cast<int *>(st_smem + SL::kHist), s_sel, warp_tot,
                 kth, n_tie, tot_ties, sync);
  }
  {
    // one ordered pass over the candidates: a thread owns 8 consecutive ones (kStCand = 8 * kStThreads)
    static_assert(kStCand == 8 * kStThreads, "one sweep covers all candidates");
    const bool rank_ties = n_heavy > 0 && n_tie < tot_ties;
    const int i0 = tid * 8;
    bool keepf[8], tief[8];
    int n_t = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + j;
      const bool valid = i < m_cand && n_heavy > 0;
      const uint32_t k = valid ? keys[i] : 0u;
      tief[j] = valid && k == kth;
      keepf[j] = valid && k > kth;
      n_t += tief[j] ? 1 : 0;
    }
    if (n_heavy > 0) {
      int tie_rank = 0, tot_tie = 0;
      if (rank_ties) tie_rank = block_excl_sum(n_t, warp_tot, tot_tie, kStWarps, sync);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (tief[j]) { keepf[j] = !rank_ties || tie_rank < n_tie; ++tie_rank; }
    }
    int n_k = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) n_k += keepf[j] ? 1 : 0;
    int tot_keep;
    int slot = block_excl_sum(n_k, warp_tot, tot_keep, kStWarps, sync);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + j;
      if (i < m_cand) {
        if (keepf[j]) heavy[slot++] = lo + i;
        else ev[i - slot] = lo + i;
      }
    }
  }
  sync();   // the lists are complete; nobody reads the selection keys any more
  st_arrive_all(2);

  const int quarter = warp & 3, half = warp >> 2;   // drain: 32 lanes of tensor memory, 32 of a tile's 64 columns
  const int row = quarter * 32 + lane;              // the evicted entry this thread tracks
  const bool live = quarter * 32 < n_ev;            // the warp's rows exist
  Top2 top, topb;   // two lists over alternate columns: two independent dependency chains
  top.init(0.f);
  topb.init(0.f);
  {
    // ---- A operand: the evicted keys
#pragma unroll
    for (int j = 0; j < kStEv / RP; ++j) {
      const int rw = j * RP + crow;
      const bool ok = rw < n_ev;
      cp_async_16(sbase + SL::kA + swz(kStEv, rw, cch), kS + (ok ? (size_t)ev[rw] * (2 * D) + cch * 16 : 0), ok);
    }
    cp_async_commit();
    if (early) {
      cp_async_wait<0>();
    } else {
      issue_keys(t0);
      issue_keys(t0 + 1);
      cp_async_wait<1>();
    }
    sync();   // the evicted keys and the first tile have landed
    // Inverse norms of the keys of tile t, four threads a row.  (The two rows of eight lanes start in different halves of
    // 128 bytes.)  Rows past the slice: 1/0 = inf, their products 0 * inf never rank.
    auto tile_norms = [&](int t) {
      const uint8_t *st = st_smem + SL::kRing + ((t - t0) % S) * SL::kStageBytes;
      const int rw = tid >> 2, q = tid & 3;
      float a = 0.f, c = 0.f;
#pragma unroll
      for (int k = 0; k < CH / 4; ++k) {
        const uint4 v = *reinterpret_cast<const uint4 *>(st + swz(kStN, rw, (k ^ (rw & 1)) * 4 + q));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) { a = fmaf(bf16_lo(w[j]), bf16_lo(w[j]), a); c = fmaf(bf16_hi(w[j]), bf16_hi(w[j]), c); }
      }
      a += c;
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      a += __shfl_xor_sync(0xffffffffu, a, 2);
      if (q == 0) cinv[((t - t0) & 3) * kStN + rw] = rsqrtf(a);
    };
    if (tid < kStEv) {   // of the evicted keys, a row per thread
      float a = 0.f, c = 0.f;
#pragma unroll
      for (int k = 0; k < CH; ++k) {
        const uint4 v = *reinterpret_cast<const uint4 *>(st_smem + SL::kA + swz(kStEv, tid, k));
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) { a = fmaf(bf16_lo(w[q]), bf16_lo(w[q]), a); c = fmaf(bf16_hi(w[q]), bf16_hi(w[q]), c); }
      }
      einv[tid] = rsqrtf(a + c);
    }
    __syncwarp();
    if (t0 < t1) tile_norms(t0);
    // Drains the accumulator of tile i (relative to t0): 32 columns of this thread's row.
    auto drain = [&](int i) {
      tc_fence_after();
      uint32_t acc[32];
      tmem_ld_32x32(tmem + ((uint32_t)(quarter * 32) << 16) + (i & 1) * kStN + half * 32, acc);
      tmem_ld_wait();
      const float *ci = cinv + (i & 3) * kStN + half * 32;
      const int c0 = (t0 + i) * kStN + half * 32;
#pragma unroll
      for (int k = 0; k < 32; k += 4)
        offer4(top, topb, __uint_as_float(acc[k]), __uint_as_float(acc[k + 1]), __uint_as_float(acc[k + 2]),
               __uint_as_float(acc[k + 3]), *reinterpret_cast<const float4 *>(ci + k), c0 + k);
    };
    // Waits (bounded) until the product of tile i has completed.
    auto wait_product = [&](int i) {
      const int ok = __all_sync(0xffffffffu, !s_abort && mbar_wait(bar_t_full + 8 * (i & 1), (i >> 1) & 1));
      if (!ok) s_abort = 1;
      return ok != 0;
    };
    for (int t = t0; t < t1; ++t) {
      const int i = t - t0;
      cp_async_wait<0>();          // the keys of tiles <= t + 1 have landed (this thread's copies)
      fence_proxy_async_smem();    // ... and are visible to the tensor core and to the stores, like the A tile
      tc_fence_before();
      if (tid == 0) bulk_wait_read();   // tile t - 1 has left its stage
      __syncwarp();
      sync();                      // everyone's; and everyone has finished the previous iteration
      tc_fence_after();
      if (i == 0) {
        // Values are compared before the division by |k_e|: the closeness margin and the threshold scale with it.  A row
        // that does not exist, or of norm zero, takes no column.
        const float ri = einv[row];
        top.init(2.f * kRankEps / ri);
        topb.init(top.thr);
        top.cut = row < n_ev && ri < CUDART_INF_F ? (p.merge_threshold - 2.f * kRankEps) / ri : CUDART_INF_F;
      }
      const uint32_t at = sbase + SL::kRing + (i % S) * SL::kStageBytes;
      if (warp == 0 && !__any_sync(0xffffffffu, s_abort) && elect_one()) {
        const uint64_t ad = umma_desc_sw128(sbase + SL::kA), bd = umma_desc_sw128(at);
#pragma unroll
        for (int k = 0; k < KSTEPS; ++k)   // (descriptor addresses count 16-byte units)
          umma_bf16(tmem + (i & 1) * kStN, ad + (k >> 2) * (kStEv * 8) + (k & 3) * 2, bd + (k >> 2) * (kStN * 8) + (k & 3) * 2,
                    IDESC, k > 0 ? 1u : 0u);
        umma_commit(bar_t_full + 8 * (i & 1));
      }
      __syncwarp();
      if (tid == 0) {   // the copy (Algorithm 1, insertion step): rows past the slice land behind the unit's new length
#pragma unroll
        for (int sub = 0; sub < SL::kSub; ++sub) tma_store_2d(&mapD, sub * 64, (int)base + t * kStN, at + sub * (kStN * 128));
        bulk_commit();
      }
      __syncwarp();
      // the previous product has completed: its stage can be refilled and its accumulator drained
      const bool prev = i > 0 && wait_product(i - 1);
      issue_keys(t + 2);   // into the stage of tile t - 1
      if (t + 1 < t1) tile_norms(t + 1);
      if (prev && live) drain(i - 1);
    }
    cp_async_wait<0>();
    if (t0 < t1 && wait_product(t1 - t0 - 1) && live) drain(t1 - t0 - 1);
  }
  if (tid == 0) {   // the keys of the slice are in dst: the last CTA's merges come after them
    bulk_wait();
    fence_proxy_async_all();
  }
  // ---- tensor memory is no longer needed
  st_sync_all(3);   // (and the copying warps' rows are in place)
  if (warp == 0 && __any_sync(0xffffffffu, s_abort)) {
    if (lane == 0) atomicOr(status_dev, KEEPKV_DEV_TIMEOUT);
    if (elect_one()) umma_commit(bar_drain);   // (a commit covers the products of its own thread: the elected one's)
    mbar_wait(bar_drain, 0);   // products still in flight get a bounded chance to retire
  }
  tc_fence_before();
  sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kStTmemCols);
  }
  // ---- per evicted row: the two lists and the two column halves folded (equal values -> lower slot),
  // scaled by the row's own inverse norm
  top.insert_any(topb.best, topb.bi);
  top.insert_any(topb.second, topb.si);
  if (half == 1) {
    xchg[row * 4] = __float_as_uint(top.best); xchg[row * 4 + 1] = (uint32_t)top.bi;
    xchg[row * 4 + 2] = __float_as_uint(top.second); xchg[row * 4 + 3] = (uint32_t)top.si;
  }
  sync();
  const int tr = kCluster ? r : 0, tR = kCluster ? R : 1;   // of the CTAs that go on
  const int per = (kStEv + tR - 1) / tR;           // CTA tr settles rows tr, tr + tR, ..: thread i the i-th of them
  const int j = tr + tid * tR;
  const bool valid = tid < per && j < n_ev;
  Top2 mine;
  mine.init(0.f);
  if (tid < n_ev) {                // threads 0..127 are the first column half of rows 0..127
    mine = top;
    mine.insert_any(__uint_as_float(xchg[row * 4]), (int)xchg[row * 4 + 1]);
    mine.insert_any(__uint_as_float(xchg[row * 4 + 2]), (int)xchg[row * 4 + 3]);
    mine.best *= einv[row];
    mine.second *= einv[row];
  }
  auto fold = [&](const uint4 v) {   // slices hold ascending slots: strict comparisons keep the lower slot on ties
    mine.insert(__uint_as_float(v.x), (int)v.z);
    mine.insert(__uint_as_float(v.y), (int)v.w);
  };
  if (kCluster) {
    __syncwarp();
    cluster_wait();                // every CTA of the unit has started
    if (tid < n_ev)
      st_shared_cluster_v4(mapa_shared(sbase + SL::kInbox + (r * per + tid / R) * 16, (uint32_t)(tid % R)), __float_as_uint(mine.best),
                           __float_as_uint(mine.second), (uint32_t)mine.bi, (uint32_t)mine.si);
    if (r == 0 && tid == 0) stats[u] = keepkv_stats{};   // (before any CTA of the unit adds to it)
    __threadfence();
    __syncwarp();
    cluster_sync_all();            // every CTA's candidates are here, and its rows in place
    mine.init(0.f);
    if (valid)
      for (int c = 0; c < R; ++c) fold(*reinterpret_cast<const uint4 *>(st_smem + SL::kInbox + (c * per + tid) * 16));
  } else if (R > 1) {
    if (valid)
      nom[(base + tid) * C_max + r] =
          make_uint4(__float_as_uint(mine.best), __float_as_uint(mine.second), (uint32_t)mine.bi, (uint32_t)mine.si);
    __threadfence();
    sync();
    if (tid == 0) {
      s_last = atomicAdd(&counters[u], 1) == R - 1;
      if (s_last) counters[u] = 0;   // ready for the next call
    }
    sync();
    if (!s_last) return;
    __threadfence();
    mine.init(0.f);
    if (valid)
      for (int c = 0; c < R; ++c) fold(__ldcg(&nom[(base + tid) * C_max + c]));
  }

  // ---- Algorithm 1, arg-max and threshold step: arg-max and threshold; the interface's exact arithmetic where the ranking is too close to call
  float *ke_s = reinterpret_cast<float *>(st_smem + SL::kKe), *kc_s = reinterpret_cast<float *>(st_smem + SL::kKc);
  int *qs = reinterpret_cast<int *>(st_smem + SL::kQ);
  int *q_tid = qs, *q_e = qs + kStEv, *q_kind = qs + 2 * kStEv, *q_a = qs + 3 * kStEv, *q_b = qs + 4 * kStEv,
      *res_slot = qs + 5 * kStEv, *res_merge = qs + 6 * kStEv;
  uint32_t *skey = reinterpret_cast<uint32_t *>(st_smem + SL::kSkey);
  int *ghead = reinterpret_cast<int *>(st_smem + SL::kGhead);
  const __nv_bfloat16 *sK = reinterpret_cast<const __nv_bfloat16 *>(src.K) + base * D;
  const float T = p.merge_threshold;
  int e = 0, slot = -1, kind = 0;
  bool merge = false;
  if (valid) {
    e = ev[j];
    if (mine.bi >= 0) {
      slot = mine.bi;
      if (!(mine.best - mine.second > kRankEps)) kind = mine.si >= 0 ? 1 : 2;
      else if (!(fabsf(mine.best - T) > kRankEps)) kind = 2;
      else merge = mine.best > T;
    }
  }
  if (tid == 0) s_nq = 0;
  sync();   // every warp has left the similarity product: the key rows' memory is free
  if (kind) {
    const int qi = atomicAdd(&s_nq, 1);
    q_tid[qi] = tid; q_e[qi] = e; q_kind[qi] = kind; q_a[qi] = mine.bi; q_b[qi] = mine.si;
  }
  sync();
  for (int qi = warp; qi < s_nq; qi += kStWarps) {
    const int ee = q_e[qi], kd = q_kind[qi], ca = q_a[qi], cb = kd == 1 ? q_b[qi] : q_a[qi];
    float u0, u1;
    exact_cosines<D>(sK + (size_t)ee * D, sK + (size_t)ret(ca) * D, sK + (size_t)ret(cb) * D, ke_s + warp * D,
                     kc_s + warp * 2 * D, u0, u1);
    int win = ca;
    float wu = u0;
    if (kd == 1 && (u1 > u0 || (u1 == u0 && cb < ca))) { win = cb; wu = u1; }
    if (lane == 0) { res_slot[q_tid[qi]] = win; res_merge[q_tid[qi]] = wu > T; }
  }
  sync();
  if (kind) { slot = res_slot[tid]; merge = res_merge[tid] != 0; }

  // ---- the decisions, to every CTA of the unit
  int *dec = reinterpret_cast<int *>(st_smem + SL::kDec);
  if (valid) {
    const int to = merge ? slot : -1;
    target[base + e] = to;
    if (!kCluster) dec[j] = to;
    else
      for (int c = 0; c < R; ++c) st_shared_cluster_u32(mapa_shared(sbase + SL::kDec + j * 4, (uint32_t)c), (uint32_t)to);
  }
  __syncwarp();
  if (!kCluster) sync();
  else cluster_sync_all();         // (behind it no CTA touches another's shared memory)

  // ---- groups: the entries to merge sorted by (slot, position); every CTA makes the same list
  const int to = tid < n_ev ? dec[tid] : -1;
  int M;
  const int off = block_excl_count(to >= 0, warp_tot, M, kStWarps, sync);
  if (to >= 0) skey[off] = ((uint32_t)to << 16) | (uint32_t)tid;
  sync();
  uint32_t mk = 0xFFFFFFFFu;
  int rank = 0;
  if (tid < M) {
    mk = skey[tid];
    for (int j = 0; j < M; ++j) rank += skey[j] < mk ? 1 : 0;
  }
  sync();
  if (tid < M) skey[rank] = mk;
  sync();
  const bool head = tid < M && (tid == 0 || (skey[tid] >> 16) != (skey[tid - 1] >> 16));
  int n_groups;
  const int pos = block_excl_count(head, warp_tot, n_groups, kStWarps, sync);
  if (head) ghead[pos] = tid;
  if (tid == 0) {
    ghead[n_groups] = M;
    if (tr == 0) {
      if (!kCluster) stats[u] = keepkv_stats{};
      stats[u].n_retained = n_ret;
      stats[u].n_evicted = n_ev;
      stats[u].n_below_T = n_ev - M;
      if (h == 0) dst.seq_len[b] = n_ret;
    }
  }
  sync();
  // ---- Algorithm 1, merge step: one warp per group, of all the unit's CTAs
  MergeCount count;
  for (int gi = tr * kStWarps + warp; gi < n_groups; gi += tR * kStWarps) {
    const int beg = ghead[gi], n = ghead[gi + 1] - beg;
    const int c = (int)(skey[beg] >> 16);
    merge_group<D>(p, src, dst, c, src, base + ret(c), [&](int t) { return ev[skey[beg + t] & 0xFFFFu]; }, n, target + base, base,
                   count);
  }
  count.flush(stats + u);
}

template <int D>
static void launch_steady_t(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                            const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                            int32_t *ret_idx, int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L,
                            int32_t *status_dev, const float *select_key, LaunchCtx &ctx) {
  using SL = StSmem<D>;
  const int U = p.B * p.H_kv;
  constexpr size_t smem_bytes = (size_t)SL::kBytes + 1024;   // slack to align the swizzled tiles
  static_assert(smem_bytes <= kStOneCtaSmem && 2 * (smem_bytes + 2048) <= 228 * 1024, "two CTAs per SM");
  static bool attr_done_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_done_dev[dev & 63]) {
    cudaFuncSetAttribute(steady_compress_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStOneCtaSmem);
    cudaFuncSetAttribute(steady_compress_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    attr_done_dev[dev & 63] = true;
  }
  CUtensorMap mapD;
  if (!make_bf16_rows_map(&mapD, dst.K, (uint64_t)p.B * p.H_kv * p.N_cap, D, kStN)) {
    if (ctx.err == cudaSuccess) ctx.err = cudaErrorInvalidValue;
    return;
  }
  // CTAs per unit: what two resident CTAs per SM can hold at once.  They are a cluster where all units' clusters are resident
  // (one lives inside a GPC: 66 of four, 90 of three), also with fewer CTAs, unless more than a quarter of them would be given up:
  // a launch for 72 units takes 43 us as clusters of three, 45 as four CTAs; one for 96 takes 60 as clusters of two, 53 as three.
  int R = 2 * sm_count() / U;
  R = R < 1 ? 1 : (R > L.nom_chunks ? L.nom_chunks : R);
  int k = R;
  while (k > 1 && resident_clusters<steady_compress_kernel<D, true>>(dev, k, kStAll, kStOneCtaSmem) < U) --k;
  uint4 *nom = reinterpret_cast<uint4 *>(ws + L.nom);
  int *counters = reinterpret_cast<int *>(ws + L.counters);
  if (k > 1 && 4 * k >= 3 * R)
    launch_pdl_cluster(steady_compress_kernel<D, true>, dim3(k, U), dim3(kStAll), smem_bytes, ctx.stream, (unsigned)k, mapD, p, src, dst,
                       budget_dev, budget_scalar, n_recent_dev, ret_idx, target, nom, L.nom_chunks, counters, stats, status_dev,
                       select_key, debug_spin_limit(), debug_withhold());
  else
    launch_pdl(steady_compress_kernel<D, false>, dim3(R, U), dim3(kStAll), smem_bytes, ctx.stream, mapD, p, src, dst, budget_dev,
               budget_scalar, n_recent_dev, ret_idx, target, nom, L.nom_chunks, counters, stats, status_dev, select_key,
               debug_spin_limit(), debug_withhold());
  KEEPKV_CHECK_LAUNCH(ctx);
}

void launch_compress_steady(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                            const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                            int32_t *ret_idx, int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L,
                            int32_t *status_dev, const float *select_key, LaunchCtx &ctx) {
  if (p.d == 128)
    launch_steady_t<128>(p, src, dst, budget_dev, budget_scalar, n_recent_dev, ret_idx, target, stats, ws, L, status_dev,
                         select_key, ctx);
  else
    launch_steady_t<64>(p, src, dst, budget_dev, budget_scalar, n_recent_dev, ret_idx, target, stats, ws, L, status_dev,
                        select_key, ctx);
}

}  // namespace keepkv
