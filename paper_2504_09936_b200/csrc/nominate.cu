// Similarity search of keepkv_compress (Algorithm 1, similarity step: U = cosineSimilarity(K_e, K_c)) on the
// 5th-generation tensor cores.  The cosine matrix is never stored: for every evicted key the kernel
// keeps the two largest cosines over the retained keys and their slots, which is all the arg-max
// of Algorithm 1 needs.  The values found here only *rank* candidates; wherever the
// ranking is closer than the accumulation error allows, the caller re-evaluates the candidates in
// the fixed fp32 arithmetic the interface defines (see resolve_kernel in compress.cu).
//
// Only columns whose cosine exceeds the merge threshold matter: an entry whose best cosine does not exceed it is dropped
// whatever its best column was.  So the product itself subtracts the threshold: eight more channels -- the row's cut
// (threshold less a margin, times the row's norm) and the column's norm, both as three bf16 terms, six cross products --
// make the accumulator  k_e . k_c - cut_e |k_c|,  and 32 columns are screened by 20 maxima and one vote.  What passes (a
// fifth of the 32 x 32 blocks at a threshold of 0.8 on keys with outlier channels) is looked at four columns at a time.
// For a threshold below kNomStatic, where nearly every block would pass, those channels are zero and the screen is the
// running cut itself: one packed multiply-add per two columns.
//
// Work item = (unit, 128 evicted rows, one chunk of 256-column tiles of the unit's retained keys).
// A persistent grid of one CTA per SM walks the items.  Inside a CTA:
//   warp 0      copies: column tiles (256 rows x D, 128-byte swizzle, and their norms), 64 channels at a time into a
//               4-stage ring, so that three quarters of it are in flight while one is multiplied;
//   warp 1      tensor cores: M = 128, N = 256, bf16 -> fp32, into one of two accumulators in tensor memory;
//   warps 2-3   gather the evicted rows of the next item from the src cache into the other A tile;
//   warps 4-19  drain: four warps per 32 rows, 64 of a tile's 256 columns each.
// Bound: the tensor pipe at the rate it sustains (with its extra sixteenth of the channels) and, beside it, the hand-overs.
// Measured, 64 units of 6554 x 1638 keys of 128 channels, 176 GFLOP: 525 us when every accumulator was scaled by its
// column's norm and tested against a cut that starts at minus infinity (1.46 instructions per row and column of a warp),
// 378 us with the scaled values screened 32 at a time against a cut that starts at the threshold (0.85), 205 us in this
// form; without the drain it is 177 us.  256 rows an item, as two products of N = 128 a column tile, measured equal.
// Every wait is bounded; a wait that runs out raises KEEPKV_DEV_TIMEOUT, every warp of the CTA leaves its loop, what is
// in flight gets a bounded time to end, tensor memory is freed.
#include "compress.cuh"
#include "ptx.cuh"

namespace keepkv {

constexpr int kNomM = 128;         // evicted rows per item (tensor-memory lanes)
constexpr int kNomN = 256;         // retained columns per tile
constexpr int kNomStages = 4;      // column ring: 64 channels of a tile each
constexpr int kNomDrainWarps = 16;
constexpr int kNomGatherWarps = 2; // (20 warps in all: 96 registers a thread)
constexpr int kNomThreads = 32 * (2 + kNomGatherWarps + kNomDrainWarps);
constexpr float kNomStatic = 0.5f; // thresholds from here on are subtracted by the product
constexpr int kNomPairCap = 4096;  // capacity and retained keys from which on pairs of CTAs search
constexpr int kNomPairColumns = 800;

template <int D>
struct NomSmem {
  static constexpr int kSub = D / 64;                     // 64-channel (128-byte) K atoms per row
  static constexpr int kABytes = kSub * kNomM * 128;
  static constexpr int kBBytes = kNomN * 128;
  static constexpr int kTiles = kNomStages / kSub;        // column tiles the ring holds
  static constexpr int kA = 0;                            // [2]: the next item is gathered while this one runs
  static constexpr int kB = 2 * kABytes;
  static constexpr int kAX = kB + kNomStages * kBBytes;   // [2][128] x 16 B  eight more channels of the rows
  static constexpr int kBX = kAX + 2 * kNomM * 16;        // [kTiles][256] x 16 B  and of the columns
  static constexpr int kZero = kBX + kTiles * kNomN * 16; // [256] x 16 B  and eight more that are zero, for all of them
  // Inverse norms of the columns outlive their tile's stages: when tile t + 2 has been multiplied, tile t has been drained.
  static constexpr int kInvTiles = kTiles + 2 <= 4 ? 4 : 8;
  static constexpr int kInv = kZero + kNomN * 16;              // f32 [kInvTiles][256]
  static constexpr int kRowInv = kInv + kInvTiles * kNomN * 4; // f32 [2][128]        inverse norms of the staged rows
  static constexpr int kXchg = kRowInv + 2 * kNomM * 4;        // u32 [2][128][3][3]  results of the later column quarters
  static constexpr int kCoarse = kXchg + 2 * kNomM * 36;       // i32 [kMaxUnits / 32]  row tiles before each 32 units
  static constexpr int kBytes = kCoarse + kMaxUnits / 32 * 4;
};

// Four columns idx..idx+3: accumulators a_i, inverse norms w_i.  Skipped by the whole warp unless a row has one at its cut.
// (What is left of a missing column's inverse norm may have any sign: -inf stays -inf.)
__device__ __forceinline__ void offer4_above(Top2 &ta, Top2 &tb, float a0, float a1, float a2, float a3, const float4 w,
                                             int idx) {
  const float v0 = a0 * fabsf(w.x), v1 = a1 * fabsf(w.y), v2 = a2 * fabsf(w.z), v3 = a3 * fabsf(w.w);
  if (!__any_sync(0xffffffffu, max3(fmaxf(v0, v1), v2, v3) >= ta.cut)) return;
  ta.insert(v0, idx); tb.insert(v1, idx + 1); ta.insert(v2, idx + 2); tb.insert(v3, idx + 3);
  ta.cut = fmaxf(ta.cut, fmaxf(ta.best, tb.best) - ta.thr);   // (it only rises: it may have started above the best)
}

struct __align__(16) NomItem { int u, m0, chunk, t0, t1, n_ev, n_ret, pad; };

// The whole warp looks an item up: among the units' row tiles first by groups of 32 units, then inside the group.
__device__ __forceinline__ NomItem nom_item(int item, int C, const int *coarse, int U, const UnitInfo *unit_info) {
  const int lane = threadIdx.x & 31, groups = (U + 31) >> 5;
  NomItem it;
  const int mg = item / C;
  it.chunk = item % C;
  int g = -1;   // last group that starts at or before mg
  for (int k = 0; k < groups; k += 32) {
    const bool le = k + lane < groups && coarse[k + lane] <= mg;
    g += __popc(__ballot_sync(0xffffffffu, le));
  }
  const int u = g * 32 + lane;
  int n_ev = 0, n_ret = 0;
  if (u < U) { const UnitInfo ui = unit_info[u]; n_ev = ui.n_ev; n_ret = ui.n_ret; }
  const int tiles = (n_ev + kNomM - 1) / kNomM;
  int x = tiles;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const int r = mg - coarse[g];
  const int at = __ffs(__ballot_sync(0xffffffffu, x > r)) - 1;   // (mg lies in this group, so one lane's sum exceeds r)
  it.u = g * 32 + at;
  it.m0 = (r - __shfl_sync(0xffffffffu, x - tiles, at)) * kNomM;
  it.n_ev = __shfl_sync(0xffffffffu, n_ev, at);
  it.n_ret = __shfl_sync(0xffffffffu, n_ret, at);
  const int T = (it.n_ret + kNomN - 1) / kNomN;
  it.t0 = it.chunk * T / C;
  it.t1 = (it.chunk + 1) * T / C;
  it.pad = 0;
  return it;
}

// kCut: the product subtracts the rows' cuts (a compile-time choice: the other screen spills 44 bytes of registers, and both in
// one kernel more).
template <int D, bool kCut>
__global__ void __launch_bounds__(kNomThreads, 1)
nominate_kernel(const __grid_constant__ CUtensorMap mapB, keepkv_params p, const __nv_bfloat16 *__restrict__ srcK,
                const int32_t *__restrict__ ev_idx, const UnitInfo *__restrict__ unit_info,
                const float *__restrict__ inv_norm, const uint4 *__restrict__ norm_ext, int32_t *sched,
                uint4 *__restrict__ nom, int C_max, int32_t *status_dev, int self_mask,
                int spin_limit, int withhold) {
  using SL = NomSmem<D>;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // a_ready[2], a_empty[2], b_full[4], b_empty[4], t_full[2], t_empty[2], drain, x_full[4][2]
  __shared__ __align__(8) uint64_t bars[4 + 2 * kNomStages + 4 + 1 + 8];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(16) NomItem s_item[2];   // what the staged rows belong to; n_ev < 0: the CTA's items are done
  __shared__ int s_wtot[kNomThreads / 32], s_wmax[kNomThreads / 32];
  __shared__ volatile int s_abort;

  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar_a_ready = smem_u32(&bars[0]), bar_a_empty = smem_u32(&bars[2]);
  const uint32_t bar_b_full = smem_u32(&bars[4]), bar_b_empty = smem_u32(&bars[8]);
  const uint32_t bar_t_full = smem_u32(&bars[12]), bar_t_empty = smem_u32(&bars[14]);
  const uint32_t bar_drain = smem_u32(&bars[16]), bar_x = smem_u32(&bars[17]);
  int *coarse = reinterpret_cast<int *>(smem + SL::kCoarse);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int U = p.B * p.H_kv;
  const size_t n_rows = (size_t)U * p.N_cap;

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_a_ready + 8 * i, kNomGatherWarps);
      mbar_init(bar_a_empty + 8 * i, 1 + kNomDrainWarps);
      mbar_init(bar_t_full + 8 * i, 1);
      mbar_init(bar_t_empty + 8 * i, kNomDrainWarps);
    }
    for (int i = 0; i < kNomStages; ++i) { mbar_init(bar_b_full + 8 * i, 1); mbar_init(bar_b_empty + 8 * i, 1); }
    for (int i = 0; i < 8; ++i) mbar_init(bar_x + 8 * i, 3);
    mbar_init(bar_drain, 1);
    s_abort = 0;
    mbar_fence_init();
    fence_proxy_async_smem();
    prefetch_tensormap(&mapB);
  }
  if (tid >= 64 && tid < 64 + kNomN) {
    reinterpret_cast<uint4 *>(smem + SL::kZero)[tid - 64] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  pdl_wait();      // barrier set-up overlaps the previous kernel's tail
  pdl_trigger();
  if (warp == 1) {   // (not before the wait: see tmem_alloc)
    tmem_alloc(smem_u32(&s_tmem), 512);
    tmem_relinquish();
  }
  int total_m = 0, t_max = 0;
  {   // exclusive prefix of 128-row tiles over the units, kept for every 32nd: one unit per thread and pass
    for (int u0 = 0; u0 < U; u0 += kNomThreads) {
      const int u = u0 + tid;
      int t = 0, cols = 0;
      if (u < U) { const UnitInfo ui = unit_info[u]; t = (ui.n_ev + kNomM - 1) / kNomM; cols = ui.n_ret; }
      const int sum = __reduce_add_sync(0xffffffffu, t), mx = __reduce_max_sync(0xffffffffu, cols);
      if (lane == 0) { s_wtot[warp] = sum; s_wmax[warp] = mx; }
      __syncthreads();
      int off = 0, tot = 0;
#pragma unroll
      for (int w = 0; w < kNomThreads / 32; ++w) {
        const int v = s_wtot[w];
        off += w < warp ? v : 0;
        tot += v;
        t_max = max(t_max, s_wmax[w]);
      }
      if (lane == 0 && u < U) coarse[u >> 5] = total_m + off;
      total_m += tot;
      __syncthreads();
    }
    t_max = (t_max + kNomN - 1) / kNomN;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  const uint32_t tmem = s_tmem;
  // Column chunks per row tile: what makes the longest CTA shortest, an item costing about a tile and a half beside its
  // tiles (first columns, publishing).  Without chunks 192 items on 148 CTAs take as long as 296.
  int C = 1;
  {
    int cost = 0x7fffffff;
    for (int c = 1; c <= C_max; ++c) {
      const int rounds = (total_m * c + (int)gridDim.x - 1) / (int)gridDim.x, k = rounds * (2 * ((t_max + c - 1) / c) + 3);
      if (k < cost) { cost = k; C = c; }
    }
  }
  const int n_items = total_m * C;
  if (blockIdx.x == 0 && tid == 0) sched[0] = C;

  if (warp == 0) {
    // ------------------------------------------------------------ column tiles
    int ring = 0, n_tiles = 0;
    bool ok = true;
    for (int n_done = 0; ok; ++n_done) {   // (watches the rows' barrier only: an item's last product waits for its columns)
      if (!__all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_a_ready + 8 * (n_done & 1), (n_done >> 1) & 1, spin_limit))) { s_abort = 1; break; }
      const NomItem it = s_item[n_done & 1];
      if (it.n_ev < 0) break;
      for (int t = it.t0; ok && t < it.t1; ++t, ++n_tiles) {
        const int row = it.u * p.N_cap + t * kNomN;
#pragma unroll
        for (int sub = 0; sub < SL::kSub; ++sub, ++ring) {
          const int s = ring % kNomStages;
          ok = __all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_b_empty + 8 * s, ((ring / kNomStages) & 1) ^ 1, spin_limit));
          if (!ok) { s_abort = 1; break; }
          if (n_tiles != withhold && elect_one()) {   // (test hook: this tile is never asked for)
            const uint32_t full = bar_b_full + 8 * s;
            const bool last = sub == SL::kSub - 1;
            mbar_expect_tx(full, SL::kBBytes + (last ? kNomN * 20 : 0));
            tma_load_2d(sbase + SL::kB + s * SL::kBBytes, &mapB, sub * 64, row, full);
            if (last) {
              bulk_load_1d(sbase + SL::kBX + n_tiles % SL::kTiles * (kNomN * 16), norm_ext + row, kNomN * 16, full);
              bulk_load_1d(sbase + SL::kInv + n_tiles % SL::kInvTiles * (kNomN * 4), inv_norm + row, kNomN * 4, full);
            }
          }
          __syncwarp();
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ products
    int ring = 0, acc = 0;
    bool ok = true;
    for (int n_done = 0; ok; ++n_done) {
      const int buf = n_done & 1;
      ok = __all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_a_ready + 8 * buf, (n_done >> 1) & 1, spin_limit));
      if (!ok) break;
      const NomItem it = s_item[buf];
      if (it.n_ev < 0) break;
      for (int t = it.t0; ok && t < it.t1; ++t, ++acc) {
        const int a = acc & 1;
        // a unit's last tile is multiplied as far as it has columns, in sixteens
        const uint32_t idesc = umma_idesc_bf16(kNomM, min(kNomN, (it.n_ret - t * kNomN + 15) & ~15));
        ok = __all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_t_empty + 8 * a, ((acc >> 1) & 1) ^ 1, spin_limit));
#pragma unroll
        for (int sub = 0; sub < SL::kSub; ++sub, ++ring) {
          const int s = ring % kNomStages;
          ok = ok && __all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_b_full + 8 * s, (ring / kNomStages) & 1, spin_limit));
          if (!ok) break;
          tc_fence_after();
          if (elect_one()) {
            const uint64_t ad = umma_desc_sw128(sbase + SL::kA + buf * SL::kABytes + sub * (kNomM * 128));
            const uint64_t bd = umma_desc_sw128(sbase + SL::kB + s * SL::kBBytes);
            const uint32_t dt = tmem + a * kNomN;
#pragma unroll
            for (int k = 0; k < 4; ++k)   // (descriptor addresses count 16-byte units)
              umma_bf16(dt, ad + k * 2, bd + k * 2, idesc, sub + k > 0 ? 1u : 0u);
            if (sub == SL::kSub - 1) {
              const uint32_t zero = sbase + SL::kZero;
              if (kCut)
                umma_bf16(dt, umma_desc_plain(sbase + SL::kAX + buf * (kNomM * 16), zero),
                          umma_desc_plain(sbase + SL::kBX + acc % SL::kTiles * (kNomN * 16), zero), idesc, 1u);
              umma_commit(bar_t_full + 8 * a);
            }
            umma_commit(bar_b_empty + 8 * s);   // the stage may be refilled once these have read it
          }
          __syncwarp();
        }
      }
      if (elect_one()) umma_commit(bar_a_empty + 8 * buf);          // the rows have been read
      __syncwarp();
    }
    if (!ok) s_abort = 1;
    if (elect_one()) umma_commit(bar_drain);
    mbar_wait_n(bar_drain, 0, spin_limit);   // every product issued above has retired (bounded)
  } else if (warp < 2 + kNomGatherWarps) {
    // ------------------------------------------------------------ rows of the next item, kNomM / kNomGatherWarps a warp
    // Asynchronous copies straight into the swizzled tile, all in flight together; then a row per lane for the norms.
    float *rowinv = reinterpret_cast<float *>(smem + SL::kRowInv);
    constexpr int RW = kNomM / kNomGatherWarps, CH = D / 8, RI = 32 / CH;   // rows a warp, 16-byte chunks a row, rows a copy
    const int r0 = (warp - 2) * RW;
    int n_done = 0;
    for (int item = blockIdx.x;; item += gridDim.x) {
      NomItem it = {0, 0, 0, 0, 0, -1, 0, 0};
      if (item < n_items) it = nom_item(item, C, coarse, U, unit_info);
      const int buf = n_done & 1;
      const size_t ubase = (size_t)it.u * p.N_cap;
      if (it.n_ev >= 0 && it.t0 == it.t1) {   // a chunk without tiles (fewer tiles than chunks): an empty result
        for (int i = it.m0 + r0 + lane; i < min(it.m0 + r0 + RW, it.n_ev); i += 32) {
          nom[it.chunk * n_rows + ubase + i] = make_uint4(0xff800000u, 0xff800000u, 0xffffffffu, 0xffffffffu);   // (-inf, none)
        }
        continue;
      }
      const int m0 = it.m0 + r0;
      int mine[RW / 32];
#pragma unroll
      for (int k = 0; k < RW / 32; ++k) mine[k] = it.n_ev >= 0 && m0 + 32 * k + lane < it.n_ev ? ev_idx[ubase + m0 + 32 * k + lane] : -1;
      if (n_done >= 2 && !__all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_a_empty + 8 * buf, ((n_done >> 1) - 1) & 1, spin_limit))) {
        s_abort = 1;
        break;
      }
      ++n_done;
      if (warp == 2 && lane == 0) s_item[buf] = it;
      if (it.n_ev < 0) {
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_a_ready + 8 * buf);
        break;
      }
      const uint32_t At = SL::kA + buf * SL::kABytes;
      const int ch = lane % CH, sub = lane / CH;
#pragma unroll
      for (int k = 0; k < RW / 32; ++k) {
#pragma unroll
        for (int i = 0; i < 32; i += RI) {
          const int e = __shfl_sync(0xffffffffu, mine[k], i + sub), r = r0 + 32 * k + i + sub;
          cp_async_16(sbase + At + (ch >> 3) * (kNomM * 128) + r * 128 + (((ch & 7) ^ (r & 7)) << 4),
                      srcK + (ubase + (e >= 0 ? e : 0)) * D + ch * 8, e >= 0);
        }
      }
      cp_async_commit();
      cp_async_wait<0>();
      __syncwarp();
#pragma unroll 1
      for (int k = 0; k < RW / 32; ++k) {
        const int r = r0 + 32 * k + lane;
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
          const uint4 v = *reinterpret_cast<const uint4 *>(smem + At + (c >> 3) * (kNomM * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4));
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) { s0 = fmaf(bf16_lo(w[q]), bf16_lo(w[q]), s0); s1 = fmaf(bf16_hi(w[q]), bf16_hi(w[q]), s1); }
        }
        // (a row that does not exist, or of norm zero: a cut no column reaches)
        const float ri = rsqrtf(s0 + s1);
        if (kCut)
          *reinterpret_cast<uint4 *>(smem + SL::kAX + buf * (kNomM * 16) + r * 16) =
              ext_row(ri < CUDART_INF_F ? (p.merge_threshold - 2.f * kRankEps) / ri : kExtNever);
        rowinv[buf * kNomM + r] = ri;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_a_ready + 8 * buf);
    }
  } else {
    // ------------------------------------------------------------ accumulator drain
    const int ew = warp - 2 - kNomGatherWarps, quarter = warp & 3;   // (a warp reads the lanes 32 (warp mod 4) ..)
    const int cq = ew >> 2;                                          // which 64 of a tile's columns
    const int row = quarter * 32 + lane;                             // row of the item
    const uint32_t xbar = bar_x + 16 * quarter;
    const float *rowinv = reinterpret_cast<const float *>(smem + SL::kRowInv);
    uint32_t *xchg = reinterpret_cast<uint32_t *>(smem + SL::kXchg);
    int acc = 0, x_phase = 0;   // x_phase: a bit per set of A tiles
    for (int n_done = 0;; ++n_done) {
      const int buf = n_done & 1;
      if (!__all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_a_ready + 8 * buf, (n_done >> 1) & 1, spin_limit))) { s_abort = 1; break; }
      const NomItem it = s_item[buf];
      if (it.n_ev < 0) break;
      const size_t ubase = (size_t)it.u * p.N_cap;
      const bool row_ok = it.m0 + row < it.n_ev;
      // Values are compared before the division by |k_e|: the closeness margin and the threshold scale with it.
      const float rinv = rowinv[buf * kNomM + row];
      const bool live = it.m0 + quarter * 32 < it.n_ev;   // some of this warp's rows exist
      Top2 top, topb;   // two lists over alternate columns: two independent dependency chains
      top.init(2.f * kRankEps / rinv);
      topb.init(top.thr);
      const float cut0 = (p.merge_threshold - 2.f * kRankEps) / rinv;
      top.cut = row_ok && rinv < CUDART_INF_F ? cut0 : CUDART_INF_F;
      bool ok = true;
      for (int t = it.t0; t < it.t1; ++t, ++acc) {
        const int a = acc & 1;
        ok = __all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_t_full + 8 * a, (acc >> 1) & 1, spin_limit));
        if (!ok) break;
        tc_fence_after();
        const int c0 = t * kNomN + cq * 64, n_valid = it.n_ret - c0;   // this warp's columns that exist, if positive
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + a * kNomN + cq * 64;
        // rows and columns are the same entries (self_mask): the column of the row's own key does not count
        const int diag = self_mask ? it.m0 + row - c0 : -1;
        const int diag0 = it.m0 + quarter * 32 - c0;
#pragma unroll 1
        for (int off = 0; live && off < 64 && off < n_valid; off += 32) {   // 32 columns at a time: the register budget of 20 warps
          uint32_t r[32];
          tmem_ld_32x32(taddr + off, r);
          tmem_ld_wait();
          // the last columns may hold other rows' data, and the row's own key does not count
          const bool masked = n_valid < off + 32 || (self_mask && diag0 < off + 32 && off < diag0 + 32);
          if (masked) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (off + i >= n_valid || off + i == diag) r[i] = 0xff800000u;   // -inf
          }
          const float4 *wv = reinterpret_cast<const float4 *>(smem + SL::kInv + acc % SL::kInvTiles * (kNomN * 4)) + (cq * 64 + off) / 4;
          if constexpr (kCut) {
            // groups of four columns; what lies above the row's cut is positive (NaNs never show)
            float gm[8];
#pragma unroll
            for (int i = 0; i < 8; ++i)
              gm[i] = max3(fmaxf(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1])), __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
            const float all = max3(max3(gm[0], gm[1], gm[2]), max3(gm[3], gm[4], gm[5]), fmaxf(gm[6], gm[7]));
            if (__any_sync(0xffffffffu, all > 0.f)) {
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                if (!__any_sync(0xffffffffu, gm[i] > 0.f)) continue;
                const float4 w = wv[i];
                const int c = c0 + off + 4 * i;
                top.insert(fmaf(__uint_as_float(r[4 * i]), fabsf(w.x), cut0), c);
                topb.insert(fmaf(__uint_as_float(r[4 * i + 1]), fabsf(w.y), cut0), c + 1);
                top.insert(fmaf(__uint_as_float(r[4 * i + 2]), fabsf(w.z), cut0), c + 2);
                topb.insert(fmaf(__uint_as_float(r[4 * i + 3]), fabsf(w.w), cut0), c + 3);
              }
            }
          } else {
            const uint64_t ncut = pack_f32x2(-top.cut, -top.cut);
            float m_a = -1.f, m_b = -1.f;   // largest value - cut, if any reaches it
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              const float4 w = wv[i / 4];
              float d0, d1, d2, d3;
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), pack_f32x2(w.x, w.y), ncut), d0, d1);
              unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), pack_f32x2(w.z, w.w), ncut), d2, d3);
              m_a = max3(m_a, d0, d1);
              m_b = max3(m_b, d2, d3);
            }
            if (__any_sync(0xffffffffu, fmaxf(m_a, m_b) >= 0.f || top.cut == -CUDART_INF_F)) {
#pragma unroll
              for (int i = 0; i < 32; i += 4)   // groups of four columns that hold a candidate of some row
                offer4_above(top, topb, __uint_as_float(r[i]), __uint_as_float(r[i + 1]), __uint_as_float(r[i + 2]),
                             __uint_as_float(r[i + 3]), wv[i / 4], c0 + off + i);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_t_empty + 8 * a);
      }
      if (!ok) { s_abort = 1; break; }
      top.insert_any(topb.best, topb.bi);
      top.insert_any(topb.second, topb.si);
      // ---- Fold the four warps' results of each row and publish the chunk's.  Those of the later columns leave theirs and
      // go on.  They can be one item ahead at most: the item after that is not gathered before this one is folded.
      uint32_t *x = xchg + (size_t)(buf * kNomM + row) * 9;
      if (cq) {   // slots are below 65535 (N_cap <= 49152); -1 = none
        uint32_t *xw = x + (cq - 1) * 3;
        xw[0] = __float_as_uint(top.best);
        xw[1] = __float_as_uint(top.second);
        xw[2] = (uint32_t)(top.bi + 1) | ((uint32_t)(top.si + 1) << 16);
        __syncwarp();
        if (lane == 0) mbar_arrive(xbar + 8 * buf);
      } else {
        if (!__all_sync(0xffffffffu, !s_abort && mbar_wait_n(xbar + 8 * buf, (x_phase >> buf) & 1, spin_limit))) { s_abort = 1; break; }
#pragma unroll
        for (int w = 0; w < 3; ++w) {
          const uint32_t sl = x[3 * w + 2];
          top.insert_any(__uint_as_float(x[3 * w]), (int)(sl & 0xffffu) - 1);
          top.insert_any(__uint_as_float(x[3 * w + 1]), (int)(sl >> 16) - 1);
        }
        if (row_ok) {
          nom[it.chunk * n_rows + ubase + it.m0 + row] =
              make_uint4(__float_as_uint(top.best * rinv), __float_as_uint(top.second * rinv), (uint32_t)top.bi, (uint32_t)top.si);
        }
      }
      x_phase ^= 1 << buf;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_a_empty + 8 * buf);
    }
  }

  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (s_abort) {
    if (tid == 0) {
      atomicOr(status_dev, KEEPKV_DEV_TIMEOUT);
      // copies still in flight get a bounded chance to land before the shared memory goes away
      for (int i = 0; i < kNomStages; ++i) { mbar_wait_n(bar_b_full + 8 * i, 0, spin_limit); mbar_wait_n(bar_b_full + 8 * i, 1, spin_limit); }
    }
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int D, bool kCut>
static void launch_nominate_t(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                              const int32_t *ev_idx, const UnitInfo *unit_info, const float *inv_norm,
                              const uint4 *norm_ext, int32_t *sched, uint4 *nom, int nom_chunks, int32_t *status_dev, LaunchCtx &ctx,
                              int self_mask) {
  using SL = NomSmem<D>;
  constexpr size_t smem_bytes = (size_t)SL::kBytes + 1024;
  static bool attr_done_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_done_dev[dev & 63]) {
    cudaFuncSetAttribute(nominate_kernel<D, kCut>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    attr_done_dev[dev & 63] = true;
  }
  CUtensorMap mapB;
  if (!make_bf16_rows_map(&mapB, dst.K, (uint64_t)p.B * p.H_kv * p.N_cap, D, kNomN)) {
    if (ctx.err == cudaSuccess) ctx.err = cudaErrorInvalidValue;
    return;
  }
  launch_pdl(nominate_kernel<D, kCut>, dim3(sm_count()), dim3(kNomThreads), smem_bytes, ctx.stream,
      mapB, p, reinterpret_cast<const __nv_bfloat16 *>(src.K), ev_idx, unit_info, inv_norm, norm_ext, sched, nom,
      nom_chunks, status_dev, self_mask, debug_spin_limit(), debug_withhold());
  KEEPKV_CHECK_LAUNCH(ctx);
}

// Large prompts go to pairs of CTAs (nominate_pair.cu).  The buffer's capacity stands for their length, which the host does not know;
// columns: how many retained keys it expects a unit to have, 0 where most rows have none or few are evicted (in place).  The whole
// call, this form against pairs, us, 8 and 64 units: 4096 -> 819 entries 40.1 / 39.0 and 101 / 93, 4096 -> 1229 42.9 / 42.6 and
// 109 / 103, 6000 -> 1800 50.3 / 48.0 and 181 / 155, 8192 -> 819 51.8 / 49.8 and 169 / 151, 8192 -> 1638 57.2 / 53.9 and 230 / 194,
// 16384 -> 1638 (8 and 32 units) 94.6 / 85.1 and 250 / 209; merge-first of 4095 (8 units) and 6007 entries (32) 101 / 83 and 382 / 230.
// What the capacity misjudges, a cache that evicts 128 entries out of a large buffer: 1766 -> 1638 30.4 / 31.9 and 54.2 / 54.2,
// 1002 -> 874 29.1 / 30.6 and 40.6 / 41.4: half of a pair's rows do not exist.  (64 channels: 16 units of 20000 -> 4000 553 / 694.)
bool nominate_pairs(const keepkv_params &p, int columns) {
  return p.d == 128 && p.merge_threshold >= kNomStatic && p.N_cap >= kNomPairCap && columns >= kNomPairColumns;
}

void launch_nominate(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst, const int32_t *ev_idx,
                     const UnitInfo *unit_info, const float *inv_norm, const uint4 *norm_ext, int32_t *sched, uint4 *nom,
                     int nom_chunks, int32_t *status_dev, LaunchCtx &ctx, int columns, int self_mask, unsigned long long *tri_best) {
  if (tri_best || nominate_pairs(p, columns)) {
    launch_nominate_pairs(p, src, dst, ev_idx, unit_info, inv_norm, norm_ext, sched, nom, nom_chunks, status_dev, ctx, tri_best);
    return;
  }
  const bool cut = p.merge_threshold >= kNomStatic;
  auto launch = p.d == 128 ? (cut ? launch_nominate_t<128, true> : launch_nominate_t<128, false>)
                           : (cut ? launch_nominate_t<64, true> : launch_nominate_t<64, false>);
  launch(p, src, dst, ev_idx, unit_info, inv_norm, norm_ext, sched, nom, nom_chunks, status_dev, ctx, self_mask);
}

}  // namespace keepkv
