// The similarity search of nominate.cu for large prompts (128 channels, a merge threshold that the product subtracts): the same values,
// lists and screen, with the tensor cores of two CTAs on one product.
//
// Work item = (unit, 256 evicted rows, one chunk of 128-column tiles of the unit's retained keys).
// A persistent grid of pairs of CTAs, one CTA per SM, walks the items.  The tensor cores of a pair work on one product (M = 256,
// N = 128, bf16 -> fp32): either CTA holds half of the rows and half of the columns and gets the accumulator of its rows, so that
// columns are read once for 256 rows.  Inside a CTA:
//   warp 0      copies: its half of the column tiles (64 rows x D, 128-byte swizzle, and the norms) into a ring of 128 KB;
//   warp 1      the pair's first CTA: products, each into the next of four accumulators; the second: tells the first what has landed;
//   warps 2-3   gather the CTA's evicted rows of the next item from the src cache into the other A tile;
//   warps 4-19  drain: four groups of four warps, each with an accumulator of its own, so that one group's waits are another's work.
// Bound: the power limit.  At 698 cycles a tile, 640 of them products, the tensor pipe runs at the 1.61 PFLOP/s of a cuBLAS
// product and the clock at 1.65 GHz; candidates, and what an item costs beside its tiles, make it 790 (47 tiles an item) to 940 (13).
// Measured, 64 units of 6554 x 1638 keys, 176 GFLOP: the loop takes 162 us, 190 us in nominate.cu's form (2059 cycles for 256 columns,
// waits of the products for copies and for the slowest of the sixteen warps that share two accumulators).  What it took, cycles
// per 256 columns: pairs with two accumulators 2189 (2853 with arrivals of the cluster's scope), copies and products
// issued by one thread's loops 2041, four accumulators with groups 2064, the last group to be done folding an item 2018, one copy of
// the code behind the screen 1876.
// Where half a block's groups of four columns hold a candidate all its columns are looked at in line.  Keys along a common direction,
// three quarters of the pairs above the threshold: 64 units of 8191 -> 1638 (the call) 1314 us with a loop over the groups, 1105 now,
// 1161 in nominate.cu's form; merge-first, 32 units of 6007, 21.5 ms with an offer to a column for every pair, 1.03 ms with one for the
// best of 32 rows, 1.05 ms in nominate.cu's form (0.92 / 0.97 / 1.42 ms for 64 centres).  With candidates rare the calls take as long
// as before.
// With 64 channels a tile's products are half as long as its drain, and this form is up to a quarter slower than nominate.cu's.
// Every wait is bounded; a wait that runs out raises KEEPKV_DEV_TIMEOUT, every warp of the CTA leaves its loop, what is
// in flight gets a bounded time to end, the pair meets, tensor memory is freed.
#include "compress.cuh"
#include "ptx.cuh"

namespace keepkv {

constexpr int kPairD = 128;         // channels
constexpr int kPairM = 128;         // evicted rows per CTA (tensor-memory lanes)
constexpr int kPairRows = 2 * kPairM; // ... and per item, which is a pair of CTAs'
constexpr int kPairN = 128;         // retained columns per tile
constexpr int kPairHalf = kPairN / 2; // ... of which a CTA holds these many
constexpr int kPairAcc = 4;         // accumulators, each with a group of four drain warps
constexpr int kPairDrainWarps = 4 * kPairAcc;
constexpr int kPairMany = 4;        // of the eight groups of four columns of a block, see the drain
constexpr int kPairTold = 32;       // entries of a drain warp's stash of offers; up to eight come at a time
constexpr int kPairGatherWarps = 2; // (20 warps in all: 96 registers a thread)
constexpr int kPairThreads = 32 * (2 + kPairGatherWarps + kPairDrainWarps);

struct PairSmem {
  static constexpr int D = kPairD;
  static constexpr int kSub = D / 64;                     // 64-channel (128-byte) K atoms per row
  static constexpr int kABytes = kSub * kPairM * 128;
  static constexpr int kBBytes = kSub * kPairHalf * 128;   // a CTA's half of a column tile
  static constexpr int kTiles = 131072 / kBBytes;         // column tiles the ring holds
  static constexpr int kA = 0;                            // [2]: the next item is gathered while this one runs
  static constexpr int kB = 2 * kABytes;
  static constexpr int kAX = kB + kTiles * kBBytes;   // [2][128] x 16 B  eight more channels of the rows
  static constexpr int kBX = kAX + 2 * kPairM * 16;        // [kTiles][64] x 16 B  and of the columns
  static constexpr int kZero = kBX + kTiles * kPairHalf * 16; // [128] x 16 B  and eight more that are zero, for all of them
  // Inverse norms of the columns outlive their tile's stage: when tile t + 2 kPairAcc has been multiplied, tile t + kPairAcc has been
  // given back by the warps that were done with tile t before.
  static constexpr int kInvTiles = kTiles + 2 * kPairAcc;
  static constexpr int kInv = kZero + kPairM * 16;              // f32 [kInvTiles][128]
  static constexpr int kRowInv = kInv + kInvTiles * kPairN * 4; // f32 [2][128]        inverse norms of the staged rows
  static constexpr int kXchg = kRowInv + 2 * kPairM * 4;        // u32 [2][128][3][3]  results of the groups that are done first
  static constexpr int kCoarse = kXchg + 2 * kPairM * 36;       // i32 [kMaxUnits / 32]  row tiles before each 32 units
  static constexpr int kBytes = kCoarse + kMaxUnits / 32 * 4;
  static constexpr int kTold = kXchg;   // a triangle's stashes of offers: nothing is exchanged there
  static_assert(kTold % 16 == 0 && kPairDrainWarps * kPairTold * 16 <= 2 * kPairM * 36, "the stashes take the place of the exchange");
};

// Two words hold the two largest cosines offered so far, with their slots, in any order of the offers: equal values go to
// the lower slot.  (Only positive ones count, so their bits are in order; an empty word is zero.  A look at the second word first is
// a trip to L2 that few offers save: 447 -> 441 us for merge-first compressions without it.)
__device__ __forceinline__ unsigned long long tri_word(float v, int slot) {
  return (unsigned long long)__float_as_uint(v) << 32 | (0xffffffffu - (unsigned)slot);
}
__device__ __forceinline__ void tri_offer(unsigned long long *best, float v, int slot) {
  if (!(v > 0.f)) return;
  const unsigned long long x = tri_word(v, slot);
  const unsigned long long old = atomicMax(best, x), less = old < x ? old : x;
  if (less) atomicMax(best + 1, less);
}

// Of the lanes m those with the two largest values (positive; of equal ones the lowest lanes).
__device__ __forceinline__ unsigned two_largest(unsigned m, float v) {
  const int lane = threadIdx.x & 31;
  uint32_t left = m >> lane & 1u ? __float_as_uint(v) : 0u;
  m = 0;
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const uint32_t most = __reduce_max_sync(0xffffffffu, left);
    const int l = __ffs(__ballot_sync(0xffffffffu, left == most)) - 1;
    m |= 1u << l;
    if (lane == l) left = 0u;
  }
  return m;
}

// A block of cosines, 32 rows (lanes) by 32 columns (r, positive floats): every lane gets the largest value of one column, its row --
// of equal values the lowest -- and the second largest value.  Halves of the columns are exchanged between neighbouring ranges
// of rows, step by step: 31 exchanges for the block.
struct ColumnTop { uint32_t best, second; int row; };
template <int kDist>
__device__ __forceinline__ ColumnTop column_meet(const ColumnTop &lo, const ColumnTop &hi) {   // of the lower and the higher column
  const bool up = threadIdx.x & kDist;
  const ColumnTop own = up ? hi : lo, give = up ? lo : hi;
  ColumnTop got;
  got.best = __shfl_xor_sync(0xffffffffu, give.best, kDist);
  got.second = kDist > 1 ? __shfl_xor_sync(0xffffffffu, give.second, kDist) : 0u;
  got.row = kDist > 1 ? __shfl_xor_sync(0xffffffffu, give.row, kDist) : (int)((threadIdx.x & 31) ^ 1);
  ColumnTop t;
  t.row = got.best + (up ? 1u : 0u) > own.best ? got.row : own.row;   // (the upper lanes' partner has the lower rows)
  t.best = max(own.best, got.best);
  t.second = max(min(own.best, got.best), max(own.second, got.second));
  return t;
}
// Column kFirst and the columns behind it, as many as lanes are met.
template <int kDist, int kFirst, int kN>
__device__ __forceinline__ ColumnTop column_top(const uint32_t (&r)[kN]) {
  if constexpr (kDist == 0) return ColumnTop{r[kFirst], 0u, (int)(threadIdx.x & 31)};
  else return column_meet<kDist>(column_top<kDist / 2, kFirst>(r), column_top<kDist / 2, kFirst + kDist>(r));
}

struct __align__(16) PairItem { int u, m0, chunk, t0, t1, n_ev, n_ret, pad; };

// Tiles of a unit's triangle in front of row tile i of T: those of the row tiles before it, each from the diagonal on.
__device__ __forceinline__ int tri_before(int i, int T) { return i * T - i * (i - 1) * (kPairRows / kPairN) / 2; }
// What a unit counts for in the division of the work: row tiles, or tiles of its triangle.
template <bool kTri>
__device__ __forceinline__ int pair_weight(int n_ev) {
  const int R = (n_ev + kPairRows - 1) / kPairRows;
  return kTri ? tri_before(R, (n_ev + kPairN - 1) / kPairN) : R;
}

// The whole warp looks up where position `at` of all units' weights lies: among the units first by groups of 32 units, then
// inside the group.  it.u, it.n_ev, it.n_ret; returned: the position inside the unit.
template <bool kTri>
__device__ __forceinline__ int pair_unit(PairItem &it, int at, const int *coarse, int U, const UnitInfo *unit_info) {
  const int lane = threadIdx.x & 31, groups = (U + 31) >> 5;
  int g = -1;   // last group that starts at or before it
  for (int k = 0; k < groups; k += 32) {
    const bool le = k + lane < groups && coarse[k + lane] <= at;
    g += __popc(__ballot_sync(0xffffffffu, le));
  }
  const int u = g * 32 + lane;
  int n_ev = 0, n_ret = 0;
  if (u < U) { const UnitInfo ui = unit_info[u]; n_ev = ui.n_ev; n_ret = ui.n_ret; }
  const int w = pair_weight<kTri>(n_ev);
  int x = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  const int r = at - coarse[g];
  const int l = __ffs(__ballot_sync(0xffffffffu, x > r)) - 1;   // (it lies in this group, so one lane's sum exceeds r)
  it.u = g * 32 + l;
  it.n_ev = __shfl_sync(0xffffffffu, n_ev, l);
  it.n_ret = __shfl_sync(0xffffffffu, n_ret, l);
  it.pad = 0;
  return r - __shfl_sync(0xffffffffu, x - w, l);
}
__device__ __forceinline__ PairItem pair_item(int item, int C, const int *coarse, int U, const UnitInfo *unit_info) {
  PairItem it;
  it.m0 = pair_unit<false>(it, item / C, coarse, U, unit_info) * kPairRows;
  it.chunk = item % C;
  const int T = (it.n_ret + kPairN - 1) / kPairN;
  it.t0 = it.chunk * T / C;
  it.t1 = (it.chunk + 1) * T / C;
  return it;
}
// The tiles from position `at` of all triangles on that share a row tile, up to position `end`.
__device__ __forceinline__ PairItem pair_item_tri(int at, int end, const int *coarse, int U, const UnitInfo *unit_info) {
  static_assert(kPairRows % kPairN == 0, "a triangle's row tiles are whole column tiles");
  PairItem it;
  const int r = pair_unit<true>(it, at, coarse, U, unit_info), R = (it.n_ev + kPairRows - 1) / kPairRows;
  const int T = (it.n_ev + kPairN - 1) / kPairN;
  int i = -1;
  for (int k = 0; k < R; k += 32) {
    const int j = k + (int)(threadIdx.x & 31);
    i += __popc(__ballot_sync(0xffffffffu, j < R && tri_before(j, T) <= r));
  }
  it.m0 = i * kPairRows;
  it.chunk = 0;
  it.t0 = i * (kPairRows / kPairN) + r - tri_before(i, T);
  it.t1 = min(T, it.t0 + end - at);
  return it;
}

// Columns of tile t that are multiplied: a unit's last tile as far as it has any, in steps of 32.
__device__ __forceinline__ int pair_cols(const PairItem &it, int t) { return min(kPairN, (it.n_ret - t * kPairN + 31) & ~31); }

// kTri: rows and columns are the same entries, and a product is taken for two cosines: tiles from the diagonal on
// only.  A pair of CTAs walks an equal range of all triangles' tiles.  What is above the threshold is offered to the row's list as
// before, and beyond the square on the diagonal to the column's as well; both are in global memory, two words each (tri_offer).
// Half the products, and the power they take: merge-first compression of 32 units of 6007 entries 493 -> 436 us.
template <bool kTri>
__global__ void __launch_bounds__(kPairThreads, 1)
nominate_pair_kernel(const __grid_constant__ CUtensorMap mapB, keepkv_params p, const __nv_bfloat16 *__restrict__ srcK,
                const int32_t *__restrict__ ev_idx, const UnitInfo *__restrict__ unit_info,
                const float *__restrict__ inv_norm, const uint4 *__restrict__ norm_ext, int32_t *sched,
                uint4 *__restrict__ nom, int C_max, int32_t *status_dev,
                unsigned long long *__restrict__ tri_best, int spin_limit, int withhold) {
  using SL = PairSmem;
  constexpr int D = kPairD;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  constexpr int kStages = SL::kTiles;
  // a_ready[2], a_empty[2], t_full, drain, x_full[4][2], b_full, b_empty; of the pair's first CTA: t_empty, both CTAs' rows[2]
  __shared__ __align__(8) uint64_t bars[4 + kPairAcc + 1 + 8 + 2 * kStages + kPairAcc + 2];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(16) PairItem s_item[2];   // what the staged rows belong to; n_ev < 0: the CTA's items are done
  __shared__ int s_wtot[kPairThreads / 32], s_wmax[kPairThreads / 32];
  __shared__ int s_done[2][4];   // per set of A tiles and 32 rows: groups that are done with the item
  __shared__ volatile int s_abort;

  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar_a_ready = smem_u32(&bars[0]), bar_a_empty = smem_u32(&bars[2]), bar_t_full = smem_u32(&bars[4]);
  const uint32_t bar_drain = bar_t_full + 8 * kPairAcc, bar_x = bar_drain + 8;
  const uint32_t bar_b_full = bar_x + 64, bar_b_empty = bar_b_full + 8 * kStages;
  const uint32_t bar_t_empty = bar_b_empty + 8 * kStages, bar_rows = bar_t_empty + 8 * kPairAcc;
  int *coarse = reinterpret_cast<int *>(smem + SL::kCoarse);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int U = p.B * p.H_kv;
  const size_t n_rows = (size_t)U * p.N_cap;
  const uint32_t rank = cluster_ctarank();          // in the pair
  const int pair = (int)cluster_id(), n_pairs = (int)gridDim.x / 2;

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_a_ready + 8 * i, kPairGatherWarps);
      mbar_init(bar_a_empty + 8 * i, 1 + kPairDrainWarps);
      mbar_init(bar_rows + 8 * i, 2 * kPairGatherWarps);
    }
    for (int i = 0; i < kPairAcc; ++i) { mbar_init(bar_t_full + 8 * i, 1); mbar_init(bar_t_empty + 8 * i, 2 * 4); }
    for (int i = 0; i < kStages; ++i) {
      mbar_init(bar_b_full + 8 * i, rank == 0 ? 2 : 1);   // the first CTA's: both halves of a tile are here
      mbar_init(bar_b_empty + 8 * i, 1);
    }
    for (int i = 0; i < 8; ++i) mbar_init(bar_x + 8 * i, 3);
    mbar_init(bar_drain, 1);
    for (int i = 0; i < 8; ++i) s_done[i >> 2][i & 3] = 0;
    s_abort = 0;
    mbar_fence_init();
    fence_proxy_async_smem();
    prefetch_tensormap(&mapB);
  }
  if (tid >= 64 && tid < 64 + kPairM) {
    reinterpret_cast<uint4 *>(smem + SL::kZero)[tid - 64] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  pdl_wait();      // barrier set-up overlaps the previous kernel's tail
  pdl_trigger();
  if (warp == 1) {   // (not before the wait: see tmem_alloc)
    tmem_alloc(CtaPair{}, smem_u32(&s_tmem), 512);
    tmem_relinquish(CtaPair{});
  }
  int total_m = 0, t_max = 0;
  {   // exclusive prefix of the units' row tiles (or tiles of triangles), kept for every 32nd: one unit per thread and pass
    for (int u0 = 0; u0 < U; u0 += kPairThreads) {
      const int u = u0 + tid;
      int t = 0, cols = 0;
      if (u < U) { const UnitInfo ui = unit_info[u]; t = pair_weight<kTri>(ui.n_ev); cols = ui.n_ret; }
      const int sum = __reduce_add_sync(0xffffffffu, t), mx = __reduce_max_sync(0xffffffffu, cols);
      if (lane == 0) { s_wtot[warp] = sum; s_wmax[warp] = mx; }
      __syncthreads();
      int off = 0, tot = 0;
#pragma unroll
      for (int w = 0; w < kPairThreads / 32; ++w) {
        const int v = s_wtot[w];
        off += w < warp ? v : 0;
        tot += v;
        t_max = max(t_max, s_wmax[w]);
      }
      if (lane == 0 && u < U) coarse[u >> 5] = total_m + off;
      total_m += tot;
      __syncthreads();
    }
    t_max = (t_max + kPairN - 1) / kPairN;
  }
  tc_fence_before();
  __syncthreads();
  // The other CTA's barriers are initialised, its columns of tensor memory allocated.  (What it relies on lies behind the fence of the
  // initialisation and its own barrier, so the arrival is relaxed: as a release a call took up to 1 us longer.)
  cluster_arrive_relaxed();
  cluster_wait();
  tc_fence_after();

  const uint32_t tmem = s_tmem;
  // Column chunks per row tile: what makes the longest CTA shortest, an item costing about a tile and a half beside its
  // tiles (first columns, publishing).  Without chunks 96 items on 74 pairs take as long as 148.
  int C = 1;
  if (!kTri) {
    int cost = 0x7fffffff;
    for (int c = 1; c <= C_max; ++c) {
      const int rounds = (total_m * c + n_pairs - 1) / n_pairs, k = rounds * ((t_max + c - 1) / c + 3);
      if (k < cost) { cost = k; C = c; }
    }
  }
  const int n_items = total_m * C;
  if (!kTri && blockIdx.x == 0 && tid == 0) sched[0] = C;

  if (warp == 0) {
    // ------------------------------------------------------------ column tiles
    // (One thread, as for the products: a vote and a warp's barrier per step were what the tensor core waited for.)
    if (elect_one()) {
      int n_tiles = 0;
      bool ok = true;
      for (int n_done = 0; ok; ++n_done) {   // (watches the rows' barrier only: an item's last product waits for its columns)
        ok = mbar_wait_or(bar_a_ready + 8 * (n_done & 1), (n_done >> 1) & 1, spin_limit, &s_abort);
        if (!ok) break;
        const PairItem it = s_item[n_done & 1];
        if (it.n_ev < 0) break;
        for (int t = it.t0; t < it.t1; ++t, ++n_tiles) {
          // the product takes the first half of the tile's columns from the first CTA, the rest from the second
          const int first = it.u * p.N_cap + t * kPairN, row = first + (int)rank * (pair_cols(it, t) / 2);
          const int s = n_tiles % kStages;
          const uint32_t full = bar_b_full + 8 * s;
          ok = mbar_wait_or(bar_b_empty + 8 * s, ((n_tiles / kStages) & 1) ^ 1, spin_limit, &s_abort);
          if (!ok) break;
          if (2 * n_tiles + (int)rank == withhold) continue;   // (test hook: this half of a tile is never asked for)
          mbar_expect_tx(full, SL::kBBytes + kPairHalf * 16 + kPairN * 4);
          tma_load_3d(sbase + SL::kB + s * SL::kBBytes, &mapB, 0, row, 0, full);
          bulk_load_1d(sbase + SL::kBX + s * (kPairHalf * 16), norm_ext + row, kPairHalf * 16, full);
          bulk_load_1d(sbase + SL::kInv + n_tiles % SL::kInvTiles * (kPairN * 4), inv_norm + first, kPairN * 4, full);
        }
      }
      if (!ok) s_abort = 1;
    }
    __syncwarp();
  } else if (warp == 1 && rank == 0) {
    // ------------------------------------------------------------ products, of both CTAs
    if (elect_one()) {
      int acc = 0;
      bool ok = true;
      const uint32_t zero = sbase + SL::kZero;
      for (int n_done = 0; ok; ++n_done) {
        const int buf = n_done & 1;
        ok = mbar_wait_or(bar_rows + 8 * buf, (n_done >> 1) & 1, spin_limit, &s_abort);
        if (!ok) break;
        const PairItem it = s_item[buf];
        if (it.n_ev < 0) break;
        const uint64_t ad = umma_desc_sw128(sbase + SL::kA + buf * SL::kABytes);
        for (int t = it.t0; t < it.t1; ++t, ++acc) {
          const int a = acc % kPairAcc, s = acc % kStages;
          const uint32_t idesc = umma_idesc_bf16(kPairRows, pair_cols(it, t)), dt = tmem + a * kPairN;
          const uint64_t bd = umma_desc_sw128(sbase + SL::kB + s * SL::kBBytes);
          ok = mbar_wait_or(bar_b_full + 8 * s, (acc / kStages) & 1, spin_limit, &s_abort) &&
               mbar_wait_or(bar_t_empty + 8 * a, ((acc / kPairAcc) & 1) ^ 1, spin_limit, &s_abort);
          if (!ok) break;
          tc_fence_after();
#pragma unroll
          for (int k = 0; k < 4 * SL::kSub; ++k)   // (descriptor addresses count 16-byte units)
            umma_bf16(CtaPair{}, dt, ad + (k >> 2) * (kPairM * 8) + (k & 3) * 2, bd + (k >> 2) * (kPairHalf * 8) + (k & 3) * 2, idesc,
                      k > 0 ? 1u : 0u);
          umma_bf16(CtaPair{}, dt, umma_desc_plain(sbase + SL::kAX + buf * (kPairM * 16), zero),
                    umma_desc_plain(sbase + SL::kBX + s * (kPairHalf * 16), zero), idesc, 1u);
          umma_commit(CtaPair{}, bar_t_full + 8 * a);
          umma_commit(CtaPair{}, bar_b_empty + 8 * s);   // the stage may be refilled once these have read it
        }
        if (!ok) break;
        umma_commit(CtaPair{}, bar_a_empty + 8 * buf);   // the rows have been read
      }
      if (!ok) s_abort = 1;
      umma_commit(CtaPair{}, bar_drain);
      mbar_wait_n(bar_drain, 0, spin_limit);   // every product issued above has retired (bounded)
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ the second CTA's columns are told to the first
    if (elect_one()) {
      const uint32_t peer = mapa_shared(bar_b_full, 0);
      int n_tiles = 0;
      bool ok = true;
      for (int n_done = 0; ok; ++n_done) {
        ok = mbar_wait_or(bar_a_ready + 8 * (n_done & 1), (n_done >> 1) & 1, spin_limit, &s_abort);
        if (!ok) break;
        const PairItem it = s_item[n_done & 1];
        if (it.n_ev < 0) break;
        for (int i = it.t1 - it.t0; i > 0; --i, ++n_tiles) {
          const int s = n_tiles % kStages;
          ok = mbar_wait_or(bar_b_full + 8 * s, (n_tiles / kStages) & 1, spin_limit, &s_abort);
          if (!ok) break;
          mbar_arrive_cluster(peer + 8 * s);
        }
      }
      if (!ok) s_abort = 1;
      mbar_wait_n(bar_drain, 0, spin_limit);
    }
    __syncwarp();
  } else if (warp < 2 + kPairGatherWarps) {
    // ------------------------------------------------------------ rows of the next item, kPairM / kPairGatherWarps a warp
    // Asynchronous copies straight into the swizzled tile, all in flight together; then a row per lane for the norms.
    float *rowinv = reinterpret_cast<float *>(smem + SL::kRowInv);
    constexpr int RW = kPairM / kPairGatherWarps, CH = D / 8, RI = 32 / CH;   // rows a warp, 16-byte chunks a row, rows a copy
    const int r0 = (warp - 2) * RW;
    const uint32_t rows = mapa_shared(bar_rows, 0);
    int n_done = 0;
    const int end = kTri ? (int)((long long)(pair + 1) * total_m / n_pairs) : n_items;
    for (int item = kTri ? (int)((long long)pair * total_m / n_pairs) : pair;;) {
      PairItem it = {0, 0, 0, 0, 0, -1, 0, 0};
      if (item < end) it = kTri ? pair_item_tri(item, end, coarse, U, unit_info) : pair_item(item, C, coarse, U, unit_info);
      item += kTri ? max(1, it.t1 - it.t0) : n_pairs;
      it.m0 += (int)rank * kPairM;
      const int buf = n_done & 1;
      const size_t ubase = (size_t)it.u * p.N_cap;
      if (!kTri && it.n_ev >= 0 && it.t0 == it.t1) {   // a chunk without tiles (fewer tiles than chunks): an empty result
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
        if (lane == 0) { mbar_arrive(bar_a_ready + 8 * buf); mbar_arrive_cluster(rows + 8 * buf); }
        break;
      }
      const uint32_t At = SL::kA + buf * SL::kABytes;
      const int ch = lane % CH, sub = lane / CH;
#pragma unroll
      for (int k = 0; k < RW / 32; ++k) {
#pragma unroll
        for (int i = 0; i < 32; i += RI) {
          const int e = __shfl_sync(0xffffffffu, mine[k], i + sub), r = r0 + 32 * k + i + sub;
          cp_async_16(sbase + At + (ch >> 3) * (kPairM * 128) + r * 128 + (((ch & 7) ^ (r & 7)) << 4),
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
          const uint4 v = *reinterpret_cast<const uint4 *>(smem + At + (c >> 3) * (kPairM * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4));
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) { s0 = fmaf(bf16_lo(w[q]), bf16_lo(w[q]), s0); s1 = fmaf(bf16_hi(w[q]), bf16_hi(w[q]), s1); }
        }
        // (a row that does not exist, or of norm zero: a cut no column reaches)
        const float ri = rsqrtf(s0 + s1);
        *reinterpret_cast<uint4 *>(smem + SL::kAX + buf * (kPairM * 16) + r * 16) =
            ext_row(ri < CUDART_INF_F ? (p.merge_threshold - 2.f * kRankEps) / ri : kExtNever);
        rowinv[buf * kPairM + r] = ri;
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(bar_a_ready + 8 * buf);
        mbar_arrive_cluster(rows + 8 * buf);
      }
    }
  } else {
    // ------------------------------------------------------------ accumulator drain
    const int ew = warp - 2 - kPairGatherWarps, quarter = warp & 3;   // (a warp reads the lanes 32 (warp mod 4) ..)
    const int grp = ew >> 2;                                         // which of the accumulators
    const int row = quarter * 32 + lane;                             // row of the item
    const uint32_t xbar = bar_x + 16 * quarter, t_empty = mapa_shared(bar_t_empty, 0);
    const float *rowinv = reinterpret_cast<const float *>(smem + SL::kRowInv);
    uint32_t *xchg = reinterpret_cast<uint32_t *>(smem + SL::kXchg);
    int acc = 0, x_phase = 0;   // x_phase: a bit per set of A tiles
    // kTri: cosines that columns have yet to hear.  An offer is two trips to L2, which up to 32 of them make together.
    const uint32_t told = sbase + SL::kTold + ew * (kPairTold * 16);   // uint4 [kPairTold]  value, row, column
    int n_told = 0;
    auto offer_told = [&] {
      __syncwarp();
      if (lane < n_told) {
        const uint4 x = ld_shared_v4(told + lane * 16);
        tri_offer(tri_best + (size_t)x.z * 4 + 2, __uint_as_float(x.x), (int)x.y);
      }
      __syncwarp();
      n_told = 0;
    };
    // Lanes m have v for column `to`.  Of the warp's rows only two can be among the column's two best.
    auto tell = [&](unsigned m, float v, int row, int to) {
      if (__popc(m) > 2) m = two_largest(m, v);
      if (m >> lane & 1u)
        st_shared_v4(told + (n_told + __popc(m & ((1u << lane) - 1u))) * 16, make_uint4(__float_as_uint(v), (uint32_t)row, (uint32_t)to, 0u));
      n_told += __popc(m);
    };
    for (int n_done = 0;; ++n_done) {
      const int buf = n_done & 1;
      if (!__all_sync(0xffffffffu, !s_abort && mbar_wait_n(bar_a_ready + 8 * buf, (n_done >> 1) & 1, spin_limit))) { s_abort = 1; break; }
      const PairItem it = s_item[buf];
      if (it.n_ev < 0) break;
      const size_t ubase = (size_t)it.u * p.N_cap;
      const bool row_ok = it.m0 + row < it.n_ev;
      // Values are compared before the division by |k_e|.
      const float rinv = rowinv[buf * kPairM + row];
      const bool live = it.m0 + quarter * 32 < it.n_ev;   // some of this warp's rows exist
      Top2 top, topb;   // two lists over alternate columns: two independent dependency chains
      top.init(0.f);
      topb.init(0.f);
      const float cut0 = (p.merge_threshold - 2.f * kRankEps) / rinv;
      bool ok = true;
      for (int t = it.t0; t < it.t1; ++t, ++acc) {
        if (acc % kPairAcc != grp) continue;
        const bool beyond = t / (kPairRows / kPairN) > it.m0 / kPairRows;   // (of a square on the diagonal both halves are multiplied)
        const int c0 = t * kPairN, n_valid = min(kPairN, it.n_ret - c0);   // columns that exist
        ok = __all_sync(0xffffffffu, mbar_wait_or(bar_t_full + 8 * grp, (acc / kPairAcc) & 1, spin_limit, &s_abort));
        if (!ok) break;
        tc_fence_after();
        const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + grp * kPairN;
        const uint32_t inv = sbase + SL::kInv + acc % SL::kInvTiles * (kPairN * 4);
        // rows and columns are the same entries: the column of the row's own key does not count
        const int diag = kTri ? it.m0 + row - c0 : -1;
        const int diag0 = it.m0 + quarter * 32 - c0;
#pragma unroll 1
        for (int off = 0; live && off < n_valid; off += 32) {   // 32 columns at a time: the register budget of 20 warps
          uint32_t r[32];
          tmem_ld_32x32(taddr + off, r);
          tmem_ld_wait();
          // the last columns may hold other rows' data, and the row's own key does not count
          const bool masked = n_valid < off + 32 || (kTri && diag0 < off + 32 && off < diag0 + 32);
          if (masked) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (off + i >= n_valid || off + i == diag) r[i] = 0xff800000u;   // -inf
          }
          // groups of four columns; what lies above the row's cut is positive (NaNs never show)
          float gm[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            gm[i] = max3(fmaxf(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1])), __uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3]));
          const float all = max3(max3(gm[0], gm[1], gm[2]), max3(gm[3], gm[4], gm[5]), fmaxf(gm[6], gm[7]));
          if (__any_sync(0xffffffffu, all > 0.f)) {
            uint32_t some = 0;   // groups of columns with a candidate
#pragma unroll
            for (int i = 0; i < 8; ++i) some |= gm[i] > 0.f ? 1u << i : 0u;
            some = __reduce_or_sync(0xffffffffu, some);
            if (__popc(some) >= kPairMany) {
              // Prompts of similar keys: the price of a block does not depend on how many pairs pass.  The rows' lists take all of
              // them, the columns' what is best for each among the warp's rows.
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 w = ld_shared_f4(inv + (off + 4 * i) * 4);
                const int c = c0 + off + 4 * i;
                const float v[4] = {fmaf(__uint_as_float(r[4 * i]), fabsf(w.x), cut0), fmaf(__uint_as_float(r[4 * i + 1]), fabsf(w.y), cut0),
                                    fmaf(__uint_as_float(r[4 * i + 2]), fabsf(w.z), cut0), fmaf(__uint_as_float(r[4 * i + 3]), fabsf(w.w), cut0)};
                top.insert(v[0], c);
                topb.insert(v[1], c + 1);
                top.insert(v[2], c + 2);
                topb.insert(v[3], c + 3);
              }
              if (kTri && beyond) {
                unsigned long long *lists = tri_best + (ubase + c0 + off + lane) * 4 + 2;
                const unsigned long long heard = off + lane < n_valid ? __ldcg(lists + 1) : ~0ull;
                ColumnTop half[2];
#pragma unroll
                for (int k = 0; k < 2; ++k) {   // (read once more: nothing spills)
                  uint32_t q[16];
                  tmem_ld_32x16(taddr + off + 16 * k, q);
                  tmem_ld_wait();
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    const float4 w = ld_shared_f4(inv + (off + 16 * k + 4 * i) * 4);
                    const float n[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j)   // (a NaN is 0)
                      q[4 * i + j] = __float_as_uint(fmaxf(fmaf(__uint_as_float(q[4 * i + j]), fabsf(n[j]), cut0) * rinv, 0.f));
                  }
                  half[k] = column_top<8, 0>(q);
                }
                const ColumnTop mine = column_meet<16>(half[0], half[1]);

                const float v = __uint_as_float(mine.best);
                const int slot = it.m0 + quarter * 32 + mine.row;
                const bool wants = v > p.merge_threshold - 2.f * kRankEps && tri_word(v, slot) > heard;
                if (wants) tri_offer(lists, v, slot);
                // (Seldom: rows of the warp that are as close to the column as its best but for the margin.  What is further
                // below the warp's best is further below the column's, and the decision looks at nothing there.)
                const float near = v - 2.f * kRankEps;
#pragma unroll 1
                for (unsigned ls = __ballot_sync(0xffffffffu, wants && __uint_as_float(mine.second) >= near); ls; ls &= ls - 1) {
                  const int i = __ffs(ls) - 1;
                  const int first = __shfl_sync(0xffffffffu, mine.row, i);
                  const float lnear = __shfl_sync(0xffffffffu, near, i);
                  uint32_t q;
                  tmem_ld_32x1(taddr + off + i, q);
                  const float n = ld_shared_f32(inv + (off + i) * 4);
                  tmem_ld_wait();
                  const float pv = fmaf(__uint_as_float(q), fabsf(n), cut0) * rinv;
                  tell(__ballot_sync(0xffffffffu, pv >= lnear && lane != first), pv, it.m0 + row, (int)ubase + c0 + off + i);
                  if (n_told > kPairTold - 8) offer_told();
                }
              }
            } else {
              // An eighth of the blocks, and mostly one group of theirs: read once more, so that there is one copy of this code
              // (with eight copies of it, a tile took 1009 cycles, with one 938).
#pragma unroll 1
              for (; some; some &= some - 1) {
                const int i = __ffs(some) - 1, c = c0 + off + 4 * i;
                uint32_t q[4];
                tmem_ld_32x4(taddr + off + 4 * i, q);
                const float4 w = ld_shared_f4(inv + (off + 4 * i) * 4);
                tmem_ld_wait();
                float v[4] = {__uint_as_float(q[0]), __uint_as_float(q[1]), __uint_as_float(q[2]), __uint_as_float(q[3])};
                const float n[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const bool counts = off + 4 * i + j < n_valid && off + 4 * i + j != diag;
                  v[j] = counts ? fmaf(v[j], fabsf(n[j]), cut0) : -CUDART_INF_F;
                }
                top.insert(v[0], c);
                topb.insert(v[1], c + 1);
                top.insert(v[2], c + 2);
                topb.insert(v[3], c + 3);
                if (kTri && beyond) {   // what the columns are to hear
                  uint32_t any4 = 0;
#pragma unroll
                  for (int j = 0; j < 4; ++j) any4 |= __uint_as_float(q[j]) > 0.f && v[j] > 0.f ? 1u << j : 0u;
#pragma unroll 1
                  for (unsigned js = __reduce_or_sync(0xffffffffu, any4); js; js &= js - 1) {
                    const int j = __ffs(js) - 1;
                    const float x = j & 2 ? (j & 1 ? v[3] : v[2]) : (j & 1 ? v[1] : v[0]);
                    tell(__ballot_sync(0xffffffffu, any4 >> j & 1u), x * rinv, it.m0 + row, (int)ubase + c + j);
                  }
                  if (n_told > kPairTold - 8) offer_told();
                }
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(t_empty + 8 * grp);
      }
      if (!ok) { s_abort = 1; break; }
      top.insert_any(topb.best, topb.bi);
      top.insert_any(topb.second, topb.si);
      if constexpr (kTri) {
        if (row_ok) {
          unsigned long long *best = tri_best + (ubase + it.m0 + row) * 4;
          if (top.bi >= 0) tri_offer(best, top.best * rinv, top.bi);
          if (top.si >= 0) tri_offer(best, top.second * rinv, top.si);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_a_empty + 8 * buf);
        continue;
      }
      // ---- Fold the four groups' results of each row and publish the chunk's: by the warp that is the last to be done.  The
      // others leave theirs, in the order in which they come, and go on; they can be one item ahead at most: the item after
      // that is not gathered before this one is folded.  (With the first group folding, it stood until the others were done, and
      // the products before its accumulator.)
      uint32_t *x = xchg + (size_t)(buf * kPairM + row) * 9;
      int order = 0;
      if (lane == 0) order = atomicAdd(&s_done[buf][quarter], 1);
      order = __shfl_sync(0xffffffffu, order, 0);
      if (order < kPairAcc - 1) {   // slots are below 65535 (N_cap <= 49152); -1 = none
        uint32_t *xw = x + order * 3;
        xw[0] = __float_as_uint(top.best);
        xw[1] = __float_as_uint(top.second);
        xw[2] = (uint32_t)(top.bi + 1) | ((uint32_t)(top.si + 1) << 16);
        __syncwarp();
        if (lane == 0) mbar_arrive(xbar + 8 * buf);
      } else {
        if (!__all_sync(0xffffffffu, !s_abort && mbar_wait_n(xbar + 8 * buf, (x_phase >> buf) & 1, spin_limit))) { s_abort = 1; break; }
        if (lane == 0) s_done[buf][quarter] = 0;
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
    if (kTri) offer_told();
  }

  // ---------------------------------------------------------------- teardown
  tc_fence_before();
  __syncthreads();
  if (s_abort) {
    if (tid == 0) {
      atomicOr(status_dev, KEEPKV_DEV_TIMEOUT);
      // copies still in flight get a bounded chance to land before the shared memory goes away
      for (int i = 0; i < kStages; ++i) { mbar_wait_n(bar_b_full + 8 * i, 0, spin_limit); mbar_wait_n(bar_b_full + 8 * i, 1, spin_limit); }
    }
    __syncthreads();
  }
  cluster_sync_all();   // neither CTA's shared memory goes away before the other has arrived at its barriers and read its operands
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(CtaPair{}, tmem, 512);
  }
}

template <bool kTri>
static void launch_pairs_t(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst, const int32_t *ev_idx,
                           const UnitInfo *unit_info, const float *inv_norm, const uint4 *norm_ext, int32_t *sched, uint4 *nom,
                           int nom_chunks, int32_t *status_dev, LaunchCtx &ctx, unsigned long long *tri_best) {
  using SL = PairSmem;
  constexpr size_t smem_bytes = (size_t)SL::kBytes + 1024;
  static bool attr_done_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_done_dev[dev & 63]) {
    cudaFuncSetAttribute(nominate_pair_kernel<kTri>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes);
    attr_done_dev[dev & 63] = true;
  }
  CUtensorMap mapB;
  if (!make_bf16_tiles_map(&mapB, dst.K, (uint64_t)p.B * p.H_kv * p.N_cap, kPairD, kPairHalf)) {
    if (ctx.err == cudaSuccess) ctx.err = cudaErrorInvalidValue;
    return;
  }
  launch_pdl_cluster(nominate_pair_kernel<kTri>, dim3(sm_count() & ~1), dim3(kPairThreads), smem_bytes, ctx.stream, 2u, mapB, p,
                     reinterpret_cast<const __nv_bfloat16 *>(src.K), ev_idx, unit_info, inv_norm, norm_ext, sched, nom, nom_chunks,
                     status_dev, tri_best, debug_spin_limit(), debug_withhold());
  KEEPKV_CHECK_LAUNCH(ctx);
}

void launch_nominate_pairs(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst, const int32_t *ev_idx,
                           const UnitInfo *unit_info, const float *inv_norm, const uint4 *norm_ext, int32_t *sched, uint4 *nom,
                           int nom_chunks, int32_t *status_dev, LaunchCtx &ctx, unsigned long long *tri_best) {
  (tri_best ? launch_pairs_t<true> : launch_pairs_t<false>)(p, src, dst, ev_idx, unit_info, inv_norm, norm_ext, sched, nom, nom_chunks,
                                                            status_dev, ctx, tri_best);
}

}  // namespace keepkv
