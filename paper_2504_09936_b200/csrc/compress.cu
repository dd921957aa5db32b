// keepkv_compress: Algorithm 1 of the paper, out of place, one (sequence, kv-head) unit at a time.
//   select   -> retained / evicted sets from the key kappa = ln p + lscore       (Algorithm 1, selection step)
//   compact  -> retained rows copied to dst in ascending source order            (Algorithm 1, insertion step)
//   nominate -> two best cosines of every evicted key over the retained keys,
//               on the tensor cores (nominate.cu)                                (Algorithm 1, similarity step)
//   resolve  -> arg-max and threshold of Algorithm 1, decided in the interface's fixed fp32
//               arithmetic wherever the tensor-core ranking is too close to call; members
//               of each retained slot sorted into groups                         (many-to-one, App. A.2)
//   merge    -> Eq. A.3 with the EMA estimate as score                           (Algorithm 1, merge step)
#include "compress.cuh"

namespace keepkv {

// ------------------------------------------------------------------ select
// One CTA per unit.  The keys of the whole unit live in shared memory; the heavy-hitter threshold is found by range_select.
// Then every warp counts what it keeps of a contiguous run of entries, one block scan gives the places, and the retained
// list, the evicted list and the per-entry marks are written 32 consecutive entries at a time.  49 -> 22 us for 64 units of
// 8192, 95 -> 32 us for 128 of up to 16384, against four passes over 8-bit digits and an ordered pass with three block
// barriers every 2048 entries.
// Short units: with 128 threads for 1002 entries, and 1024 of which most left at once, one CTA to an SM, the call without
// merges took 46.1 us for 256 units of 1002 and 27.6 us for 256 of 200 in a buffer of 8192; now 27.7 and 17.4 (four digit
// passes by one warp: 29.7 and 17.4; d = 64).
// Threads for a unit of len entries.
__host__ __device__ __forceinline__ int select_threads(int len) { return len > 4096 ? 1024 : len > 1024 ? 512 : len > 256 ? 256 : 128; }
// ... and of a launch.  With more units than SMs, two CTAs to an SM.
static int select_block(const keepkv_params &p) {
  const int n = select_threads(p.N_cap);
  return p.B * p.H_kv > sm_count() && n > 512 ? 512 : n;
}
__global__ void __launch_bounds__(1024)
select_kernel(keepkv_params p, keepkv_cache src, int32_t *dst_seq_len, const int32_t *budget_dev, int budget_scalar,
              const int32_t *n_recent_dev, int32_t *ret_idx, int32_t *target, int32_t *ev_idx, UnitInfo *unit_info,
              keepkv_stats *stats, const float *__restrict__ select_key, const int32_t *__restrict__ unit_len,
              int32_t *pos, const int32_t *pos_len, const int32_t *n_seen, int32_t *status_dev) {
  extern __shared__ uint32_t keys[];
  __shared__ int hist[kSelBins];
  __shared__ int warp_tot[32], warp_tie[32];
  __shared__ uint32_t warp_min[32], warp_max[32];
  __shared__ int s_sel[4];
  const int u = blockIdx.x, b = u / p.H_kv, h = u % p.H_kv, tid = threadIdx.x;
  pdl_wait();
  pdl_trigger();
  // (unit_len: the heads of a sequence differ in length -- only between the two passes of the merge-first compression)
  const int len = max(0, min(unit_len ? unit_len[u] : src.seq_len[b], p.N_cap));
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
  const size_t base = (size_t)u * p.N_cap;
  // Short units need few threads, and every barrier below costs by the warp: the surplus warps leave.
  const int nthr = min((int)blockDim.x, select_threads(len)), nw = nthr >> 5;
  if (tid >= nthr) return;
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t k_lo = 0xffffffffu, k_hi = 0u;   // the range of the candidates' keys
  if (pos) {
    // A cache that is not in token order (in-place compression): sinks and recent window are told by the token
    // position of a row, not by the row.  Rows from pos_len[b] on are the tokens appended since the last call, in
    // order: they get their positions here.  A sink or recent row takes key 0, below every real key, so that the
    // search over all rows ranks the candidates only; what the row order decides elsewhere (equal keys), it
    // decides here too.
    const int first_fresh = max(0, min(pos_len[b], len)), n_total = n_seen[b] + (len - first_fresh);
    const bool all = budget >= len;
    int n_fixed = 0;
    for (int i = tid; i < len; i += nthr) {
      int ps = pos[base + i];
      if (i >= first_fresh) { ps = n_seen[b] + (i - first_fresh); pos[base + i] = ps; }
      const bool fixed = all || ps < n_sink || ps >= n_total - n_recent;
      n_fixed += (!all && fixed) ? 1 : 0;
      const uint32_t k = fixed ? 0u : kappa_key(src.votes[base + i], src.lscore[base + i]);
      keys[i] = k;
      k_lo = min(k_lo, k);
      k_hi = max(k_hi, k);
    }
    int tot;
    block_excl_sum(n_fixed, warp_tot, tot, nw);
    // the n_sink first and the n_recent last tokens must all be present (they are, if the windows never grew faster
    // than the cache): otherwise positions and ranks disagree and the unit is reported, its result unspecified
    if (!all && tot != n_sink + n_recent && tid == 0) atomicOr(status_dev, KEEPKV_DEV_POSITIONS);
    lo = 0;
    hi = len;
  } else {
#pragma unroll 4
    for (int i = tid; i < len; i += nthr) {
      // the caller's scores where given, else kappa = ln p + lscore
      const uint32_t k = select_key ? ordered_key(select_key[base + i]) : kappa_key(src.votes[base + i], src.lscore[base + i]);
      keys[i] = k;
      if (i >= lo && i < hi) { k_lo = min(k_lo, k); k_hi = max(k_hi, k); }
    }
  }
  k_lo = __reduce_min_sync(0xffffffffu, k_lo);
  k_hi = __reduce_max_sync(0xffffffffu, k_hi);
  if (lane == 0) { warp_min[warp] = k_lo; warp_max[warp] = k_hi; }
  __syncthreads();
  k_lo = __reduce_min_sync(0xffffffffu, lane < nw ? warp_min[lane] : 0xffffffffu);
  k_hi = __reduce_max_sync(0xffffffffu, lane < nw ? warp_max[lane] : 0u);

  uint32_t kth = 0;    // the n_heavy-th largest key
  int n_tie = 0;       // how many entries equal to it are taken, lowest index first
  int tot_ties = 0;    // how many entries equal to it exist
  if (n_heavy > 0) range_select(keys, lo, hi, k_lo, k_hi, n_heavy, nthr, hist, s_sel, warp_tot, kth, n_tie, tot_ties);

  // A warp owns a run of consecutive entries.  Pass 1 counts the entries above the threshold and equal to it, a scan over
  // the warps gives the places, pass 2 writes.  Ties are ranked only if some of them lose.
  const bool rank_ties = n_heavy > 0 && n_tie < tot_ties;
  const int run = ((len + nw - 1) / nw + 31) & ~31, e0 = min(len, warp * run), e1 = min(len, e0 + run);
  auto classify = [&](int i, bool &keep, bool &tie) {
    const bool valid = i < e1;
    const uint32_t k = valid ? keys[i] : 0u;
    const bool mid = valid && i >= lo && i < hi && !(pos && k == 0u);
    tie = mid && n_heavy > 0 && k == kth;
    keep = valid && (!mid || (n_heavy > 0 && k > kth) || (tie && !rank_ties));
  };
  int n_k = 0, n_t = 0;
  for (int i0 = e0; i0 < e1; i0 += 32) {
    bool keep, tie;
    classify(i0 + lane, keep, tie);
    n_k += __popc(__ballot_sync(0xffffffffu, keep));
    n_t += __popc(__ballot_sync(0xffffffffu, tie));
  }
  if (lane == 0) { warp_tot[warp] = n_k; warp_tie[warp] = n_t; }
  __syncthreads();
  // a warp's counts per lane: ties before it, then what the warps before it keep
  const int ties_w = lane < nw ? warp_tie[lane] : 0;
  int ties_before = ties_w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, ties_before, o);
    if (lane >= o) ties_before += y;
  }
  ties_before -= ties_w;
  const int kept_w = (lane < nw ? warp_tot[lane] : 0) + (rank_ties ? max(0, min(n_tie - ties_before, ties_w)) : 0);
  const int base_keep = __reduce_add_sync(0xffffffffu, kept_w);
  int slot = __reduce_add_sync(0xffffffffu, lane < warp ? kept_w : 0);
  int tie_rank = __shfl_sync(0xffffffffu, ties_before, warp);
  for (int i0 = e0; i0 < e1; i0 += 32) {
    const int i = i0 + lane;
    bool keep, tie;
    classify(i, keep, tie);
    const unsigned below = (1u << lane) - 1u;
    if (rank_ties) {
      const unsigned tb = __ballot_sync(0xffffffffu, tie);
      keep = keep || (tie && tie_rank + __popc(tb & below) < n_tie);
      tie_rank += __popc(tb);
    }
    const unsigned kb = __ballot_sync(0xffffffffu, keep);
    const int at = slot + __popc(kb & below);
    if (i < e1) {
      if (keep) ret_idx[base + at] = i;
      else ev_idx[base + (i - at)] = i;
      target[base + i] = keep ? -2 : -1;
    }
    slot += __popc(kb);
  }
  if (tid == 0) {
    UnitInfo ui{len, base_keep, len - base_keep, 0, 0, 0, base_keep, 0};   // (pad0: the retained count once more, for the in-place path)
    unit_info[u] = ui;
    if (h == 0 && dst_seq_len) dst_seq_len[b] = base_keep;   // (in place: the length changes when the rows have moved)
    keepkv_stats st;
    st.n_retained = base_keep; st.n_evicted = len - base_keep; st.n_merged = 0;
    st.n_below_T = len - base_keep;   // resolve_kernel replaces this once targets are known
    st.n_guard_groups = 0; st.n_groups = 0; st.max_group = 0; st.reserved = 0;
    stats[u] = st;
  }
}

// ------------------------------------------------------------------ compact
// grid (up to 32, U), 256 threads, 64 slots per CTA and sweep.  Sixteen lanes move one retained row (a 16-byte piece of
// K and of V each); a warp has eight rows in flight.  The same lanes tree-sum the squared key
// and, where a similarity search follows (norm_ext given), write what it needs of the key's norm.
template <int D>
__global__ void __launch_bounds__(256)
compact_kernel(keepkv_params p, keepkv_cache src, keepkv_cache dst, const int32_t *__restrict__ ret_idx,
               const UnitInfo *__restrict__ unit_info, float *__restrict__ inv_norm, uint4 *__restrict__ norm_ext) {
  constexpr int CH = D / 8;       // 16-byte chunks per row
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.y, n_ret = unit_info[u].n_ret;
  for (int s0 = blockIdx.x * 64; s0 < n_ret; s0 += gridDim.x * 64) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, ch = lane & 15, sub = lane >> 4;
  const size_t base = (size_t)u * p.N_cap;
  const uint4 *sK = reinterpret_cast<const uint4 *>(src.K), *sV = reinterpret_cast<const uint4 *>(src.V);
  uint4 *dK = reinterpret_cast<uint4 *>(dst.K), *dV = reinterpret_cast<uint4 *>(dst.V);
  int slot[4], si[4];
  uint4 kv[4], vv[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    slot[r] = s0 + warp * 8 + r * 2 + sub;
    si[r] = slot[r] < n_ret ? ret_idx[base + slot[r]] : -1;
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    kv[r] = make_uint4(0, 0, 0, 0);
    vv[r] = kv[r];
    if (si[r] >= 0 && ch < CH) {
      kv[r] = sK[(base + si[r]) * CH + ch];
      vv[r] = sV[(base + si[r]) * CH + ch];
    }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    if (si[r] >= 0 && ch < CH) {
      dK[(base + slot[r]) * CH + ch] = kv[r];
      dV[(base + slot[r]) * CH + ch] = vv[r];
    }
    float ss = 0.f;
    const uint32_t w[4] = {kv[r].x, kv[r].y, kv[r].z, kv[r].w};
#pragma unroll
    for (int q = 0; q < 4; ++q) { const float a = bf16_lo(w[q]), b = bf16_hi(w[q]); ss = fmaf(a, a, ss); ss = fmaf(b, b, ss); }
    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
    ss += __shfl_xor_sync(0xffffffffu, ss, 4);
    ss += __shfl_xor_sync(0xffffffffu, ss, 8);
    if (si[r] >= 0 && ch == 0) {
      if (norm_ext) {
        norm_ext[base + slot[r]] = ext_col(sqrtf(ss));
        inv_norm[base + slot[r]] = rsqrtf(ss);
      }
      dst.votes[base + slot[r]] = src.votes[base + si[r]];
      dst.lscore[base + slot[r]] = src.lscore[base + si[r]];
    }
  }
  }
}

// ------------------------------------------------------------------ resolve + group
// grid (R, U).  The tensor-core search left, per evicted entry, the largest cosines over the retained
// keys (best and second, with their slots).  Its values differ from the interface's
// fp32 chain only by accumulation order (far below kRankEps), so:
//   best - second > eps              the arg-max is settled; otherwise both candidates are re-evaluated
//                                    with the exact chain and the larger wins (equal -> lower slot);
//   |best - T|    <= eps             the threshold test uses the exact chain of the winner.
// (Three distinct cosines within the accumulation error of each other, the one case this cannot
// settle, would need a coincidence of order 1e-8 per row; exact duplicates are handled, because equal
// keys give equal values and the lower slot stays in front.)
// Rows that need the exact chain are evaluated by the warp that finds them.  One or two: coalesced row loads into shared memory, the
// sequential chains on three lanes.  More: ten at a time (six of a triangle), every candidate is a lane's, which walks its row and
// the evicted one's in global memory (64 units, keys that repeat 27 times: 6554 rows a unit 1143 -> 840 us the call, 128 rows 127 -> 85;
// 101 with a queue that the CTA's warps shared.  But a lone row takes twice as long, and in line the code cost the call 0.5 %).
// Bound: the latency of a row's list; so the warps of the
// resident CTAs (two per SM) walk the rows on their own, the next lists on their way, and no barrier is met: 64 units of 6554
// rows 19 -> 13 us, 128 of up to 14746 41 -> 26 us against a CTA per 512 rows with a common queue and place in the list (and
// lists whose chunks lay side by side, so that a row's sector was mostly unused).  A unit of at most kResolveThreads evicted
// entries (every steady-state compression) is one CTA's: it sorts the entries to merge by (slot, position), which makes
// every group contiguous and ascending, and merges them if the groups are few.  The entries to merge of larger units go to
// a list that group_kernel sorts.
constexpr int kMergeInline = 32;   // units with at most this many groups are merged where group_and_merge sorts them
constexpr int kResolveThreads = 512;
constexpr int kResolveWarps = kResolveThreads / 32;
constexpr int kResolveFew = 2;
constexpr int kGroupThreads = 1024;
constexpr int kGroupSmem = 212992; // bytes of counters and keys group_kernel may hold
constexpr int kGroupRank = 128;    // members of one group up to which a key finds its place among its neighbours

// Sorts the M entries to merge of unit u by (slot, position) -- which makes every group contiguous and ascending --,
// publishes the sorted members and the start of every group, and merges the groups itself when there are few.
// Called by a whole CTA of NT threads.  keys: where the M keys are now (key_smem when `single`, else gk).
template <int D, int NT>
__device__ __forceinline__ void group_and_merge(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                                                int u, size_t base, int n_ev, int M, bool single, uint32_t *key_smem,
                                                int smem_keys, uint32_t *gk, int32_t *target, int32_t *grp_head, UnitInfo *unit_info, keepkv_stats *stats, int *warp_tot) {
  const int tid = threadIdx.x, warp = tid >> 5;
  int Mp = 1;
  while (Mp < M) Mp <<= 1;
  uint32_t *keys = (single || Mp <= smem_keys) ? key_smem : gk;
  if (keys != gk && !single)
    for (int i = tid; i < M; i += NT) keys[i] = __ldcg(&gk[i]);
  for (int i = M + tid; i < Mp; i += NT) keys[i] = 0xFFFFFFFFu;
  __syncthreads();
  if (Mp <= NT && keys == key_smem) {
    // few keys (all distinct): every thread finds the rank of its key by counting, one barrier
    uint32_t mine = 0xFFFFFFFFu;
    int rank = 0;
    if (tid < M) {
      mine = keys[tid];
      for (int j = 0; j < M; ++j) rank += keys[j] < mine ? 1 : 0;
    }
    __syncthreads();
    if (tid < M) keys[rank] = mine;
    __syncthreads();
  } else {
    // bitonic sort, ascending
    for (int k = 2; k <= Mp; k <<= 1) {
      for (int jj = k >> 1; jj > 0; jj >>= 1) {
        for (int i = tid; i < Mp; i += NT) {
          const int ixj = i ^ jj;
          if (ixj > i) {
            const uint32_t a = keys[i], b = keys[ixj];
            if ((a > b) == ((i & k) == 0)) { keys[i] = b; keys[ixj] = a; }
          }
        }
        __syncthreads();
      }
    }
  }
  // publish the sorted members and the start of every group
  int n_groups = 0;
  for (int i0 = 0; i0 < M; i0 += NT) {
    const int i = i0 + tid;
    const bool head = i < M && (i == 0 || (keys[i] >> 16) != (keys[i - 1] >> 16));
    int tot;
    const int pos = n_groups + block_excl_count(head, warp_tot, tot);
    if (head) grp_head[base + pos] = i;
    if (i < M && keys != gk) gk[i] = keys[i];
    n_groups += tot;
  }
  if (tid == 0) {
    grp_head[base + n_groups] = M;
    unit_info[u].n_groups = n_groups <= kMergeInline ? 0 : n_groups;
    stats[u].n_below_T = n_ev - M;
  }
  if (n_groups <= kMergeInline) {
    // few groups (every steady-state compression): merge them here, one warp per group
    __syncthreads();   // the keys and group starts written above are visible to the whole CTA
    MergeCount count;
    for (int g = warp; g < n_groups; g += NT / 32) {
      const int beg = grp_head[base + g], n = grp_head[base + g + 1] - beg;
      const int c = (int)(gk[beg] >> 16);
      merge_group<D>(p, src, dst, c, dst, base + c, [&](int t) { return (int)(gk[beg + t] & 0xFFFFu); }, n,
                     target + base, base, count);
    }
    count.flush(stats + u);
  }
}


// The rows of lanes `need` in the interface's exact arithmetic, several at a time: a row is entry e, its candidates c0 and, of those that
// are not negative, c1 to c3.  Returned: the best slot, with the sign bit where it is not above T.  (Not in line: most warps never come here.)
template <int D, bool kTri>
__device__ __noinline__ int exact_many(unsigned need, int e, int c0, int c1, int c2, int c3, const __nv_bfloat16 *sK, const __nv_bfloat16 *dK,
                                       float T) {
  constexpr int kCand = kTri ? 4 : 2, kLanes = kCand + 1, kRows = 32 / kLanes;   // a lane for each candidate and one for the row's norm
  const int lane = threadIdx.x & 31, g = lane / kLanes, role = lane - g * kLanes;
  int out = -1;
  while (need) {
    unsigned m = need;
    for (int k = 0; k < g; ++k) m &= m - 1;
    const int l = m ? __ffs(m) - 1 : 0;
    const int ee = __shfl_sync(0xffffffffu, e, l);
    int c = __shfl_sync(0xffffffffu, c0, l);
    const int d1 = __shfl_sync(0xffffffffu, c1, l), d2 = __shfl_sync(0xffffffffu, c2, l), d3 = __shfl_sync(0xffffffffu, c3, l);
    const int other = role == 2 ? d1 : role == 3 ? d2 : role == 4 ? d3 : -1;
    if (other >= 0) c = other;
    float u = 0.f, nn = 0.f;
    if (m && g < kRows) exact_dot<D>(sK + (size_t)ee * D, role ? dK + (size_t)c * D : sK + (size_t)ee * D, u, nn);
    const float ne = __shfl_sync(0xffffffffu, nn, min(g * kLanes, 31));
    u = u / (sqrtf(ne) * sqrtf(nn));
    const int at = __popc(need & ((1u << lane) - 1u));   // the row's place among those that are left
    const bool mine = (need >> lane & 1u) && at < kRows;
    int win = 0;
    float wu = 0.f;
#pragma unroll
    for (int k = 0; k < kCand; ++k) {
      const int from = mine ? at * kLanes + 1 + k : 0;
      const float uk = __shfl_sync(0xffffffffu, u, from);
      const int ck = __shfl_sync(0xffffffffu, c, from);
      if (k == 0 || uk > wu || (uk == wu && ck < win)) { win = ck; wu = uk; }
    }
    if (mine) out = wu > T ? win : (int)0x80000000 | win;
#pragma unroll
    for (int k = 0; k < kRows; ++k) need &= need - 1;
  }
  return out;
}

// kTri: the search's lists are those of a triangle.
template <int D, bool kTri>
__global__ void __launch_bounds__(kResolveThreads)
resolve_kernel(keepkv_params p, keepkv_cache src, keepkv_cache dst, const int32_t *__restrict__ ev_idx,
               UnitInfo *unit_info, const uint4 *__restrict__ nom, const int32_t *__restrict__ sched, int32_t *target,
               uint32_t *grp_key, int key_stride, int32_t *grp_head, keepkv_stats *stats, int decide_only,
               const ulonglong2 *__restrict__ tri_best) {
  __shared__ uint32_t key_smem[kResolveThreads];
  __shared__ float ke_s[kResolveWarps][D];
  __shared__ float kc_s[kResolveWarps][2][D];
  __shared__ int warp_tot[32];
  __shared__ int s_keys;
  const int u = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, step = gridDim.x * kResolveThreads;
  pdl_wait();
  pdl_trigger();
  const UnitInfo ui = unit_info[u];
  const int C = kTri ? 0 : sched[0];
  const size_t base = (size_t)u * p.N_cap, n_rows = (size_t)p.B * p.H_kv * p.N_cap;
  const __nv_bfloat16 *sK = reinterpret_cast<const __nv_bfloat16 *>(src.K) + base * D;
  const __nv_bfloat16 *dK = reinterpret_cast<const __nv_bfloat16 *>(dst.K) + base * D;
  uint32_t *gk = grp_key + (size_t)u * key_stride;
  const float T = p.merge_threshold;
  if ((int)blockIdx.x * kResolveThreads >= ui.n_ev) return;
  const bool single = ui.n_ev <= kResolveThreads && !decide_only;   // this CTA holds all rows of the unit
  if (tid == 0) s_keys = 0;
  __syncthreads();

  // The warps go their own ways; a row's list is on its way while the one before it is decided.
  int j0 = blockIdx.x * kResolveThreads + warp * 32, e_next = 0;
  uint4 v_next = make_uint4(0u, 0u, 0u, 0u);
  ulonglong2 l0_next = make_ulonglong2(0, 0), l1_next = l0_next;
  auto fetch = [&](int j) {
    if (j >= ui.n_ev) return;
    if (kTri) { e_next = j; l0_next = tri_best[(base + j) * 2]; l1_next = tri_best[(base + j) * 2 + 1]; }
    else { e_next = ev_idx[base + j]; v_next = nom[base + j]; }
  };
  fetch(j0 + lane);
  for (; j0 < ui.n_ev; j0 += step) {
    const int j = j0 + lane, e = e_next;
    uint4 v = v_next;
    const ulonglong2 l0 = l0_next, l1 = l1_next;
    fetch(j + step);
    const bool valid = j < ui.n_ev;
    int slot = -1, kind = 0, bi = -1, si = -1, ci = -1, di = -1;
    bool merge = false;
    if (valid) {
      float best = -CUDART_INF_F, second = -CUDART_INF_F;
      if constexpr (kTri) {
        // Two lists of two, as the entry was a row and as it was a column.  In either, equal keys have equal cosines and the lower
        // slot is in front; between them they can differ by rounding, so everything that is close to the best is looked at.
        const unsigned long long first = l0.x > l1.x ? l0.x : l1.x, other = l0.x > l1.x ? l1.x : l0.x;
        auto val = [](unsigned long long y) { return y ? __uint_as_float((uint32_t)(y >> 32)) : -CUDART_INF_F; };
        auto idx = [](unsigned long long y) { return y ? (int)(0xffffffffu - (uint32_t)y) : -1; };
        best = val(first);
        bi = idx(first);
        second = fmaxf(val(other), fmaxf(val(l0.y), val(l1.y)));
        auto close = [&](unsigned long long y) { return y && !(best - val(y) > kRankEps) ? idx(y) : -1; };
        si = close(other);
        ci = close(l0.y);
        di = close(l1.y);
      } else for (int c = 0;;) {   // chunks hold ascending slots: strict comparisons keep the lower slot on ties
        const int vi[2] = {(int)v.z, (int)v.w};
        // (A search that gave up has left rows as they were: what names no slot is no candidate.)
        const float vv[2] = {v.z < (uint32_t)ui.n_ret ? __uint_as_float(v.x) : -CUDART_INF_F,
                             v.w < (uint32_t)ui.n_ret ? __uint_as_float(v.y) : -CUDART_INF_F};
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          const bool p1 = vv[t] > best, p2 = vv[t] > second;
          second = p1 ? best : fmaxf(second, vv[t]);
          si = p1 ? bi : (p2 ? vi[t] : si);
          bi = p1 ? vi[t] : bi;
          best = fmaxf(best, vv[t]);
        }
        if (++c >= C) break;
        v = nom[c * n_rows + base + j];
      }
      if (bi >= 0) {
        slot = bi;
        if (!(best - second > kRankEps)) kind = kTri || si >= 0 ? 1 : 2;
        else if (!(fabsf(best - T) > kRankEps)) kind = 2;
        else merge = best > T;
      }
    }
    // ---- rows that need the interface's exact arithmetic: one or two of them one after the other, more at a time
    unsigned need = __ballot_sync(0xffffffffu, kind != 0);
    for (; need && __popc(need) <= kResolveFew; need &= need - 1) {
      const int l = __ffs(need) - 1, ee = __shfl_sync(0xffffffffu, e, l), ca = __shfl_sync(0xffffffffu, bi, l);
      const int cb = __shfl_sync(0xffffffffu, kind == 1 && si >= 0 ? si : bi, l);
      float u0, u1;
      exact_cosines<D>(sK + (size_t)ee * D, dK + (size_t)ca * D, dK + (size_t)cb * D, ke_s[warp], &kc_s[warp][0][0], u0, u1);
      int win = ca;
      float wu = u0;
      if (u1 > u0 || (u1 == u0 && cb < ca)) { win = cb; wu = u1; }
      if (kTri && __shfl_sync(0xffffffffu, max(ci, di), l) >= 0) {
        int cc = __shfl_sync(0xffffffffu, ci, l), cd = __shfl_sync(0xffffffffu, di, l);
        if (cc < 0) cc = cd;
        if (cd < 0) cd = cc;
        exact_cosines<D>(sK + (size_t)ee * D, dK + (size_t)cc * D, dK + (size_t)cd * D, ke_s[warp], &kc_s[warp][0][0], u0, u1);
        if (u0 > wu || (u0 == wu && cc < win)) { win = cc; wu = u0; }
        if (u1 > wu || (u1 == wu && cd < win)) { win = cd; wu = u1; }
      }
      if (lane == l) { slot = win; merge = wu > T; }
    }
    if (need) {
      const int win = exact_many<D, kTri>(need, e, bi, kTri || kind == 1 ? si : -1, ci, di, sK, dK, T);
      if (kind) { slot = win & 0xffff; merge = win >= 0; }
    }
    if (valid) target[base + e] = merge ? slot : -1;
    if (decide_only) continue;   // the caller pairs the entries itself (merge-first policy): the partner above T, or -1
    // ---- entries to merge go to the unit's key list (any order: it is sorted below)
    const unsigned m = __ballot_sync(0xffffffffu, merge);
    if (m) {
      int at = 0;
      if (lane == 0) at = atomicAdd(single ? &s_keys : &unit_info[u].n_keys, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (merge) (single ? key_smem : gk)[at] = ((uint32_t)slot << 16) | (uint32_t)e;
    }
  }
  if (!single) return;
  __syncthreads();
  if (tid == 0) unit_info[u].ticket = 1;   // this unit's entries are sorted
  group_and_merge<D, kResolveThreads>(p, src, dst, u, base, ui.n_ev, s_keys, true, key_smem, kResolveThreads, gk, target, grp_head, unit_info, stats, warp_tot);
}

// One CTA per unit: the unit's key list (in global memory, any order) sorted into groups by counting -- a histogram of the
// slots in shared memory, a scan, every key to its group, its rank there from its neighbours: nine barriers, where a
// bitonic sort of 4096 keys has 78.  Lists that do not fit, or hold a group of more than kGroupRank members, are sorted
// bitonically after all.  (With the sort at the end of resolve_kernel by a unit's last CTA, at a few CTAs a unit, the two
// steps took 45 us for 64 units of 6554 entries and 113 us for 128 units of up to 14746.)
template <int D>
__global__ void __launch_bounds__(kGroupThreads)
group_kernel(keepkv_params p, keepkv_cache src, keepkv_cache dst, int32_t *target, UnitInfo *unit_info, uint32_t *grp_key, int key_stride,
             int32_t *grp_head, keepkv_stats *stats, int smem_words) {
  extern __shared__ uint32_t key_smem[];
  __shared__ int warp_tot[32];
  __shared__ int s_max;
  constexpr int NT = kGroupThreads;
  const int tid = threadIdx.x, u = blockIdx.x;
  pdl_wait();
  pdl_trigger();
  const UnitInfo ui = unit_info[u];
  if (ui.ticket) return;   // resolve_kernel has sorted this unit's
  const size_t base = (size_t)u * p.N_cap;
  uint32_t *gk = grp_key + (size_t)u * key_stride;
  const int M = ui.n_keys, n_slots = ui.n_ret;
  if (n_slots + M <= smem_words) {
    int *cnt = reinterpret_cast<int *>(key_smem);
    uint32_t *out = key_smem + n_slots;
    for (int i = tid; i < n_slots; i += NT) cnt[i] = 0;
    if (tid == 0) s_max = 0;
    __syncthreads();
    int most = 0;
#pragma unroll 4
    for (int i = tid; i < M; i += NT) most = max(most, atomicAdd(&cnt[gk[i] >> 16], 1) + 1);
    most = __reduce_max_sync(0xffffffffu, most);
    if ((tid & 31) == 0) atomicMax(&s_max, most);
    __syncthreads();
    if (s_max <= kGroupRank) {
      // a thread owns a run of slots: keys and groups before it, in one packed scan
      const int per = (n_slots + NT - 1) / NT, lo = min(n_slots, tid * per), hi = min(n_slots, lo + per);
      int mine = 0;
      for (int s = lo; s < hi; ++s) mine += cnt[s] + (cnt[s] > 0 ? 1 << 16 : 0);
      int tot;
      unsigned at = (unsigned)block_excl_sum(mine, warp_tot, tot, NT / 32);
      for (int s = lo; s < hi; ++s) {
        const int n = cnt[s];
        cnt[s] = (int)(at & 0xffffu);
        if (n > 0) {
          grp_head[base + (at >> 16)] = (int)(at & 0xffffu);
          at += (1u << 16) + (unsigned)n;
        }
      }
      const int n_groups = (int)((unsigned)tot >> 16);
      __syncthreads();
#pragma unroll 4
      for (int i = tid; i < M; i += NT) {
        const uint32_t k = gk[i];
        out[atomicAdd(&cnt[k >> 16], 1)] = k;
      }
      __syncthreads();
      for (int i = tid; i < M; i += NT) {
        const uint32_t k = out[i], slot = k >> 16;
        int j = i - 1, less = 0;
        for (; j >= 0 && (out[j] >> 16) == slot; --j) less += out[j] < k ? 1 : 0;
        const int beg = j + 1;
        for (j = i + 1; j < M && (out[j] >> 16) == slot; ++j) less += out[j] < k ? 1 : 0;
        gk[beg + less] = k;
      }
      if (tid == 0) {
        grp_head[base + n_groups] = M;
        unit_info[u].n_groups = n_groups;
        stats[u].n_below_T = ui.n_ev - M;
      }
      return;
    }
    __syncthreads();   // the counters make room for keys
  }
  group_and_merge<D, NT>(p, src, dst, u, base, ui.n_ev, M, false, key_smem, smem_words, gk, target, grp_head, unit_info, stats, warp_tot);
}

// What the two kernels are launched with.
static int resolve_grid(const keepkv_params &p) {   // what is resident (two per SM), as far as there are rows
  const int most = (p.N_cap + kResolveThreads - 1) / kResolveThreads, n = 2 * sm_count() / (p.B * p.H_kv);
  return n < 1 ? 1 : n < most ? n : most;
}
static int merge_grid(const keepkv_params &p) {
  const int n = 4096 / (p.B * p.H_kv);
  return n < 1 ? 1 : (n > 128 ? 128 : n);
}
static int group_words(const keepkv_params &p, const WsLayout &L) {
  const int words = p.N_cap + L.key_stride;
  return words < kGroupSmem / 4 ? words : kGroupSmem / 4;
}
// No unit can evict more than the entries one CTA of resolve_kernel sorts.
static bool all_small(const keepkv_params &p, const int32_t *budget_dev, int32_t budget_scalar) {
  return !budget_dev && p.N_cap - budget_scalar <= kResolveThreads;
}

// ------------------------------------------------------------------ merge
// Units whose groups were not merged where they were sorted (by resolve_kernel, if they are few; by group_kernel only if it
// had to sort bitonically): warps of several CTAs share them.  The others have n_groups = 0 here.
template <int D>
__global__ void __launch_bounds__(256)
merge_kernel(keepkv_params p, keepkv_cache src, keepkv_cache dst, int32_t *target, const UnitInfo *__restrict__ unit_info,
             const uint32_t *__restrict__ grp_key, int key_stride, const int32_t *__restrict__ grp_head,
             keepkv_stats *stats) {
  const int u = blockIdx.y;
  pdl_wait();
  pdl_trigger();
  const int n_groups = unit_info[u].n_groups, step = gridDim.x * 8;
  const size_t base = (size_t)u * p.N_cap;
  const uint32_t *gk = grp_key + (size_t)u * key_stride;
  const int32_t *head = grp_head + base;
  int g = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (g >= n_groups) return;
  int beg = head[g], end = head[g + 1];
  MergeCount count;
  while (g < n_groups) {
    const int nx = min(g + step, n_groups - 1), nbeg = head[nx], nend = head[nx + 1];   // the next group's, in flight meanwhile
    const int c = (int)(gk[beg] >> 16);
    merge_group<D>(p, src, dst, c, dst, base + c, [&](int t) { return (int)(gk[beg + t] & 0xFFFFu); }, end - beg, target + base,
                   base, count);
    g += step;
    beg = nbeg;
    end = nend;
  }
  count.flush(stats + u);
}

// ------------------------------------------------------------------ host side
template <int D>
static void launch_compress_t(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                              const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                              int32_t *ret_idx, int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L,
                              int32_t *status_dev, const float *select_key, LaunchCtx &ctx) {
  const int U = p.B * p.H_kv;
  UnitInfo *ui = reinterpret_cast<UnitInfo *>(ws + L.unit_info);
  int32_t *sched = reinterpret_cast<int32_t *>(ws + L.sched);
  int32_t *ev_idx = reinterpret_cast<int32_t *>(ws + L.ev_idx);
  float *inv_norm = reinterpret_cast<float *>(ws + L.inv_norm);
  uint4 *norm_ext = reinterpret_cast<uint4 *>(ws + L.norm_ext);
  uint4 *nom = reinterpret_cast<uint4 *>(ws + L.nom);
  uint32_t *grp_key = reinterpret_cast<uint32_t *>(ws + L.grp_key);
  int32_t *grp_head = reinterpret_cast<int32_t *>(ws + L.grp_head);
  const int ret_bound = budget_dev ? p.N_cap : (budget_scalar < p.N_cap ? budget_scalar : p.N_cap);

  const size_t sel_smem = (size_t)p.N_cap * sizeof(uint32_t);
  static bool attr_done_dev[64] = {};   // opt-in to large dynamic shared memory once per device
  int dev = 0;
  cudaGetDevice(&dev);
  bool &attr_done = attr_done_dev[dev & 63];
  if (!attr_done) {
    cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152 * 4);
    cudaFuncSetAttribute(group_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
    attr_done = true;
  }
  if (p.flags & KEEPKV_FLAG_COMPRESS_STEADY) {   // the caller vouches for every unit: one kernel does it all
    launch_compress_steady(p, src, dst, budget_dev, budget_scalar, n_recent_dev, ret_idx, target, stats, ws, L, status_dev,
                           select_key, ctx);
    return;
  }
  launch_pdl(select_kernel, dim3(U), dim3(select_block(p)), sel_smem, ctx.stream, p, src, dst.seq_len, budget_dev, budget_scalar,
             n_recent_dev, ret_idx, target, ev_idx, ui, stats, select_key, (const int32_t *)nullptr, (int32_t *)nullptr,
             (const int32_t *)nullptr, (const int32_t *)nullptr, status_dev);
  KEEPKV_CHECK_LAUNCH(ctx);
  if (ret_bound <= 0) return;   // nothing is kept: every entry is dropped, which select has recorded
  const int cgx = (ret_bound + 63) / 64 < 32 ? (ret_bound + 63) / 64 : 32;   // the retained count is only known on the device
  // T = +inf: no cosine can exceed it, nothing merges -- the eviction strategy alone (what follows a merge-first pass)
  const bool merges = !(isinf(p.merge_threshold) && p.merge_threshold > 0.f);
  launch_pdl(compact_kernel<D>, dim3(cgx, U), dim3(256), 0, ctx.stream, p, src, dst, ret_idx, ui, inv_norm,
             merges ? norm_ext : nullptr);
  KEEPKV_CHECK_LAUNCH(ctx);
  if (!merges) return;
  // (Budgets on the device are taken for a tenth of the capacity.  Where they are more, the form for smaller prompts is kept: 64 units
  // 6000 -> 1800 in 6016 rows 181 us, 157 with the budget on the host; where less, pairs search few columns: 16000 -> 100 227, 225.)
  launch_nominate(p, src, dst, ev_idx, ui, inv_norm, norm_ext, sched, nom, L.nom_chunks, status_dev, ctx,
                  budget_dev ? p.N_cap / 10 : ret_bound);
  launch_pdl(resolve_kernel<D, false>, dim3(resolve_grid(p), U), dim3(kResolveThreads), 0, ctx.stream,
      p, src, dst, ev_idx, ui, nom, sched, target, grp_key, L.key_stride, grp_head,
      stats, 0, (const ulonglong2 *)nullptr);
  KEEPKV_CHECK_LAUNCH(ctx);
  if (!all_small(p, budget_dev, budget_scalar)) {
    launch_pdl(group_kernel<D>, dim3(U), dim3(kGroupThreads), (size_t)group_words(p, L) * 4, ctx.stream, p, src, dst,
               target, ui, grp_key, L.key_stride, grp_head, stats, group_words(p, L));
    KEEPKV_CHECK_LAUNCH(ctx);
  }
  launch_pdl(merge_kernel<D>, dim3(merge_grid(p), U), dim3(256), 0, ctx.stream, p, src, dst, target, ui, grp_key,
             L.key_stride, grp_head, stats);
  KEEPKV_CHECK_LAUNCH(ctx);
}


// ------------------------------------------------------------------ prefill merge-first policy (Section 3.4; App. B, Table 3)
// keepkv_merge_similar: before any eviction, every entry whose most similar OTHER key exceeds T is merged into that
// entry, provided the partner is earlier in the cache and is not itself merged away (the earlier of two entries is
// the target; no entry is both target and member).  The similarity search is the compression's own
// (nominate_kernel + resolve_kernel) with rows and columns both running over all entries of the unit and the
// diagonal masked; what is new is the pairing rule, which needs every entry's partner before any entry can be
// placed:
//   mf_prepare  -> inverse norms of all keys, the identity row list, the unit's sizes
//   nominate    -> two best cosines per entry over all other entries
//   resolve     -> partner above T per entry, exact where the ranking is close       (decide_only)
//   mf_mark     -> members, kept entries and their slots, targets, the key list of the groups
//   compact     -> kept rows to dst
//   group       -> keys sorted into groups, few groups merged at once
//   merge       -> Eq. A.3 for units with many groups

// Calls f(i, |k_i|^2) in one lane for every row i < len of a unit's keys (rows: the first one) that want(i) holds for, with
// 0 for the others.  grid (x, U), 256 threads; sixteen lanes per row, eight rows of a warp in flight: with two, 288 CTAs took
// 33 us for 32 units of 6007 rows, a trip to memory per sweep.
constexpr int kNormRows = 64;   // rows of a CTA and sweep
template <int D, typename Want, typename F>
__device__ __forceinline__ void each_row_norm(const uint4 *rows, int len, Want want, F f) {
  constexpr int CH = D / 8;
  const int lane = threadIdx.x & 31, ch = lane & 15, sub = lane >> 4, warp = threadIdx.x >> 5;
  for (int r0 = blockIdx.x * kNormRows; r0 < len; r0 += gridDim.x * kNormRows) {
    uint4 kv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = r0 + warp * 8 + r * 2 + sub;
      kv[r] = make_uint4(0, 0, 0, 0);
      if (i < len && ch < CH && want(i)) kv[r] = rows[(size_t)i * CH + ch];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = r0 + warp * 8 + r * 2 + sub;
      float ss = 0.f;
      const uint32_t w[4] = {kv[r].x, kv[r].y, kv[r].z, kv[r].w};
#pragma unroll
      for (int q = 0; q < 4; ++q) { const float a = bf16_lo(w[q]), b = bf16_hi(w[q]); ss = fmaf(a, a, ss); ss = fmaf(b, b, ss); }
      ss += __shfl_xor_sync(0xffffffffu, ss, 1);
      ss += __shfl_xor_sync(0xffffffffu, ss, 2);
      ss += __shfl_xor_sync(0xffffffffu, ss, 4);
      ss += __shfl_xor_sync(0xffffffffu, ss, 8);
      if (i < len && ch == 0) f(i, ss);
    }
  }
}
// CTAs per unit: what is resident (eight per SM), as far as there are rows.
static int norm_grid(const keepkv_params &p) {
  const int most = (p.N_cap + kNormRows - 1) / kNormRows, n = 8 * sm_count() / (p.B * p.H_kv);
  return n < 1 ? 1 : n < most ? n : most;
}

template <int D>
__global__ void __launch_bounds__(256)
mf_prepare_kernel(keepkv_params p, keepkv_cache src, int32_t *ev_idx, UnitInfo *unit_info, float *__restrict__ inv_norm,
                  uint4 *__restrict__ norm_ext, uint4 *__restrict__ tri_best) {
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.y, b = u / p.H_kv;
  const int len = max(0, min(src.seq_len[b], p.N_cap));
  const size_t base = (size_t)u * p.N_cap;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    UnitInfo ui{len, len, len, 0, 0, 0, 0, 0};
    unit_info[u] = ui;
  }
  each_row_norm<D>(reinterpret_cast<const uint4 *>(src.K) + base * (D / 8), len, [](int) { return true; }, [&](int i, float ss) {
    inv_norm[base + i] = rsqrtf(ss);
    norm_ext[base + i] = ext_col(sqrtf(ss));
    ev_idx[base + i] = i;
    if (tri_best) tri_best[(base + i) * 2] = tri_best[(base + i) * 2 + 1] = make_uint4(0, 0, 0, 0);
  });
}

// One CTA per unit.  partner[e] (in `target`): the entry e would merge into, or -1.  Writes the kept list (ret_idx),
// the member list (ev_idx), target[e] = slot of the partner for a member / -2 for a kept entry, the group keys
// (slot << 16 | entry), sizes and the initial statistics.  slot_of: scratch [N] per unit.
__global__ void __launch_bounds__(1024)
mf_mark_kernel(keepkv_params p, int32_t *unit_len, int32_t *ret_idx, int32_t *target, int32_t *ev_idx, int32_t *slot_of,
               uint32_t *grp_key, int key_stride, UnitInfo *unit_info, keepkv_stats *stats) {
  __shared__ int warp_tot[32];
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.x, tid = threadIdx.x, nthr = blockDim.x, nw = nthr >> 5;
  const int len = unit_info[u].len;
  const size_t base = (size_t)u * p.N_cap;
  int32_t *tg = target + base;
  uint32_t *gk = grp_key + (size_t)u * key_stride;
  auto wants = [&](int e) { const int t = tg[e]; return t >= 0 && t < e; };
  // pass 1: kept entries and their slots (a thread owns a run of consecutive entries)
  constexpr int RUN = 4;
  int n_keep = 0;
  for (int start = 0; start < len; start += nthr * RUN) {
    const int i0 = start + tid * RUN;
    bool mem[RUN];
    int n_k = 0;
#pragma unroll
    for (int r = 0; r < RUN; ++r) {
      const int e = i0 + r;
      mem[r] = e < len && wants(e) && !wants(tg[e]);   // its partner stays: e is a member
      n_k += (e < len && !mem[r]) ? 1 : 0;
    }
    int tot;
    int slot = n_keep + block_excl_sum(n_k, warp_tot, tot, nw);
#pragma unroll
    for (int r = 0; r < RUN; ++r) {
      const int e = i0 + r;
      if (e < len) {
        if (mem[r]) {
          ev_idx[base + (e - slot)] = e;
          slot_of[base + e] = -1 - (e - slot);   // a member: its position among the members
        } else {
          ret_idx[base + slot] = e;
          slot_of[base + e] = slot;
          ++slot;
        }
      }
    }
    n_keep += tot;
  }
  __syncthreads();   // (block scope: the global writes above are visible to the whole CTA)
  // pass 2: members look up the slot of their partner (partners are read before any target is overwritten:
  // a member's partner is a kept entry, and kept entries' targets are rewritten to -2 only after the barrier below)
  for (int e = tid; e < len; e += nthr) {
    const int so = slot_of[base + e];
    if (so < 0) {
      const int pos = -1 - so, slot = slot_of[base + tg[e]];
      gk[pos] = ((uint32_t)slot << 16) | (uint32_t)e;
      slot_of[base + e] = -0x40000000 + slot;   // remembered for the rewrite below
    }
  }
  __syncthreads();
  for (int e = tid; e < len; e += nthr) {
    const int so = slot_of[base + e];
    tg[e] = so < 0 ? so + 0x40000000 : -2;
  }
  if (tid == 0) {
    const int n_ev = len - n_keep;
    UnitInfo ui{len, n_keep, n_ev, 0, n_ev, 0, 0, 0};   // n_keys: every member is an entry to merge
    unit_info[u] = ui;
    unit_len[u] = n_keep;
    keepkv_stats st;
    st.n_retained = n_keep; st.n_evicted = n_ev; st.n_merged = 0; st.n_below_T = 0;
    st.n_guard_groups = 0; st.n_groups = 0; st.max_group = 0; st.reserved = 0;
    stats[u] = st;
  }
}

// Budget of each sequence for the eviction pass: the caller's, capped by the sequence's shortest merged head (the
// heads of a sequence share one seq_len, so they must all end at the same length).
__global__ void mf_budget_kernel(keepkv_params p, const int32_t *budget_dev, int budget_scalar, const int32_t *unit_len,
                                 int32_t *eff_budget) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= p.B) return;
  int m = p.N_cap;
  for (int h = 0; h < p.H_kv; ++h) m = min(m, unit_len[b * p.H_kv + h]);
  const int budget = max(0, min(budget_dev ? budget_dev[b] : budget_scalar, p.N_cap));
  eff_budget[b] = min(budget, m);
}

// What the caller sees of the two passes: the prompt index of every row of the result, and one record of statistics.
__global__ void mf_compose_kernel(keepkv_params p, const int32_t *seq_len, const int32_t *__restrict__ ret1,
                                  const int32_t *__restrict__ ret2, int32_t *ret_out, const keepkv_stats *st1,
                                  const UnitInfo *unit_info, const int32_t *prompt_len, keepkv_stats *stats_out) {
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.y, b = u / p.H_kv;
  const size_t base = (size_t)u * p.N_cap;
  const int n = seq_len[b];
  if (ret_out)
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x)
      ret_out[base + s] = ret1[base + ret2[base + s]];
  if (stats_out && blockIdx.x == 0 && threadIdx.x == 0) {
    keepkv_stats st = st1[u];
    st.n_evicted = st.n_retained + st.n_evicted - n;   // of the prompt's entries (kept + merged away in the merge pass)
    st.n_retained = n;
    st.n_below_T = 0;
    stats_out[u] = st;
  }
}

template <int D>
static void launch_compress_merge_first_t(const keepkv_params &p, const keepkv_cache &cache, const keepkv_cache &scratch,
                                          const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                                          int32_t *ret_idx_out, keepkv_stats *stats_out, char *ws, const WsLayout &L,
                                          int32_t *status_dev, LaunchCtx &ctx) {
  const int U = p.B * p.H_kv;
  UnitInfo *ui = reinterpret_cast<UnitInfo *>(ws + L.unit_info);
  int32_t *sched = reinterpret_cast<int32_t *>(ws + L.sched);
  int32_t *ret1 = reinterpret_cast<int32_t *>(ws + L.ret_idx);      // kept entries of the merge pass
  int32_t *target = reinterpret_cast<int32_t *>(ws + L.target);
  int32_t *ev_idx = reinterpret_cast<int32_t *>(ws + L.ev_idx);
  float *inv_norm = reinterpret_cast<float *>(ws + L.inv_norm);
  uint4 *norm_ext = reinterpret_cast<uint4 *>(ws + L.norm_ext);
  uint4 *nom = reinterpret_cast<uint4 *>(ws + L.nom);
  uint32_t *grp_key = reinterpret_cast<uint32_t *>(ws + L.grp_key);
  int32_t *grp_head = reinterpret_cast<int32_t *>(ws + L.grp_head);
  keepkv_stats *st1 = reinterpret_cast<keepkv_stats *>(ws + L.stats2);
  keepkv_stats *st2 = reinterpret_cast<keepkv_stats *>(ws + L.stats);
  int32_t *unit_len = reinterpret_cast<int32_t *>(ws + L.unit_len);
  int32_t *eff_budget = reinterpret_cast<int32_t *>(ws + L.eff_budget);
  static bool attr_done_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_done_dev[dev & 63]) {
    cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152 * 4);
    cudaFuncSetAttribute(group_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
    attr_done_dev[dev & 63] = true;
  }
  // The search's lists, 32 bytes a row, lie where the scratch cache's keys come later.
  unsigned long long *tri_best = nominate_pairs(p, p.N_cap) ? reinterpret_cast<unsigned long long *>(scratch.K) : nullptr;
  // ---- pass 1: similar entries merged with each other, cache -> scratch (every head keeps its own length for now)
  launch_pdl(mf_prepare_kernel<D>, dim3(norm_grid(p), U), dim3(256), 0, ctx.stream, p, cache, ev_idx, ui, inv_norm, norm_ext,
             reinterpret_cast<uint4 *>(tri_best));
  KEEPKV_CHECK_LAUNCH(ctx);
  // rows and columns are the same keys: the "retained" operand of the search is the prompt itself
  launch_nominate(p, cache, cache, ev_idx, ui, inv_norm, norm_ext, sched, nom, L.nom_chunks, status_dev, ctx, p.N_cap, 1,
                  tri_best);
  auto resolve = resolve_kernel<D, false>;
  if constexpr (D == 128) { if (tri_best) resolve = resolve_kernel<D, true>; }   // (the search by pairs takes 128 channels)
  launch_pdl(resolve, dim3(resolve_grid(p), U), dim3(kResolveThreads), 0,
      ctx.stream, p, cache, cache, ev_idx, ui, nom, sched, target, grp_key, L.key_stride, grp_head,
      st1, 1, (const ulonglong2 *)tri_best);
  KEEPKV_CHECK_LAUNCH(ctx);
  launch_pdl(mf_mark_kernel, dim3(U), dim3(1024), 0, ctx.stream, p, unit_len, ret1, target, ev_idx, grp_head, grp_key,
             L.key_stride, ui, st1);
  KEEPKV_CHECK_LAUNCH(ctx);
  const int cgx = (p.N_cap + 63) / 64 < 32 ? (p.N_cap + 63) / 64 : 32;
  launch_pdl(compact_kernel<D>, dim3(cgx, U), dim3(256), 0, ctx.stream, p, cache, scratch, ret1, ui, inv_norm, (uint4 *)nullptr);
  KEEPKV_CHECK_LAUNCH(ctx);
  launch_pdl(group_kernel<D>, dim3(U), dim3(kGroupThreads), (size_t)group_words(p, L) * 4, ctx.stream, p, cache, scratch,
             target, ui, grp_key, L.key_stride, grp_head, st1, group_words(p, L));
  KEEPKV_CHECK_LAUNCH(ctx);
  launch_pdl(merge_kernel<D>, dim3(merge_grid(p), U), dim3(256), 0, ctx.stream, p, cache, scratch, target, ui, grp_key,
             L.key_stride, grp_head, st1);
  KEEPKV_CHECK_LAUNCH(ctx);
  // ---- pass 2: the eviction strategy alone, scratch -> cache
  launch_pdl(mf_budget_kernel, dim3((p.B + 127) / 128), dim3(128), 0, ctx.stream, p, budget_dev, budget_scalar, unit_len,
             eff_budget);
  KEEPKV_CHECK_LAUNCH(ctx);
  int32_t *ret2 = grp_head;   // (free again: the groups are merged)
  launch_pdl(select_kernel, dim3(U), dim3(select_block(p)), (size_t)p.N_cap * sizeof(uint32_t), ctx.stream, p, scratch, cache.seq_len,
             (const int32_t *)eff_budget, 0, n_recent_dev, ret2, target, ev_idx, ui, st2, (const float *)nullptr,
             (const int32_t *)unit_len, (int32_t *)nullptr, (const int32_t *)nullptr, (const int32_t *)nullptr, status_dev);
  KEEPKV_CHECK_LAUNCH(ctx);
  launch_pdl(compact_kernel<D>, dim3(cgx, U), dim3(256), 0, ctx.stream, p, scratch, cache, ret2, ui, inv_norm, (uint4 *)nullptr);
  KEEPKV_CHECK_LAUNCH(ctx);
  if (ret_idx_out || stats_out) {
    launch_pdl(mf_compose_kernel, dim3(4, U), dim3(256), 0, ctx.stream, p, cache.seq_len, ret1, ret2, ret_idx_out, st1, ui,
               unit_len, stats_out);
    KEEPKV_CHECK_LAUNCH(ctx);
  }
}

void launch_compress_merge_first(const keepkv_params &p, const keepkv_cache &cache, const keepkv_cache &scratch,
                                 const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                                 int32_t *ret_idx_out, keepkv_stats *stats_out, char *ws, const WsLayout &L,
                                 int32_t *status_dev, LaunchCtx &ctx) {
  if (p.d == 128)
    launch_compress_merge_first_t<128>(p, cache, scratch, budget_dev, budget_scalar, n_recent_dev, ret_idx_out, stats_out, ws,
                                       L, status_dev, ctx);
  else
    launch_compress_merge_first_t<64>(p, cache, scratch, budget_dev, budget_scalar, n_recent_dev, ret_idx_out, stats_out, ws,
                                      L, status_dev, ctx);
}


// ------------------------------------------------------------------ Algorithm 1 in place (periodic mode, Section 1)
// keepkv_compress_inplace: "discard (k_e, v_e), (k_c, v_c) and insert (k_r, v_r)" taken literally.  Retained entries
// stay where they are, a merged entry overwrites its target's row, and only the retained rows beyond the new
// length move (into the rows of evicted entries below it), so a compression touches O(evicted + merged) rows
// instead of rewriting the cache.  The cache is then no longer in token order: a position array tells sinks and
// recent window (select_kernel in position mode).  The similarity search runs over the cache as it lies: its
// columns are all rows of the unit, and the rows that are not retained are taken out by a NaN in place of their
// inverse norm (a NaN never passes the strict comparisons of the search).
//   select (positions) -> ip_prepare (norms) -> ip_columns -> nominate -> resolve (+ few merges) -> group -> merge -> ip_move
template <int D>
__global__ void __launch_bounds__(256)
ip_prepare_kernel(keepkv_params p, keepkv_cache c, const int32_t *__restrict__ target, int32_t *ident, UnitInfo *unit_info,
                  float *__restrict__ inv_norm, uint4 *__restrict__ norm_ext) {
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.y;
  const int len = unit_info[u].len;
  const size_t base = (size_t)u * p.N_cap;
  auto kept = [&](int i) { return target[base + i] == -2; };
  each_row_norm<D>(reinterpret_cast<const uint4 *>(c.K) + base * (D / 8), len, kept, [&](int i, float ss) {
    const bool k = kept(i);
    norm_ext[base + i] = ext_col(k ? sqrtf(ss) : kExtNever);
    inv_norm[base + i] = k ? rsqrtf(ss) : __int_as_float(0x7fffffff);   // a row that is not retained is no column
    ident[base + i] = i;   // the slot of a target is its row
  });
}

// The search's column count is the unit's length (all rows lie in the operand); the rest of the record stays.
__global__ void ip_columns_kernel(UnitInfo *unit_info, int U) {
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.x * blockDim.x + threadIdx.x;
  if (u < U) unit_info[u].n_ret = unit_info[u].len;
}

// One CTA per unit: the retained rows at or above the new length move into the evicted rows below it, both in
// ascending order (ev_idx is ascending: the holes are its head; kept is ascending: the movers are its tail).  Then
// the new lengths are published.
template <int D>
__global__ void __launch_bounds__(256)
ip_move_kernel(keepkv_params p, keepkv_cache c, int32_t *pos, int32_t *pos_len, int32_t *n_seen,
               const int32_t *__restrict__ kept, const int32_t *__restrict__ ev_idx, const UnitInfo *__restrict__ unit_info,
               int32_t *moved_from) {
  constexpr int CH = D / 8;
  __shared__ int s_holes;
  pdl_wait();
  pdl_trigger();
  const int u = blockIdx.x, b = u / p.H_kv, h = u % p.H_kv, tid = threadIdx.x;
  const UnitInfo ui = unit_info[u];
  const int n_ret = ui.pad0, n_ev = ui.n_ev;   // pad0: the number of retained rows (n_ret holds the column count of the search)
  const size_t base = (size_t)u * p.N_cap;
  if (tid == 0) {   // holes = evicted rows below n_ret: a prefix of the ascending list
    int lo = 0, hi = n_ev;
    while (lo < hi) { const int mid = (lo + hi) >> 1; if (ev_idx[base + mid] < n_ret) lo = mid + 1; else hi = mid; }
    s_holes = lo;
  }
  __syncthreads();
  const int n_holes = s_holes;
  if (moved_from)
    for (int r = tid; r < n_ret; r += blockDim.x) moved_from[base + r] = r;
  __syncthreads();
  uint4 *K = reinterpret_cast<uint4 *>(c.K), *V = reinterpret_cast<uint4 *>(c.V);
  for (int idx = tid; idx < n_holes * 2 * CH; idx += blockDim.x) {   // a row pair (K, V) is 2 * CH pieces of 16 bytes
    const int k = idx / (2 * CH), piece = idx % (2 * CH);
    const int to = ev_idx[base + k], from = kept[base + (n_ret - n_holes + k)];
    uint4 *A = piece < CH ? K : V;
    const int ch = piece < CH ? piece : piece - CH;
    A[(base + to) * CH + ch] = A[(base + from) * CH + ch];
  }
  for (int k = tid; k < n_holes; k += blockDim.x) {
    const int to = ev_idx[base + k], from = kept[base + (n_ret - n_holes + k)];
    c.votes[base + to] = c.votes[base + from];
    c.lscore[base + to] = c.lscore[base + from];
    pos[base + to] = pos[base + from];
    if (moved_from) moved_from[base + to] = from;
  }
  if (h == 0 && tid == 0) {
    const int len = ui.len, first_fresh = max(0, min(pos_len[b], len));
    c.seq_len[b] = n_ret;
    n_seen[b] += len - first_fresh;
    pos_len[b] = n_ret;
  }
}

template <int D>
static void launch_compress_inplace_t(const keepkv_params &p, const keepkv_cache &c, int32_t *pos, int32_t *pos_len,
                                      int32_t *n_seen, const int32_t *budget_dev, int32_t budget_scalar,
                                      const int32_t *n_recent_dev, int32_t *moved_from, int32_t *target, keepkv_stats *stats,
                                      char *ws, const WsLayout &L, int32_t *status_dev, LaunchCtx &ctx) {
  const int U = p.B * p.H_kv;
  UnitInfo *ui = reinterpret_cast<UnitInfo *>(ws + L.unit_info);
  int32_t *sched = reinterpret_cast<int32_t *>(ws + L.sched);
  int32_t *ident = reinterpret_cast<int32_t *>(ws + L.ret_idx);    // slot -> row: the identity here
  int32_t *kept = reinterpret_cast<int32_t *>(ws + L.kept);        // retained rows, ascending
  int32_t *ev_idx = reinterpret_cast<int32_t *>(ws + L.ev_idx);
  float *inv_norm = reinterpret_cast<float *>(ws + L.inv_norm);
  uint4 *norm_ext = reinterpret_cast<uint4 *>(ws + L.norm_ext);
  uint4 *nom = reinterpret_cast<uint4 *>(ws + L.nom);
  uint32_t *grp_key = reinterpret_cast<uint32_t *>(ws + L.grp_key);
  int32_t *grp_head = reinterpret_cast<int32_t *>(ws + L.grp_head);
  static bool attr_done_dev[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (!attr_done_dev[dev & 63]) {
    cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 49152 * 4);
    cudaFuncSetAttribute(group_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kGroupSmem);
    attr_done_dev[dev & 63] = true;
  }
  launch_pdl(select_kernel, dim3(U), dim3(select_block(p)), (size_t)p.N_cap * sizeof(uint32_t), ctx.stream, p, c, (int32_t *)nullptr,
             budget_dev, budget_scalar, n_recent_dev, kept, target, ev_idx, ui, stats, (const float *)nullptr,
             (const int32_t *)nullptr, pos, (const int32_t *)pos_len, (const int32_t *)n_seen, status_dev);
  KEEPKV_CHECK_LAUNCH(ctx);
  launch_pdl(ip_prepare_kernel<D>, dim3(norm_grid(p), U), dim3(256), 0, ctx.stream, p, c, (const int32_t *)target, ident, ui, inv_norm, norm_ext);
  KEEPKV_CHECK_LAUNCH(ctx);
  const bool merges = !(isinf(p.merge_threshold) && p.merge_threshold > 0.f);
  if (merges) {
    launch_pdl(ip_columns_kernel, dim3((U + 127) / 128), dim3(128), 0, ctx.stream, ui, U);
    KEEPKV_CHECK_LAUNCH(ctx);
    launch_nominate(p, c, c, ev_idx, ui, inv_norm, norm_ext, sched, nom, L.nom_chunks, status_dev, ctx, 0);
    launch_pdl(resolve_kernel<D, false>, dim3(resolve_grid(p), U), dim3(kResolveThreads), 0, ctx.stream,
        p, c, c, ev_idx, ui, nom, sched, target, grp_key, L.key_stride, grp_head,
        stats, 0, (const ulonglong2 *)nullptr);
    KEEPKV_CHECK_LAUNCH(ctx);
    if (!all_small(p, budget_dev, budget_scalar)) {
      launch_pdl(group_kernel<D>, dim3(U), dim3(kGroupThreads), (size_t)group_words(p, L) * 4, ctx.stream, p, c, c,
                 target, ui, grp_key, L.key_stride, grp_head, stats, group_words(p, L));
      KEEPKV_CHECK_LAUNCH(ctx);
    }
    launch_pdl(merge_kernel<D>, dim3(merge_grid(p), U), dim3(256), 0, ctx.stream, p, c, c, target, ui, grp_key,
               L.key_stride, grp_head, stats);
    KEEPKV_CHECK_LAUNCH(ctx);
  }
  launch_pdl(ip_move_kernel<D>, dim3(U), dim3(256), 0, ctx.stream, p, c, pos, pos_len, n_seen, (const int32_t *)kept,
             (const int32_t *)ev_idx, (const UnitInfo *)ui, moved_from);
  KEEPKV_CHECK_LAUNCH(ctx);
}

void launch_compress_inplace(const keepkv_params &p, const keepkv_cache &c, int32_t *pos, int32_t *pos_len, int32_t *n_seen,
                             const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                             int32_t *moved_from, int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L,
                             int32_t *status_dev, LaunchCtx &ctx) {
  if (p.d == 128)
    launch_compress_inplace_t<128>(p, c, pos, pos_len, n_seen, budget_dev, budget_scalar, n_recent_dev, moved_from, target,
                                   stats, ws, L, status_dev, ctx);
  else
    launch_compress_inplace_t<64>(p, c, pos, pos_len, n_seen, budget_dev, budget_scalar, n_recent_dev, moved_from, target,
                                  stats, ws, L, status_dev, ctx);
}

void launch_compress(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                     const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev, int32_t *ret_idx,
                     int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L, int32_t *status_dev,
                     LaunchCtx &ctx, const float *select_key) {
  if (p.d == 128)
    launch_compress_t<128>(p, src, dst, budget_dev, budget_scalar, n_recent_dev, ret_idx, target, stats, ws, L,
                           status_dev, select_key, ctx);
  else
    launch_compress_t<64>(p, src, dst, budget_dev, budget_scalar, n_recent_dev, ret_idx, target, stats, ws, L,
                          status_dev, select_key, ctx);
}

}  // namespace keepkv
