// Device helpers shared by the kernels of keepkv_compress (compress.cu: the general pipeline;
// compress_steady.cu: the single-kernel path of a steady-state compression).
#pragma once
#include <type_traits>

#include "common.cuh"

namespace keepkv {

constexpr float kRankEps = 1e-4f;   // tensor-core cosines closer than this are re-evaluated in the interface's fp32 chain

// ------------------------------------------------------------------ block scans
// The barrier of the threads that take part (the block, unless the kernel has warps with other work).
struct BlockSync { __device__ __forceinline__ void operator()() const { __syncthreads(); } };
// The sums of warp_tot over the warps before this one and over all nw <= 32, a warp's value per lane.  (A loop over 32 warps is
// half a microsecond of shared-memory latency.)
__device__ __forceinline__ int warps_before(const int *warp_tot, int &total, int nw) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, v = lane < nw ? warp_tot[lane] : 0;
  total = __reduce_add_sync(0xffffffffu, v);
  return __reduce_add_sync(0xffffffffu, lane < warp ? v : 0);
}
// Exclusive prefix count of `flag` over the first nw warps of the block in thread order (the other
// warps have left the kernel); total returned through `total`.
template <typename Sync = BlockSync>
__device__ __forceinline__ int block_excl_count(bool flag, int *warp_tot, int &total, int nw, Sync sync = Sync()) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, flag);
  const int in_warp = __popc(bal & ((1u << lane) - 1u));
  sync();  // warp_tot may still be read from the previous call
  if (lane == 0) warp_tot[warp] = __popc(bal);
  sync();
  return warps_before(warp_tot, total, nw) + in_warp;
}
__device__ __forceinline__ int block_excl_count(bool flag, int *warp_tot, int &total) {
  return block_excl_count(flag, warp_tot, total, (int)(blockDim.x >> 5));
}

// Exclusive prefix sum of small non-negative ints over the block (thread order).
template <typename Sync = BlockSync>
__device__ __forceinline__ int block_excl_sum(int v, int *warp_tot, int &total, int nw, Sync sync = Sync()) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  sync();
  if (lane == 31) warp_tot[warp] = x;
  sync();
  return warps_before(warp_tot, total, nw) + x - v;
}

// ------------------------------------------------------------------ selection key
// Order-preserving map of an fp32 value to u32 (-0 folded onto +0 so equal floats give equal keys).
__device__ __forceinline__ uint32_t ordered_key(float x) {
  x += 0.0f;
  const uint32_t b = __float_as_uint(x);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
// kappa = ln p + lscore in fp64, rounded once to fp32 (p = 1 needs no logarithm)
__device__ __forceinline__ uint32_t kappa_key(float pv, float ls) {
  const float kappa = (pv == 1.0f) ? ls : (float)(log((double)pv) + (double)ls);
  return ordered_key(kappa);
}

// nthr threads (a power of two, 64 to 1024; thread tid) find the kr-th largest of keys[lo..hi), all of which lie in
// [k_lo, k_hi], by histograms of kSelBins bins over that range: the bin that holds it becomes the next range, so three
// passes settle any 32-bit key, and a bin with one key ends the search.  (The leading byte of most keys coincides: fixed
// 8-bit digits put the counts into a few bins, which took a pass more and one atomic per distinct digit of a warp.)  kth =
// that key, n_tie = how many entries equal to it belong to the kr largest (lowest index first), tot_ties = how many
// entries equal to it exist.  hist: kSelBins words, sh: four, warp_tot: one per warp of shared memory.
constexpr int kSelBins = 2048;
// Where a bin's count lies: a thread sums consecutive bins, up to 32, and unswizzled those of a warp's lanes met in a bank.
__device__ __forceinline__ int sel_bin(int b) { return b ^ ((b >> 5) & 31); }
template <typename Sync = BlockSync>
__device__ __forceinline__ void range_select(const uint32_t *keys, int lo, int hi, uint32_t k_lo, uint32_t k_hi, int kr, int nthr,
                                             int *hist, int *sh, int *warp_tot, uint32_t &kth, int &n_tie, int &tot_ties,
                                             Sync sync = Sync()) {
  const int tid = threadIdx.x, bpt = kSelBins / nthr;
  for (;;) {
    const int shift = max(0, 21 - __clz(k_hi - k_lo));   // (bits of the span less the 11 of a bin number)
    for (int i = tid; i < kSelBins; i += nthr) hist[i] = 0;
    sync();
#pragma unroll 4
    for (int i = lo + tid; i < hi; i += nthr) {
      const uint32_t k = keys[i];
      if (k >= k_lo && k <= k_hi) atomicAdd(&hist[sel_bin((int)((k - k_lo) >> shift))], 1);
    }
    sync();
    // bins from the top: thread t owns bins kSelBins - 1 - t * bpt downwards
    int sum = 0;
#pragma unroll 4
    for (int j = 0; j < bpt; ++j) sum += hist[sel_bin(kSelBins - 1 - tid * bpt - j)];
    int tot;
    int above = block_excl_sum(sum, warp_tot, tot, nthr >> 5, sync);
    if (above < kr && above + sum >= kr) {
      int bin = kSelBins - 1 - tid * bpt;
      int n = hist[sel_bin(bin)];
      while (above + n < kr) {
        above += n;
        n = hist[sel_bin(--bin)];
      }
      sh[0] = bin;
      sh[1] = kr - above;
      sh[2] = n;
    }
    sync();   // (not written again before the barriers of the next pass)
    k_lo += (uint32_t)sh[0] << shift;
    k_hi = min(k_hi, k_lo + ((1u << shift) - 1u));
    kr = sh[1];
    if (shift == 0) break;
    if (sh[2] == 1) {   // the only key in the range
#pragma unroll 4
      for (int i = lo + tid; i < hi; i += nthr) {
        const uint32_t k = keys[i];
        if (k >= k_lo && k <= k_hi) sh[3] = (int)k;
      }
      sync();
      k_lo = (uint32_t)sh[3];
      break;
    }
  }
  kth = k_lo;
  n_tie = kr;
  tot_ties = sh[2];
}

// ------------------------------------------------------------------ tensor-core ranking: top two of a row
// Running top two of one row.  Only values within `thr` of the running best are looked at: the
// final best can only be larger, so every value within thr of the FINAL best has been inserted, and
// (best, second) are exact among those -- which is all the caller's closeness tests use.
// A warp holds 32 rows, and the drain is bound by the ALU pipe (compares and selects), so a group of
// four columns is either skipped by the whole warp -- four fused multiply-adds give v - cut and the
// sign bits are AND-ed -- or updated by the whole warp with selects only (no divergent branch).
struct Top2 {
  float best, second, cut, thr;
  int bi, si;
  __device__ __forceinline__ void init(float thr_) {
    best = second = cut = -CUDART_INF_F;
    thr = thr_;
    bi = si = -1;
  }
  // Comparisons are strict, so among equal values the one seen first (the lower slot) stays in
  // front, and a NaN (a zero-norm key) is never taken.
  __device__ __forceinline__ void insert(float v, int idx) {
    const bool p1 = v > best, p2 = v > second;
    second = p1 ? best : fmaxf(second, v);
    si = p1 ? bi : (p2 ? idx : si);
    bi = p1 ? idx : bi;
    best = fmaxf(best, v);
  }
  // Insert for candidates that arrive out of slot order (the other tracker of the thread): equal values
  // go to the lower slot, as if the columns had been scanned in order.
  __device__ __forceinline__ void insert_any(float v, int idx) {
    const bool p1 = v > best || (v == best && idx < bi), p2 = v > second || (v == second && idx < si);
    second = p1 ? best : (p2 ? v : second);
    si = p1 ? bi : (p2 ? idx : si);
    bi = p1 ? idx : bi;
    best = p1 ? v : best;
  }
};

// Two trackers per thread, one for the even and one for the odd columns, so that the select chains of
// neighbouring columns do not wait on each other.  Both share one cut (kept in ta.cut), taken from the larger of
// their two bests: the row's final best is at least that, so a value below the cut cannot be within thr of it,
// whichever list it would have gone to; what the two lists hold together still contains the row's two largest
// values within thr of its best.  (A cut from the smaller best lets through everything between the two bests,
// and with 32 rows per warp the warp-wide skip then hardly ever fires.)
// a_i: accumulators, w_i: inverse norms of the four columns idx..idx+3.
__device__ __forceinline__ void offer4(Top2 &ta, Top2 &tb, float a0, float a1, float a2, float a3, const float4 w,
                                       int idx) {
  const float ncut = -ta.cut;
  const uint32_t s = __float_as_uint(fmaf(a0, w.x, ncut)) & __float_as_uint(fmaf(a1, w.y, ncut)) &
                     __float_as_uint(fmaf(a2, w.z, ncut)) & __float_as_uint(fmaf(a3, w.w, ncut));
  if (!__any_sync(0xffffffffu, (int)s >= 0)) return;   // no lane has a value that is not below its cut
  ta.insert(a0 * w.x, idx); tb.insert(a1 * w.y, idx + 1); ta.insert(a2 * w.z, idx + 2); tb.insert(a3 * w.w, idx + 3);
  ta.cut = fmaxf(ta.cut, fmaxf(ta.best, tb.best) - ta.thr);   // (a cut only rises: it may have started above the best)
}

// ------------------------------------------------------------------ the cut inside the product
// c |k_c| as six products of bf16 terms (c = c1 + c2 + c3 and likewise the norm; what is left out is below 2^-23 of it):
// eight more channels of a row and of a column, whose product subtracts it from the accumulator.
constexpr float kExtNever = 1.2676506e30f;   // 2^100: a row no column reaches, a column that reaches no row
__device__ __forceinline__ void bf16_terms(float x, float &t1, float &t2, float &t3) {
  t1 = __bfloat162float(__float2bfloat16_rn(x));
  t2 = __bfloat162float(__float2bfloat16_rn(x - t1));
  t3 = x - t1 - t2;
}
__device__ __forceinline__ uint4 ext_row(float c) {
  float a, b, d;
  bf16_terms(c, a, b, d);
  return make_uint4(pack_bf16(-a, -a), pack_bf16(-b, -a), pack_bf16(-b, -d), 0u);
}
__device__ __forceinline__ uint4 ext_col(float n) {
  float a, b, d;
  bf16_terms(n, a, b, d);
  return make_uint4(pack_bf16(a, b), pack_bf16(a, d), pack_bf16(b, a), 0u);
}

// ------------------------------------------------------------------ the interface's cosine
// One warp evaluates cos(k_e, k_a) and cos(k_e, k_b) in the fixed fp32 arithmetic of the interface:
// dot and squared norms by fused multiply-add from 0 over channels 0..D-1, then dot/(sqrtf(n_e)*sqrtf(n_c)).
// ke_s [D] and kc_s [2][D] are the warp's staging rows in shared memory.  Results in every lane.
template <int D>
__device__ __forceinline__ void exact_cosines(const __nv_bfloat16 *ke, const __nv_bfloat16 *ka, const __nv_bfloat16 *kb,
                                              float *ke_s, float *kc_s, float &ua, float &ub) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  for (int c = lane; c < D; c += 32) {
    ke_s[c] = __bfloat162float(ke[c]);
    kc_s[c] = __bfloat162float(ka[c]);
    kc_s[D + c] = __bfloat162float(kb[c]);
  }
  __syncwarp();
  // lanes 0 and 1: dot and |k_c|^2 of one candidate each; lane 2: |k_e|^2
  const float *x = ke_s, *y = lane == 2 ? ke_s : kc_s + (lane & 1) * D;
  float dot = 0.f, nn = 0.f;
  if (lane < 3)
    for (int c = 0; c < D; ++c) { dot = fmaf(x[c], y[c], dot); nn = fmaf(y[c], y[c], nn); }
  const float ne = __shfl_sync(0xffffffffu, nn, 2);
  const float uu = dot / (sqrtf(ne) * sqrtf(nn));
  ua = __shfl_sync(0xffffffffu, uu, 0);
  ub = __shfl_sync(0xffffffffu, uu, 1);
}

// The same sums by one thread: x . y and |y|^2.
template <int D>
__device__ __forceinline__ void exact_dot(const __nv_bfloat16 *x, const __nv_bfloat16 *y, float &dot, float &nn) {
  const uint4 *xp = reinterpret_cast<const uint4 *>(x), *yp = reinterpret_cast<const uint4 *>(y);
  dot = nn = 0.f;
#pragma unroll 2
  for (int k = 0; k < D / 8; ++k) {
    const uint4 a = xp[k], b = yp[k];
    const uint32_t aw[4] = {a.x, a.y, a.z, a.w}, bw[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float b0 = bf16_lo(bw[q]), b1 = bf16_hi(bw[q]);
      dot = fmaf(bf16_lo(aw[q]), b0, dot);
      nn = fmaf(b0, b0, nn);
      dot = fmaf(bf16_hi(aw[q]), b1, dot);
      nn = fmaf(b1, b1, nn);
    }
  }
}

// ------------------------------------------------------------------ merge
// One warp per group.  With a_i = ln p_i + lscore_i over the group K'_e (target first, then members
// ascending):  omega = softmax(a),  v_r = sum omega_i v_i,  k_r = gamma * sum omega_i k_i,
// gamma = L / lambda_bar,  L = LSE(a) - ln(sum p),  lambda_bar = sum omega_i lscore_i,  p_r = sum p,
// lscore_r = L   (Eq. A.3 in logarithms).  c: the target's slot in dst, (tc, ti): a cache and row that hold the target as
// it was, member(t): source index of the t-th member (ascending), target_u: the unit's per-entry targets.
// Bound: the chain of dependent loads of the warp with the largest group.  So the target is read where it was copied to (its
// source index would be one load more), members are known by source index, the first kMergePre rows are requested with the
// votes, before the weights are known, the others eight at a time, and beyond 31 members every lane weighs its own (one
// after the other in all lanes, a group of 45 was what 35 us of a launch over 15000 groups waited for).
constexpr int kMergePre = 4;

// What a warp has merged: added to the unit's statistics once, when it has done all its groups.
struct MergeCount {
  int merged = 0, groups = 0, guarded = 0, most = 0;
  __device__ __forceinline__ void flush(keepkv_stats *st) const {
    if ((threadIdx.x & 31) || !groups) return;
    if (merged) { atomicAdd(&st->n_merged, merged); atomicMax(&st->max_group, most); }
    if (guarded) atomicAdd(&st->n_guard_groups, guarded);
    atomicAdd(&st->n_groups, groups);
  }
};
template <int D, typename MemberFn>
__device__ __forceinline__ void merge_group(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                                            int c, const keepkv_cache &tc, size_t ti, MemberFn member, int n, int32_t *target_u,
                                            size_t base,
                                            MergeCount &count) {
  constexpr int EPL = D / 32;
  const int lane = threadIdx.x & 31;
  const float *votes = src.votes + base, *ls = src.lscore + base;
  const __nv_bfloat16 *sK = reinterpret_cast<const __nv_bfloat16 *>(src.K) + base * D;
  const __nv_bfloat16 *sV = reinterpret_cast<const __nv_bfloat16 *>(src.V) + base * D;

  // The group's scalars: L = LSE(a) - ln(sum p) and lambda_bar cancel to almost nothing when the members' log-scores sit
  // near zero, and gamma = L / lambda_bar then carries whatever relative error they have into every channel of the
  // merged key (an fp32 L of 1e-5 is off by a percent).  So groups near the cancellation, and large ones, are evaluated in
  // fp64, the others in fp32; the row sums stay fp32.
  float ka[EPL], va[EPL];
  double lbar = 0.0, L, Ps;
#pragma unroll
  for (int e = 0; e < EPL; ++e) { ka[e] = 0.f; va[e] = 0.f; }
  using Row = typename std::conditional<EPL == 4, uint2, uint32_t>::type;   // a lane's part of a row
  const Row *rK = reinterpret_cast<const Row *>(sK) + lane, *rV = reinterpret_cast<const Row *>(sV) + lane;
  const Row *qK = reinterpret_cast<const Row *>(reinterpret_cast<const __nv_bfloat16 *>(tc.K) + ti * D) + lane;
  const Row *qV = reinterpret_cast<const Row *>(reinterpret_cast<const __nv_bfloat16 *>(tc.V) + ti * D) + lane;
  auto add_row = [&](const Row kk, const Row vv, float om) {
    if constexpr (EPL == 4) {
      ka[0] = fmaf(om, bf16_lo(kk.x), ka[0]); ka[1] = fmaf(om, bf16_hi(kk.x), ka[1]);
      ka[2] = fmaf(om, bf16_lo(kk.y), ka[2]); ka[3] = fmaf(om, bf16_hi(kk.y), ka[3]);
      va[0] = fmaf(om, bf16_lo(vv.x), va[0]); va[1] = fmaf(om, bf16_hi(vv.x), va[1]);
      va[2] = fmaf(om, bf16_lo(vv.y), va[2]); va[3] = fmaf(om, bf16_hi(vv.y), va[3]);
    } else {
      ka[0] = fmaf(om, bf16_lo(kk), ka[0]); ka[1] = fmaf(om, bf16_hi(kk), ka[1]);
      va[0] = fmaf(om, bf16_lo(vv), va[0]); va[1] = fmaf(om, bf16_hi(vv), va[1]);
    }
  };
  auto accumulate = [&](int i, float om) { add_row(rK[(size_t)i * 32], rV[(size_t)i * 32], om); };
  auto wsum_d = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  auto wmax_d = [](double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  };
  const double NEG_INF = -CUDART_INF;
  if (n < 32) {
    // the usual case: lane 0 holds the target, lane t the t-th member, so that their votes and scores are
    // fetched together and the row loads of the accumulation do not wait on one another
    const int idx = lane == 0 ? 0 : (lane <= n ? member(lane - 1) : -1);
    Row kp[kMergePre], vp[kMergePre];
#pragma unroll
    for (int t = 0; t < kMergePre; ++t) {
      const int i = __shfl_sync(0xffffffffu, idx, t);
      if (t == 0) { kp[t] = __ldcg(qK); vp[t] = __ldcg(qV); }
      else if (t <= n) { kp[t] = rK[(size_t)i * 32]; vp[t] = rV[(size_t)i * 32]; }
    }
    float pv = 0.f, lsv = 0.f;
    if (lane == 0) { pv = __ldcg(tc.votes + ti); lsv = __ldcg(tc.lscore + ti); }
    else if (idx >= 0) { pv = votes[idx]; lsv = ls[idx]; }
    // fp32 first: with |L| and |lambda_bar| away from zero its error (about 1e-6 absolute) is far below bf16
    // resolution in gamma; only a group near the cancellation is evaluated again in fp64 (a warp-uniform choice)
    float om;
    {
      const float a = idx >= 0 ? logf(pv) + lsv : -CUDART_INF_F;
      const float M = warp_max(a);
      const float Z = warp_sum(idx >= 0 ? expf(a - M) : 0.f);
      const float Psf = warp_sum(pv);
      const float Lam = M + logf(Z);
      const float Lf = Lam - logf(Psf);
      om = idx >= 0 ? expf(a - Lam) : 0.f;
      const float lbf = warp_sum(om * lsv);
      Ps = (double)Psf; L = (double)Lf; lbar = (double)lbf;
    }
    if (!(fabs(L) >= 0.25 && fabs(lbar) >= 0.25)) {
      const double a = idx >= 0 ? log((double)pv) + (double)lsv : NEG_INF;
      const double M = wmax_d(a);
      const double Z = wsum_d(idx >= 0 ? exp(a - M) : 0.0);
      Ps = wsum_d((double)pv);
      const double Lam = M + log(Z);
      L = Lam - log(Ps);
      const double omd = idx >= 0 ? exp(a - Lam) : 0.0;
      lbar = wsum_d(omd * (double)lsv);
      om = (float)omd;
    }
#pragma unroll
    for (int t = 0; t < kMergePre; ++t) {
      const float w = __shfl_sync(0xffffffffu, om, t);
      if (t <= n) add_row(kp[t], vp[t], w);
    }
#pragma unroll 8
    for (int t = kMergePre; t <= n; ++t) accumulate(__shfl_sync(0xffffffffu, idx, t), __shfl_sync(0xffffffffu, om, t));
  } else {
    // Larger groups: 32 members at a time, one a lane, three times over (maximum, sums, weights with the rows); fp64.
    const float pc = __ldcg(tc.votes + ti), lc = __ldcg(tc.lscore + ti);
    const double a_c = log((double)pc) + (double)lc;
    double M = a_c;
    for (int t = lane; t < n; t += 32) { const int e = member(t); M = fmax(M, log((double)votes[e]) + (double)ls[e]); }
    M = wmax_d(M);
    double Z = 0.0;
    Ps = 0.0;
    if (lane == 0) { Z = exp(a_c - M); Ps = (double)pc; }
    for (int t = lane; t < n; t += 32) {
      const int e = member(t);
      Z += exp(log((double)votes[e]) + (double)ls[e] - M);
      Ps += (double)votes[e];
    }
    Z = wsum_d(Z);
    Ps = wsum_d(Ps);
    const double Lam = M + log(Z);
    L = Lam - log(Ps);
    const double om_c = exp(a_c - Lam);
    lbar = lane == 0 ? om_c * (double)lc : 0.0;
    add_row(__ldcg(qK), __ldcg(qV), (float)om_c);
    for (int t0 = 0; t0 < n; t0 += 32) {
      const int e = t0 + lane < n ? member(t0 + lane) : 0;
      double omd = 0.0;
      if (t0 + lane < n) {
        const double lsi = (double)ls[e];
        omd = exp(log((double)votes[e]) + lsi - Lam);
        lbar += omd * lsi;
      }
      const float om = (float)omd;
      const int m = min(32, n - t0);
#pragma unroll 8
      for (int t = 0; t < m; ++t) accumulate(__shfl_sync(0xffffffffu, e, t), __shfl_sync(0xffffffffu, om, t));
    }
    lbar = wsum_d(lbar);
  }
  const double gamma_d = L / lbar;
  const float gamma = (float)gamma_d;
  const bool ok = gamma_d > (double)p.gamma_min && gamma_d <= (double)p.gamma_max && fabs(lbar) >= 1e-6;
  if (!ok) {
    // guard: the members are dropped after all and the target keeps the row copied by compaction
    for (int t = lane; t < n; t += 32) target_u[member(t)] = -1;
    ++count.guarded;
    ++count.groups;
    return;
  }
  __nv_bfloat16 *dK = reinterpret_cast<__nv_bfloat16 *>(dst.K) + (base + c) * D;
  __nv_bfloat16 *dV = reinterpret_cast<__nv_bfloat16 *>(dst.V) + (base + c) * D;
  if constexpr (EPL == 4) {
    uint2 ko, vo;
    ko.x = pack_bf16(gamma * ka[0], gamma * ka[1]); ko.y = pack_bf16(gamma * ka[2], gamma * ka[3]);
    vo.x = pack_bf16(va[0], va[1]); vo.y = pack_bf16(va[2], va[3]);
    *reinterpret_cast<uint2 *>(dK + lane * 4) = ko;
    *reinterpret_cast<uint2 *>(dV + lane * 4) = vo;
  } else {
    *reinterpret_cast<uint32_t *>(dK + lane * 2) = pack_bf16(gamma * ka[0], gamma * ka[1]);
    *reinterpret_cast<uint32_t *>(dV + lane * 2) = pack_bf16(va[0], va[1]);
  }
  if (lane == 0) {
    dst.votes[base + c] = (float)Ps;
    dst.lscore[base + c] = (float)L;
  }
  count.merged += n;
  ++count.groups;
  count.most = max(count.most, n);
}

// the single-kernel path of a steady-state compression (compress_steady.cu)
void launch_compress_steady(const keepkv_params &p, const keepkv_cache &src, const keepkv_cache &dst,
                            const int32_t *budget_dev, int32_t budget_scalar, const int32_t *n_recent_dev,
                            int32_t *ret_idx, int32_t *target, keepkv_stats *stats, char *ws, const WsLayout &L,
                            int32_t *status_dev, const float *select_key, LaunchCtx &ctx);

}  // namespace keepkv
