// Step 2b of VMoBA: global (per head) threshold selection of (query, key-block) pairs
// (Eq. 3 TopkMask, Eq. 4 threshold k), and emission of the work lists the attention
// kernels consume.
//
// Sorting the head's pool and accumulating normalised similarity until tau is reached is
// equivalent to finding the weighted quantile of the scores under the softmax weights:
// the cutoff is the largest score c with mass{score >= c} >= tau * Z.  That is found without a sort, by one of two
// routes that the size of the pool decides:
//
//   small   : select_pool_kernel, a cluster per head with the scores on chip, does everything before fill (pool_plan)
//   larger  : init (+ minmax, unless the caller hands over each head's score range)
//             -> hist level 0 -> scan -> hist level 1 -> scan -> hist level 2 -> scan (cutoff): histogram refinements, linear in
//             the score, fp64 bin masses; level 1 copies the pairs of the level-0 crossing bin aside, and level 2 reads that
//             short list instead of the score matrix; then mark .. fill
//
//   mark    : mask bits (one comparison per pair) + per (segment, block) counts + per-segment pair totals
//   offsets : CSR offsets by key block (kb_ptr) and by query (q_ptr)
//   fill    : q_idx (queries of each key block, ascending) and q_pairs (pairs of each query)
//
// Every pass streams the score matrix with 16-byte loads and is bound by HBM bandwidth, the small route by latency.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "common.cuh"

namespace vmoba {

constexpr int kBins = 2048;
constexpr int kBins0 = 512;    // level 0 uses fewer bins, each replicated once per lane
constexpr int kSegThreads = 512;
constexpr int kCandStage = 1024;      // pairs of the crossing bin that a CTA of the level-1 pass gathers

struct HeadState {
  uint32_t min_key, max_key;   // order-preserving keys of the head's extreme scores
  float anchor[3];             // lower edge of the interval refined at each level
  float inv[3];                // bins per unit score at each level
  int bin[3];                  // crossing bin found at each level
  int resolved;                // the level-1 crossing bin held a single distinct score: level 2 is skipped
  double Z;                    // sum of all weights
  double target;               // tau * Z
  double mass_above;           // weight of everything above the crossing bin so far
  unsigned long long cnt_above;
  uint32_t cutoff_key;
  unsigned int cand_cnt;       // pairs of the level-0 crossing bin, copied aside by the level-1 pass
  int cand_ok;                 // every one of them found room in the list: level 2 reads the list
  float bin0_off;              // -anchor[0] * inv[0]: the level-0 bin of s is floor(s * inv[0] + bin0_off)
  uint32_t pad;
};

// bin of a score at refinement level L given the state; monotone non-decreasing in s.
// Unnormalised softmax weight of a pair relative to the head's largest score (Eq. 4 accumulates these
// in descending score order).  One definition for every histogram level and for the final exact
// steps, so that the masses they hand to each other are sums of the same numbers; the fast
// exponential (one multiply, one ex2) is within a few ulp of expf over the range that carries mass.
// One fused multiply-add and one ex2 per pair: exp(sigma (s - smax)) = 2^(s c - smax c) with c = sigma log2(e);
// c and smax c do not depend on the pair and leave the loops.
__device__ __forceinline__ float pair_weight(float sigma, float s, float smax) {
  const float c = sigma * 1.4426950408889634f;
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(fmaf(s, c, -smax * c)));
  return y;
}

// Level 0 sees every pair: its bin is one fused multiply-add (bin0_off = -anchor[0] * inv[0], a number of bins, so
// its rounding moves a bin edge by a few millionths of a bin) and an integer clamp.  The finer levels keep the
// subtraction first: their inv is so large that the product form would cancel.
__device__ __forceinline__ int bin_at(const HeadState& hs, int L, float s) {
  if (L == 0) return min(max(__float2int_rd(fmaf(s, hs.inv[0], hs.bin0_off)), 0), kBins0 - 1);
  float t = (s - hs.anchor[L]) * hs.inv[L];
  int b = t > 0.f ? (int)fminf(t, (float)(kBins - 1)) : 0;
  return b;
}

// Streams the P scores of one head through f(value); blockIdx.x strides over chunks.  DOWN: from the end of the head to
// its start, which finds in L2 what the pass before read or wrote last.
template <bool DOWN, typename F>
__device__ __forceinline__ void for_each_score(const float* __restrict__ base, long long P, F f) {
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long nth = (long long)gridDim.x * blockDim.x;
  if ((reinterpret_cast<uintptr_t>(base) & 15u) == 0) {
    long long P4 = P >> 2;
    const float4* b4 = reinterpret_cast<const float4*>(base);
    long long i = tid;
    for (; i + 3 * nth < P4; i += 4 * nth) {     // four independent 16-byte loads in flight
      float4 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = __ldg(b4 + (DOWN ? P4 - 1 - (i + j * nth) : i + j * nth));
#pragma unroll
      for (int j = 0; j < 4; ++j) { f(x[j].x); f(x[j].y); f(x[j].z); f(x[j].w); }
    }
    for (; i < P4; i += nth) {
      float4 x = __ldg(b4 + (DOWN ? P4 - 1 - i : i));
      f(x.x); f(x.y); f(x.z); f(x.w);
    }
    for (long long i = (P4 << 2) + tid; i < P; i += nth) f(__ldg(base + i));
  } else {
    for (long long i = tid; i < P; i += nth) f(__ldg(base + i));
  }
}

// Key of a score under the head-wide rules: that of float_key, but a NaN without a sign has the place of -0 (one with a sign lies
// below -inf), so that a diverged score neither sets the head's range nor is taken for its largest.  Said here, because what
// float_key makes of a NaN is the compiler's choice: where the value is also a float, it may take `bits | sign` for a float negation,
// which returns any NaN.
__device__ __forceinline__ uint32_t pool_key(float f) {
  return __float_as_int(f) > 0x7f800000 ? 0x7fffffffu : float_key(f);
}

__global__ void __launch_bounds__(256)
minmax_kernel(const float* __restrict__ scores, long long P, HeadState* __restrict__ st) {
  if (!grid_begin()) return;
  const int bh = blockIdx.y;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
  for_each_score<false>(scores + (long long)bh * P, P, [&](float s) {
    const uint32_t k = pool_key(s);
    kmin = min(kmin, k);
    kmax = max(kmax, k);
  });
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&st[bh].min_key, kmin);
    atomicMax(&st[bh].max_key, kmax);
  }
}

// Start of a call: the per-head state and, for the head-wide rules, the histogram arrays (one kernel instead of
// a memset per array).  If the caller knows each head's score range (range: [BH][2] = minimum, maximum, as
// vmoba_block_scores_range writes them), the level-0 bins are laid over it here and no pass of the selection's
// own has to look for it.
__global__ void init_state_kernel(HeadState* st, int BH, const float* __restrict__ range, unsigned int* __restrict__ g_cnt,
                                  double* __restrict__ g_w, uint32_t* __restrict__ g_minkey,
                                  uint32_t* __restrict__ g_maxkey) {
  if (!grid_begin()) return;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g_cnt && i < (long long)BH * kBins) { g_cnt[i] = 0u; g_w[i] = 0.0; g_minkey[i] = 0xffffffffu; g_maxkey[i] = 0u; }
  if (i >= BH) return;
  HeadState h;
  memset(&h, 0, sizeof(h));
  h.min_key = 0xffffffffu;
  h.max_key = 0u;
  h.cutoff_key = 0xffffffffu;      // the per-query rules take the minimum of their row cutoffs into it
  if (range) {
    const float lo = range[2 * i], hi = range[2 * i + 1];
    h.min_key = float_key(lo);
    h.max_key = float_key(hi);
    const float span = hi - lo;
    h.anchor[0] = lo;
    h.inv[0] = span > 0.f ? (float)kBins0 / span : 0.f;
    h.bin0_off = -lo * h.inv[0];
  }
  st[i] = h;
}

// Level L >= 1 histogram: pairs that fall in the crossing bins of all earlier levels add
// (1, exp(sigma * (s - max))) to their level-L bin.  The smallest key of each bin is tracked too,
// which turns the last crossing bin into an exact fp32 cutoff; at level 1 also the largest, so that
// a crossing bin with a single distinct score ends the search there.
template <int L>
__global__ void __launch_bounds__(256)
hist_kernel(const float* __restrict__ scores, long long P, const HeadState* __restrict__ st, float sigma, int unit_w,
            unsigned int* __restrict__ g_cnt, double* __restrict__ g_w, uint32_t* __restrict__ g_minkey,
            uint32_t* __restrict__ g_maxkey, float* __restrict__ cand, long long ccap, unsigned int* __restrict__ cand_cnt) {
  if (!grid_begin()) return;
  __shared__ unsigned int s_cnt[kBins];
  __shared__ float s_w[kBins];
  __shared__ uint32_t s_min[kBins];
  __shared__ uint32_t s_max[L == 1 ? kBins : 1];
  __shared__ float s_cand[L == 1 ? kCandStage : 1];
  __shared__ unsigned int s_cand_n, s_cand_at;
  const int bh = blockIdx.y;
  const HeadState hs = st[bh];
  if (L == 2 && hs.resolved) return;     // level 1 already pinned the cutoff: nothing to refine
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) {
    s_cnt[i] = 0; s_w[i] = 0.f;
    s_min[i] = 0xffffffffu;
    if (L == 1) s_max[i] = 0u;
  }
  if (threadIdx.x == 0) s_cand_n = 0u;
  __syncthreads();
  const float smax = key_float(hs.max_key);
  // level 1 copies the pairs of the level-0 crossing bin (one bin of 512: few) to the head's list; level 2 reads
  // the list instead of the matrix if all of them found room.  They are gathered in shared memory and get their places
  // with one atomic per CTA: with one each, a warp waits for the answer at every pair (white inputs, 55 million pairs:
  // 142 us against 68).
  float* list = cand ? cand + (long long)bh * ccap : nullptr;
  const bool from_list = L == 2 && hs.cand_ok;
  const float* src = from_list ? list : scores + (long long)bh * P;
  const long long n_src = from_list ? (long long)hs.cand_cnt : P;
  for_each_score<L == 1>(src, n_src, [&](float s) {
    if (L >= 1 && bin_at(hs, 0, s) != hs.bin[0]) return;
    if (L == 1 && list) {
      unsigned int pos = atomicAdd(&s_cand_n, 1u);
      if (pos < kCandStage) s_cand[pos] = s;
      else {
        pos = atomicAdd(cand_cnt + bh * (sizeof(HeadState) / sizeof(unsigned int)), 1u);
        if (pos < ccap) list[pos] = s;
      }
    }
    if (L >= 2 && bin_at(hs, 1, s) != hs.bin[1]) return;
    int b = bin_at(hs, L, s);
    atomicAdd(&s_cnt[b], 1u);
    atomicAdd(&s_w[b], unit_w ? 1.0f : pair_weight(sigma, s, smax));
    const uint32_t key = pool_key(s);
    atomicMin(&s_min[b], key);
    if (L == 1) atomicMax(&s_max[b], key);
  });
  __syncthreads();
  if (L == 1 && list) {
    const unsigned int n = min(s_cand_n, (unsigned int)kCandStage);
    if (n && threadIdx.x == 0)
      s_cand_at = atomicAdd(cand_cnt + bh * (sizeof(HeadState) / sizeof(unsigned int)), n);
    __syncthreads();
    for (unsigned int k = threadIdx.x; k < n; k += blockDim.x)
      if (s_cand_at + k < ccap) list[s_cand_at + k] = s_cand[k];
  }
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) {
    unsigned int c = s_cnt[i];
    if (c) {
      atomicAdd(&g_cnt[(long long)bh * kBins + i], c);
      atomicAdd(&g_w[(long long)bh * kBins + i], (double)s_w[i]);
      atomicMin(&g_minkey[(long long)bh * kBins + i], s_min[i]);
      if (L == 1) atomicMax(&g_maxkey[(long long)bh * kBins + i], s_max[i]);
    }
  }
}

// Level 0 sees every pair, and scores cluster: with one set of bins most lanes of a warp hit the
// same few addresses and the shared-memory atomics serialise.  Here every bin has one copy per lane
// in 32 consecutive words (a warp's updates always fall into 32 different banks), and only the
// masses are kept: the scan needs no counts at this level.
constexpr int kRep = 32;
__global__ void __launch_bounds__(512)
hist0_kernel(const float* __restrict__ scores, long long P, const HeadState* __restrict__ st, float sigma, int unit_w,
             double* __restrict__ g_w) {
  if (!grid_begin()) return;
  extern __shared__ float s_wr[];   // [kBins0][kRep]
  const int bh = blockIdx.y;
  const HeadState hs = st[bh];
  for (int i = threadIdx.x; i < kBins0 * kRep; i += blockDim.x) s_wr[i] = 0.f;
  __syncthreads();
  const float smax = key_float(hs.max_key);
  const int rep = threadIdx.x & (kRep - 1);
  for_each_score<false>(scores + (long long)bh * P, P, [&](float s) {
    atomicAdd(&s_wr[bin_at(hs, 0, s) * kRep + rep], unit_w ? 1.0f : pair_weight(sigma, s, smax));
  });
  __syncthreads();
  for (int i = threadIdx.x; i < kBins0; i += blockDim.x) {
    float w = 0.f;
#pragma unroll
    for (int r = 0; r < kRep; ++r) w += s_wr[i * kRep + ((r + i) & (kRep - 1))];
    if (w > 0.f) atomicAdd(&g_w[(long long)bh * kBins + i], (double)w);
  }
}

// One CTA (1024 threads, two bins each) per head: walk the bins from the top, find the bin in
// which the cumulative mass first reaches the target, record it and clear the histogram.
template <int L>
__global__ void __launch_bounds__(1024)
scan_kernel(HeadState* __restrict__ st, float tau, double count_target, unsigned int* __restrict__ g_cnt,
            double* __restrict__ g_w,
            uint32_t* __restrict__ g_minkey, uint32_t* __restrict__ g_maxkey, int64_t* __restrict__ k_per_head,
            float* __restrict__ cutoff_per_head, long long ccap) {
  if (!grid_begin()) return;
  __shared__ double s_wsum[32];
  __shared__ unsigned long long s_csum[32];
  __shared__ int s_cross;
  __shared__ int s_lowest;
  __shared__ uint32_t s_minkey;
  const int bh = blockIdx.x;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  HeadState hs = st[bh];
  if (L == 2 && hs.resolved) return;     // cutoff written at level 1; the histogram arrays are clear
  // element e = 0..2047 walks bins from the top: bin = 2047 - e; thread t owns e = 2t, 2t+1
  const long long hb = (long long)bh * kBins;
  const long long i0 = hb + (kBins - 1 - 2 * t), i1 = hb + (kBins - 2 - 2 * t);
  double w0 = g_w[i0], w1 = g_w[i1];
  // level 0 keeps masses only: a bin counts as occupied when its mass is positive
  unsigned long long c0 = L == 0 ? (w0 > 0.0) : g_cnt[i0], c1 = L == 0 ? (w1 > 0.0) : g_cnt[i1];
  uint32_t mk0 = 0xffffffffu, mk1 = 0xffffffffu, xk0 = 0u, xk1 = 0u;
  if (L >= 1) { mk0 = g_minkey[i0]; mk1 = g_minkey[i1]; }
  if (L == 1) { xk0 = g_maxkey[i0]; xk1 = g_maxkey[i1]; }
  // clear for the next level / next call
  g_w[i0] = 0.0; g_w[i1] = 0.0;
  if (L >= 1) { g_cnt[i0] = 0u; g_cnt[i1] = 0u; g_minkey[i0] = 0xffffffffu; g_minkey[i1] = 0xffffffffu; }
  if (L == 1) { g_maxkey[i0] = 0u; g_maxkey[i1] = 0u; }
  double wl = w0 + w1;
  unsigned long long cl = c0 + c1;
  // inclusive warp scan
  double wi = wl; unsigned long long ci = cl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    double wv = __shfl_up_sync(0xffffffffu, wi, o);
    unsigned long long cv = __shfl_up_sync(0xffffffffu, ci, o);
    if (lane >= o) { wi += wv; ci += cv; }
  }
  if (lane == 31) { s_wsum[warp] = wi; s_csum[warp] = ci; }
  if (t == 0) { s_cross = -1; s_lowest = -1; s_minkey = 0xffffffffu; }
  __syncthreads();
  if (warp == 0) {
    double wv = s_wsum[lane]; unsigned long long cv = s_csum[lane];
    double wi2 = wv; unsigned long long ci2 = cv;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      double a = __shfl_up_sync(0xffffffffu, wi2, o);
      unsigned long long b = __shfl_up_sync(0xffffffffu, ci2, o);
      if (lane >= o) { wi2 += a; ci2 += b; }
    }
    s_wsum[lane] = wi2 - wv;    // exclusive
    s_csum[lane] = ci2 - cv;
  }
  __syncthreads();
  const double w_excl = s_wsum[warp] + (wi - wl);            // mass of all elements before e = 2t
  const unsigned long long c_excl = s_csum[warp] + (ci - cl);
  __shared__ double s_total;
  if (t == 1023) s_total = w_excl + wl;
  __syncthreads();
  // unit weights (count_target >= 0): the masses are pair counts and the target is the budget itself
  if (L == 0) {
    hs.Z = s_total;
    hs.target = count_target >= 0.0 ? count_target : (double)tau * s_total;
    hs.mass_above = 0.0; hs.cnt_above = 0ull;
  }
  const double need = hs.target - hs.mass_above;    // mass still to be covered inside this level
  // crossing element: first e with inclusive mass >= need (and a non-empty bin)
  int my_cross = -1;
  if (c0 && w_excl < need && w_excl + w0 >= need) my_cross = 2 * t;
  else if (c1 && w_excl + w0 < need && w_excl + w0 + w1 >= need) my_cross = 2 * t + 1;
  if (my_cross >= 0) atomicMax(&s_cross, kBins - 1 - my_cross);      // as a bin index
  // lowest non-empty bin = fallback when rounding keeps the sum below `need`
  if (c1) atomicMax(&s_lowest, 2 * t + 1);
  else if (c0) atomicMax(&s_lowest, 2 * t);
  __syncthreads();
  int cross_bin = s_cross;
  if (cross_bin < 0) cross_bin = s_lowest >= 0 ? kBins - 1 - s_lowest : 0;
  // mass / count strictly above the crossing bin
  const int e_cross = kBins - 1 - cross_bin;
  __shared__ double s_above_w;
  __shared__ unsigned long long s_above_c;
  __shared__ uint32_t s_cross_min, s_cross_max;
  if (2 * t == e_cross) { s_above_w = w_excl; s_above_c = c_excl; s_cross_min = mk0; s_cross_max = xk0; }
  if (2 * t + 1 == e_cross) { s_above_w = w_excl + w0; s_above_c = c_excl + c0; s_cross_min = mk1; s_cross_max = xk1; }
  if (L == 2) {
    // exact cutoff: smallest key among the bins at or above the crossing bin
    uint32_t mk = 0xffffffffu;
    if (2 * t <= e_cross) mk = min(mk, mk0);
    if (2 * t + 1 <= e_cross) mk = min(mk, mk1);
    mk = __reduce_min_sync(0xffffffffu, mk);
    if (lane == 0) atomicMin(&s_minkey, mk);
  }
  __syncthreads();
  if (t == 0) {
    hs.bin[L] = cross_bin;
    // level 2 may read the list if level 1 copied the level-0 crossing bin to it in full
    if (L == 1) hs.cand_ok = (long long)hs.cand_cnt <= ccap ? 1 : 0;
    hs.mass_above += s_above_w;
    hs.cnt_above += s_above_c;
    if (L < 2) {
      hs.anchor[L + 1] = hs.inv[L] > 0.f ? hs.anchor[L] + (float)cross_bin / hs.inv[L] : hs.anchor[L];
      hs.inv[L + 1] = fminf(hs.inv[L] * (float)kBins, 1e30f);
      // one distinct score in the crossing bin: everything above it is below the target and the
      // bin reaches it, so that score is the cutoff
      if (L == 1 && tau < 1.0f && s_cross_min == s_cross_max && s_cross_min != 0xffffffffu) {
        hs.resolved = 1;
        hs.cutoff_key = s_cross_min;
        cutoff_per_head[bh] = key_float(hs.cutoff_key);
      }
    } else {
      hs.cutoff_key = s_minkey;
      if (tau >= 1.0f) hs.cutoff_key = hs.min_key;
      cutoff_per_head[bh] = key_float(hs.cutoff_key);
    }
    st[bh] = hs;
  }
}

// After minmax: level-0 anchors.
__global__ void setup_level0_kernel(HeadState* st, int BH) {
  if (!grid_begin()) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= BH) return;
  float lo = key_float(st[i].min_key), hi = key_float(st[i].max_key);
  float range = hi - lo;
  st[i].anchor[0] = lo;
  st[i].inv[0] = range > 0.f ? (float)kBins0 / range : 0.f;
  st[i].bin0_off = -lo * st[i].inv[0];
}

// mark: a CTA takes a segment of QSEG consecutive queries of one head (a contiguous run of
// QSEG * Nb scores), sets the mask bits in shared memory, counts selections per key block,
// then writes mask words, per-(segment, block) counts and the segment's pair total.
__global__ void __launch_bounds__(kSegThreads)
mark_kernel(const float* __restrict__ scores, const HeadState* __restrict__ st, int S, int Nb, int mw, int QSEG,
            int nseg, int own_sb, uint32_t* __restrict__ mask_bits, int* __restrict__ seg_cnt,
            int* __restrict__ seg_total, uint32_t* __restrict__ tmask) {
  if (!grid_begin()) return;
  extern __shared__ uint32_t sm[];
  const int TW = QSEG >> 5;                           // words of a block's column over the segment's queries
  uint32_t* s_mask = sm;                              // [QSEG][mw]
  int* s_cnt = reinterpret_cast<int*>(sm + QSEG * mw);  // [Nb]
  uint32_t* s_tm = sm + QSEG * mw + Nb;               // [TW][Nb]: the same bits, a word per 32 queries and key block
  __shared__ int s_total;
  // segments in token order over all heads: the histogram pass before ended at every head's start, which is still in L2
  const unsigned id = blockIdx.y * gridDim.x + blockIdx.x;
  const int seg = (int)(id / gridDim.y), bh = (int)(id - (unsigned)seg * gridDim.y);
  const int q0 = seg * QSEG;
  const int nq = min(QSEG, S - q0);
  const uint32_t cutoff = st[bh].cutoff_key;
  const float cut = key_float(cutoff);
  for (int i = threadIdx.x; i < QSEG * mw; i += blockDim.x) s_mask[i] = 0u;
  for (int i = threadIdx.x; i < Nb; i += blockDim.x) s_cnt[i] = 0;
  for (int i = threadIdx.x; i < Nb * TW; i += blockDim.x) s_tm[i] = 0u;
  if (threadIdx.x == 0) s_total = 0;
  __syncthreads();
  const float* base = scores + ((long long)bh * S + q0) * Nb;
  const long long n = (long long)nq * Nb;
  // (query, block) of element i of the segment by reciprocal: i < QSEG * Nb < 2^23, and (i + 0.5) / Nb is at
  // least 0.5 / Nb away from an integer, the rounding error far less (a fix-up step covers the rest)
  const float inv_nb = 1.0f / (float)Nb;
  auto mark = [&](long long i, float s) {
    if (s < cut && own_sb <= 0) return;       // the common case: one comparison, no index arithmetic (what is left: NaN, zeros, the selected)
    const bool sel = pool_key(s) >= cutoff;
    if (!sel && own_sb <= 0) return;
    const int ii = (int)i;
    int ql = (int)(((float)ii + 0.5f) * inv_nb), j = ii - ql * Nb;
    if (j < 0) { --ql; j += Nb; } else if (j >= Nb) { ++ql; j -= Nb; }     // belt and braces for huge Nb
    // own_sb > 0: a query also keeps the block it lies in (block-major position / tokens per block)
    if (sel || (q0 + ql) / own_sb == j) {
      atomicOr(&s_mask[ql * mw + (j >> 5)], 1u << (j & 31));
      atomicOr(&s_tm[(ql >> 5) * Nb + j], 1u << (ql & 31));
      atomicAdd(&s_cnt[j], 1);
    }
  };
  if ((reinterpret_cast<uintptr_t>(base) & 15u) == 0) {
    const float4* b4 = reinterpret_cast<const float4*>(base);
    long long n4 = n >> 2;
    // four independent 16-byte loads per thread in flight
    long long i = threadIdx.x;
    for (; i + 3 * (long long)blockDim.x < n4; i += 4 * (long long)blockDim.x) {
      float4 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = __ldg(b4 + i + j * (long long)blockDim.x);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long e = 4 * (i + j * (long long)blockDim.x);
        mark(e, x[j].x); mark(e + 1, x[j].y); mark(e + 2, x[j].z); mark(e + 3, x[j].w);
      }
    }
    for (; i < n4; i += blockDim.x) {
      float4 x = __ldg(b4 + i);
      mark(4 * i, x.x); mark(4 * i + 1, x.y); mark(4 * i + 2, x.z); mark(4 * i + 3, x.w);
    }
    for (long long i = (n4 << 2) + threadIdx.x; i < n; i += blockDim.x) mark(i, __ldg(base + i));
  } else {
    for (long long i = threadIdx.x; i < n; i += blockDim.x) mark(i, __ldg(base + i));
  }
  __syncthreads();
  uint32_t* gm = mask_bits + ((long long)bh * S + q0) * mw;
  int local = 0;
  for (int i = threadIdx.x; i < nq * mw; i += blockDim.x) {
    uint32_t wv = s_mask[i];
    gm[i] = wv;
    local += __popc(wv);
  }
  local = __reduce_add_sync(0xffffffffu, local);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(&s_total, local);
  int* sc = seg_cnt + ((long long)bh * nseg + seg) * Nb;
  for (int i = threadIdx.x; i < Nb; i += blockDim.x) sc[i] = s_cnt[i];
  uint32_t* tm = tmask + ((long long)bh * nseg + seg) * Nb * TW;
  for (int i = threadIdx.x; i < Nb * TW; i += blockDim.x) tm[i] = s_tm[i];
  __syncthreads();
  if (threadIdx.x == 0) seg_total[bh * nseg + seg] = s_total;
}

// offsets A: per (head, block) turn the per-segment counts into exclusive prefixes along the
// segments and record the block's total.  A CTA takes 32 blocks of a head (lane: block), a warp a run of about eight of their
// segments.  Bound by the latency of its loads: 1,680 blocks x 64 segments 3.3 us, 3,360 x 169 3.5; with a thread per block,
// eight segments after eight, 7.3 and 12.2.
__global__ void __launch_bounds__(1024)
seg_prefix_kernel(int* __restrict__ seg_cnt, int* __restrict__ kb_total, int Nb, int nseg) {
  if (!grid_begin()) return;
  __shared__ int s_sum[32][32];              // [run][block]
  const int groups = (Nb + 31) / 32, bh = blockIdx.x / groups;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_runs = blockDim.x >> 5;
  const int j = (blockIdx.x - bh * groups) * 32 + lane, per = (nseg + n_runs - 1) / n_runs;
  const int s0 = min(nseg, warp * per), s1 = j < Nb ? min(nseg, s0 + per) : s0;
  int* col = seg_cnt + (long long)bh * nseg * Nb + j;
  int run = 0;
  if (n_runs > 1) {
    int sum = 0;
#pragma unroll 8
    for (int s = s0; s < s1; ++s) sum += col[(long long)s * Nb];
    s_sum[warp][lane] = sum;
    __syncthreads();
#pragma unroll 8
    for (int w = 0; w < warp; ++w) run += s_sum[w][lane];
  }
  // eight segments per trip: their loads go out together (the stores of a trip would otherwise order them)
  for (int s = s0; s < s1; s += 8) {
    int c[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) c[k] = s + k < s1 ? col[(long long)(s + k) * Nb] : 0;
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (s + k < s1) { col[(long long)(s + k) * Nb] = run; run += c[k]; }
  }
  if (warp == n_runs - 1 && j < Nb) kb_total[(long long)bh * Nb + j] = run;
}

__global__ void __launch_bounds__(1024)
offsets_kernel(const int* __restrict__ kb_total, int* __restrict__ kb_ptr, long long n_kb,
               const int* __restrict__ seg_total, int* __restrict__ seg_qoff, long long n_seg,
               int BH, int Nb, int64_t* __restrict__ k_per_head, long long capacity,
               int* __restrict__ q_ptr_last, int32_t* __restrict__ dev_status) {
  if (!grid_begin()) return;
  __shared__ long long total_a, total_b;
  block_exclusive_scan([&](long long i) { return kb_total[i]; }, kb_ptr, n_kb, &total_a);
  block_exclusive_scan([&](long long i) { return seg_total[i]; }, seg_qoff, n_seg, &total_b);
  __syncthreads();
  // a warp per head
  for (int bh = threadIdx.x >> 5; bh < BH; bh += blockDim.x >> 5) {
    long long a = 0;
    for (int j = threadIdx.x & 31; j < Nb; j += 32) a += kb_total[(long long)bh * Nb + j];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if ((threadIdx.x & 31) == 0) k_per_head[bh] = a;
  }
  if (threadIdx.x == 0) {
    *q_ptr_last = (int)min(total_a, (long long)INT32_MAX);
    if (total_a > capacity) set_status(dev_status, VMOBA_ERR_CAPACITY);
  }
}

// fill: a CTA re-reads its segment's mask words and derives q_ptr for its queries; then thread = query walks the query's
// set bits.  The position of a pair in q_idx is that of its block's first selecting query in the segment plus the
// selecting queries below in the block's column of the segment (column words of the mark kernel, prefixed per word).  Both
// lists of a segment are put together in shared memory, by block and by query, and written out in runs; a segment with
// more pairs than the stage holds writes its entries one by one.  Bound by the latency of a CTA's steps, so that the shared
// memory is kept small: with what counts a segment's queries in 16 bits, and a stage of the rule's size where that is known, three
// CTAs share an SM.  8.2 million pairs, nine per query: 106 us (137 with 32 bits and two CTAs, 273 with a warp per key block that
// wrote q_pairs entry by entry); 0.33 million 23 (31); 12.6 million, 32 per query, beyond the stage: 155.
constexpr int kStage = 6144;
__global__ void __launch_bounds__(kSegThreads)
fill_kernel(const uint32_t* __restrict__ mask_bits, const uint32_t* __restrict__ tmask, int S, int Nb, int mw, int QSEG,
            int nseg, int* __restrict__ kb_ptr, const int* __restrict__ seg_cnt, const int* __restrict__ seg_qoff,
            int* __restrict__ q_idx, int* __restrict__ q_ptr, int* __restrict__ q_pairs, long long capacity,
            const int* __restrict__ kb_excl, const int64_t* __restrict__ k_per_head, int32_t* __restrict__ dev_status, int stage) {
  if (!grid_begin()) return;
  extern __shared__ uint32_t sm[];
  const int TW = QSEG >> 5;
  uint32_t* s_mask = sm;                                    // [QSEG][mw]
  uint32_t* s_tm = s_mask + QSEG * mw;                      // [TW][Nb] column words
  int* s_off = reinterpret_cast<int*>(s_tm + Nb * TW);      // [Nb + 1] entries in front of the block
  int* s_pos = s_off + Nb + 1;                              // [Nb] position of the segment's first entry of the block in q_idx
  int* s_pair = s_pos + Nb;                                 // [stage] q_pairs entries by query
  uint16_t* s_idx = reinterpret_cast<uint16_t*>(s_pair + stage);      // [stage] queries of the segment, by block
  uint16_t* s_pre = s_idx + stage;                          // [TW][Nb] the block's entries in front of that word
  __shared__ int s_warp[kSegThreads / 32];
  const int seg = blockIdx.x, bh = blockIdx.y;
  const int q0 = seg * QSEG;
  const int nq = min(QSEG, S - q0);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = blockDim.x >> 5;
  // exclusive scan of one value per thread over the CTA
  auto scan = [&](int v) {
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    __syncthreads();
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      int x = lane < nwarps ? s_warp[lane] : 0;
      int xi = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, xi, o);
        if (lane >= o) xi += y;
      }
      if (lane < nwarps) s_warp[lane] = xi - x;
    }
    __syncthreads();
    return s_warp[warp] + inc - v;
  };
  const uint32_t* gm = mask_bits + ((long long)bh * S + q0) * mw;
  const uint32_t* tm = tmask + ((long long)bh * nseg + seg) * Nb * TW;
  const int* sc = seg_cnt + ((long long)bh * nseg + seg) * Nb;
  for (int i = t; i < nq * mw; i += blockDim.x) s_mask[i] = gm[i];
  for (int i = t; i < Nb * TW; i += blockDim.x) s_tm[i] = tm[i];
  // kb_excl: the offsets so far are counted from the head's first pair, and this kernel adds the pairs of the heads before
  long long base = 0;
  if (kb_excl) {
    for (int h = lane; h < bh; h += 32) base += k_per_head[h];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(0xffffffffu, base, o);
  }
  for (int j = t; j < Nb; j += blockDim.x) {        // (clamped: beyond INT32_MAX is beyond every capacity)
    const long long first = kb_excl ? base + kb_excl[(long long)bh * (Nb + 1) + j] : (long long)kb_ptr[(long long)bh * Nb + j];
    s_pos[j] = (int)min(first + sc[j], (long long)INT32_MAX);
    if (kb_excl && seg == 0) kb_ptr[(long long)bh * Nb + j] = (int)min(first, (long long)INT32_MAX);
  }
  if (kb_excl && seg == 0 && bh == (int)gridDim.y - 1 && t == 0) {
    const long long all = base + k_per_head[bh];
    kb_ptr[(long long)gridDim.y * Nb] = q_ptr[(long long)gridDim.y * S] = (int)min(all, (long long)INT32_MAX);
    if (all > capacity) set_status(dev_status, VMOBA_ERR_CAPACITY);
  }
  const long long qbase = base + seg_qoff[bh * nseg + seg];
  __syncthreads();
  {
    const int per = (Nb + blockDim.x - 1) / blockDim.x, j0 = min(t * per, Nb), j1 = min(j0 + per, Nb);
    int c = 0;
    for (int j = j0; j < j1; ++j)
      for (int w = 0; w < TW; ++w) c += __popc(s_tm[w * Nb + j]);
    int run = scan(c);
    for (int j = j0; j < j1; ++j) {
      s_off[j] = run;
      for (int w = 0; w < TW; ++w) { s_pre[w * Nb + j] = (uint16_t)(run - s_off[j]); run += __popc(s_tm[w * Nb + j]); }
    }
    if (j1 == Nb && j0 < j1) s_off[Nb] = run;
  }
  int cnt = 0;
  if (t < nq)
    for (int w = 0; w < mw; ++w) cnt += __popc(s_mask[t * mw + w]);
  int mine = scan(cnt);                              // this query's next entry of q_pairs, counted from the segment's first
  const int total = s_off[Nb];
  if (t < nq) q_ptr[(long long)bh * S + q0 + t] = (int)min(qbase + mine, (long long)INT32_MAX);
  const bool staged = total <= stage;
  if (t < nq) {
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (int w = 0; w < mw; ++w) {
      uint32_t word = s_mask[t * mw + w];
      while (word) {
        const int j = 32 * w + __ffs(word) - 1;
        word &= word - 1;
        const int in_block = s_pre[warp * Nb + j] + __popc(s_tm[warp * Nb + j] & lt_mask);
        const long long pos = (long long)s_pos[j] + in_block;
        const int entry = (int)min(pos, (long long)INT32_MAX);
        if (staged) {
          s_idx[s_off[j] + in_block] = (uint16_t)t;
          s_pair[mine] = entry;
        } else if (pos < capacity) {
          q_idx[pos] = q0 + t;
          if (qbase + mine < capacity) q_pairs[qbase + mine] = entry;
        }
        ++mine;
      }
    }
  }
  if (!staged) return;
  __syncthreads();
  for (int i = t; i < total; i += blockDim.x)
    if (qbase + i < capacity && s_pair[i] < capacity) q_pairs[qbase + i] = s_pair[i];
  // a quarter warp per block's run
  for (int j = t >> 3; j < Nb; j += blockDim.x >> 3) {
    const int o0 = s_off[j], n = s_off[j + 1] - o0;
    const long long pos = s_pos[j];
    for (int i = t & 7; i < n; i += 8)
      if (pos + i < capacity) q_idx[pos + i] = q0 + s_idx[o0 + i];
  }
}

// ------------------------------------------------------------------------------------------
// Per-query ("local") rules, N_b <= 1024.  Block j = l + 32 i is bit l of mask word i.
constexpr int kLocalMaxWords = 32;

// The smallest key a warp selected in a run of rows, handed to the head's state with one atomic per run and head
// (with one atomic per row, tens of thousands of them queue on one address per head).
struct RunCutoff {
  uint32_t cut = 0xffffffffu;
  long long head = -1;
  __device__ __forceinline__ void note(HeadState* st, int lane, long long h, uint32_t c) {
    if (h != head) {
      flush(st, lane);
      head = h;
      cut = 0xffffffffu;
    }
    cut = min(cut, c);
  }
  __device__ __forceinline__ void flush(HeadState* st, int lane) {
    if (lane == 0 && head >= 0) atomicMin(&st[head].cutoff_key, cut);
  }
};

// Midpoint of a score interval for the bisections below: the arithmetic mean where that lies strictly inside (the
// scores of a row spread roughly evenly, so about log2(row length) + 4 steps separate the k-th from the next), else
// (an infinite end) the middle of the ordered bit patterns.  Returns false when nothing lies between the ends.
__device__ __forceinline__ bool split_interval(float lo, float hi, float& mid) {
  mid = 0.5f * lo + 0.5f * hi;
  if (mid > lo && mid < hi) return true;
  const uint32_t a = float_key(lo), b = float_key(hi);
  mid = key_float(a + ((b - a) >> 1));
  return mid > lo && mid < hi;
}

// The searches below compare scores as floats, which gives a NaN no place; the rule does (a NaN's key lies beyond those of the
// infinities), and every query keeps exactly k blocks.  Rows with a NaN are found by a maximum that hands NaN on, at the price
// of one that does not, and are searched on the scores' keys.  These are made from words that are never floats: as a float
// operation, setting a NaN's sign is free to return any NaN, and did.
__device__ __forceinline__ uint32_t key_of_bits(uint32_t u) {
  if (u == 0x80000000u) u = 0u;      // -0 ties with +0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// over a converged warp (sm_100: on floats as they are)
__device__ __forceinline__ float warp_max_nan(float x) {
  float d;
  asm volatile("redux.sync.max.NaN.f32 %0, %1, 0xffffffff;" : "=f"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float warp_min(float x) {
  float d;
  asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(d) : "f"(x));
  return d;
}

// Top-k per query, one warp per row: lane l holds blocks l + 32 i.  Search over the row's score range for a threshold
// that k scores reach; it usually ends early, on a threshold that exactly k scores reach, and otherwise on the k-th
// score itself, whose ties are then taken in block order.  The first probe is the threshold of the row before (rows
// of a run are neighbours of one head), the next ones step away from it by doubling amounts, and once two probes
// enclose the threshold the interval is halved.  A step is a compare and an add per word and one warp reduction: the
// kernel is bound by instruction issue.  280 blocks, k = 9, 907,200 rows (1.0 GB of scores): 0.38 ms (0.44 with the row's smallest
// score looked for as well and ten words instead of nine); plain halving
// from the row's minimum and maximum 0.80 ms, a search over the 32 key bits in an instantiation of 16 words 3.08 ms.
template <int MW>
__global__ void __launch_bounds__(256)
select_topk_kernel(const float* __restrict__ scores, int S, int Nb, int mw, int k, int own_sb,
                   uint32_t* __restrict__ mask_bits, HeadState* __restrict__ st, long long n_rows) {
  if (!grid_begin()) return;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  const uint32_t lt_mask = (1u << lane) - 1u;
  // a run of consecutive rows per warp: one head (or two), and the next row is requested while this one is worked on
  const long long per_warp = (n_rows + nwarps - 1) / nwarps;
  const long long row_begin = warp * per_warp, row_end = min(n_rows, row_begin + per_warp);
  if (row_begin >= row_end) return;
  int head = (int)(row_begin / S), pos = (int)(row_begin - (long long)head * S);
  float low = INFINITY;                 // smallest score this lane has selected in the head so far
  int on_keys = 0, first = pos;         // rows of the head that were searched on keys; the run's first row in it
  uint32_t low_key = 0xffffffffu;       // smallest cutoff of those
  auto flush = [&]() {
    uint32_t key = __reduce_min_sync(0xffffffffu, float_key(low));
    if (on_keys > 0) key = on_keys < pos - first ? min(key, low_key) : low_key;
    if (lane == 0) atomicMin(&st[head].cutoff_key, key);
    low = INFINITY;
    on_keys = first = 0;
    low_key = 0xffffffffu;
  };
  float next[MW];
  auto load_row = [&](const float* sr) {
#pragma unroll
    for (int i = 0; i < MW; ++i) next[i] = lane + 32 * i < Nb ? __ldg(sr + 32 * i) : -INFINITY;
  };
  const float* src = scores + row_begin * Nb + lane;
  load_row(src);
  uint32_t* out = mask_bits + row_begin * mw + lane;
  float t_prev = NAN;                   // threshold of the row before
  for (long long row = row_begin; row < row_end; ++row) {
    float x[MW];
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      x[i] = next[i];
      mx = max_nan(mx, x[i]);
    }
    src += Nb;
    if (row + 1 < row_end) load_row(src);
    // the row's smallest score, which only a search that does not start from the row before needs
    auto smallest = [&]() {
      float mn = INFINITY;
#pragma unroll
      for (int i = 0; i < MW; ++i)
        if (lane + 32 * i < Nb) mn = fminf(mn, x[i]);
      return warp_min(mn);
    };
    // invariant: at least k scores reach lo, fewer than k reach hi (or lo == hi)
    float hi = warp_max_nan(mx), lo = -INFINITY;
    const bool has_nan = hi != hi;
    bool exact = false;                 // exactly k scores reach lo
    if (k < Nb && !has_nan) {
      // (a block the row does not have counts as -inf, which no threshold above the row's minimum lets through)
      auto count_ge = [&](float c) {
        int n = 0;
#pragma unroll
        for (int i = 0; i < MW; ++i) n += x[i] >= c ? 1 : 0;
        return __reduce_add_sync(0xffffffffu, n);
      };
      // First step: a share of the way from the threshold before to the row's maximum, which holds more of the row the larger k is.
      // 280 blocks x 201,600 rows, whole selection, 1/8 against 1/16: rows alike, k = 9, 134 / 131 us, k = 2 112 / 113; at random, k = 9,
      // 150 / 152, k = 2 135 / 139.
      // Where the threshold before lies at or above the row's largest score, or every score reaches it, the row is unlike the one
      // before, and the search starts from the middle of its own range: rows a thousand apart 181 us (198 without; 140 blocks 136 and
      // 154, 48 blocks 113 and 134).
      float mid = t_prev, step = (k > 4 ? 0.0625f : 0.125f) * (hi - mid);
      bool below = false, above = false, go = mid < hi;
      int n = 0;
      if (go) {
        n = count_ge(mid);
        go = n < Nb;
      }
      if (!go) {
        lo = smallest();
        step = 0.015625f * (hi - lo);
        go = split_interval(lo, hi, mid);
        if (go) n = count_ge(mid);
        else if (count_ge(hi) >= k) lo = hi;        // two neighbouring values at most: is the larger one the k-th?
      }
      if (go) {
        for (;;) {
          if (n >= k) { lo = mid; below = true; } else { hi = mid; above = true; }
          if (n == k) { exact = true; break; }
          const float far = below ? lo + step : hi - step;
          if (!(below && above) && far > lo && far < hi) {
            mid = far;
            step += step;
          } else if (!split_interval(lo, hi, mid)) {
            // lo and hi are neighbours: hi itself may be the k-th score if it is the row's maximum (never probed)
            if (!above && count_ge(hi) >= k) lo = hi;
            break;
          }
          n = count_ge(mid);
        }
        t_prev = lo;
      }
    }
    uint32_t my_word = 0u;
    if (has_nan) {
      // the largest key that k blocks reach, bit by bit; blocks above it, and those at it in block order.  (The row is read
      // again word by word: rare, and with the registers of the other search it would cost that one its warps.)
      const uint32_t* sr = reinterpret_cast<const uint32_t*>(scores) + row * Nb + lane;
      auto key_at = [&](int i) { return key_of_bits(__ldg(sr + 32 * i)); };
      auto count_keys = [&](auto pred) {
        int n = 0;
#pragma unroll 1
        for (int i = 0; lane + 32 * i < Nb; ++i) n += pred(key_at(i)) ? 1 : 0;
        __syncwarp();
        return __reduce_add_sync(0xffffffffu, n);
      };
      uint32_t c = 0u;
#pragma unroll 1
      for (uint32_t bit = 0x80000000u; bit; bit >>= 1)
        if (count_keys([&](uint32_t key) { return key >= (c | bit); }) >= k) c |= bit;
      int need = k - count_keys([&](uint32_t key) { return key > c; });
#pragma unroll 1
      for (int i = 0; i < mw; ++i) {
        const bool in = lane + 32 * i < Nb;
        const uint32_t key = in ? key_at(i) : 0u;
        const uint32_t e = __ballot_sync(0xffffffffu, in && key == c);
        const bool sel = in && (key > c || (key == c && __popc(e & lt_mask) < need));
        need -= __popc(e);
        const uint32_t word = __ballot_sync(0xffffffffu, sel);
        if (lane == i) my_word = word;
      }
      low_key = min(low_key, c);
      ++on_keys;
    } else if (exact) {
#pragma unroll
      for (int i = 0; i < MW; ++i) {
        const bool sel = x[i] >= lo;
        const uint32_t word = __ballot_sync(0xffffffffu, sel);
        if (lane == i) my_word = word;
        if (sel) low = fminf(low, x[i]);
      }
    } else {
      int above = 0;
#pragma unroll
      for (int i = 0; i < MW; ++i) above += x[i] > lo ? 1 : 0;
      int need = k - __reduce_add_sync(0xffffffffu, above);      // of the scores equal to lo, in block order
#pragma unroll
      for (int i = 0; i < MW; ++i) {
        const bool in = lane + 32 * i < Nb;
        const uint32_t e = __ballot_sync(0xffffffffu, in && x[i] == lo);
        const bool sel = in && (x[i] > lo || (x[i] == lo && __popc(e & lt_mask) < need));
        need -= __popc(e);
        const uint32_t word = __ballot_sync(0xffffffffu, sel);
        if (lane == i) my_word = word;
        if (sel) low = fminf(low, x[i]);
      }
    }
    if (own_sb > 0) {                   // the query's own block, if it is to be kept
      const int own = pos / own_sb;
      if ((own >> 5) == lane) my_word |= 1u << (own & 31);
    }
    if (lane < mw) *out = my_word;
    out += mw;
    if (++pos == S) { flush(); pos = 0; ++head; }
  }
  if (pos > 0) flush();
}

// Top-k per query for rows of up to 32 blocks, one THREAD per row: the same bisection on a row held in registers, with
// no warp reductions at all (a warp per row leaves lanes idle and pays two dozen reductions for a row of 80 bytes).
// The CTA's rows are contiguous in memory and go through shared memory (odd row pitch: no bank conflicts).
// 20 blocks, k = 6, 393,120 rows: 31 us (131 us with a warp per row that took the blocks one by one, best first).
constexpr int kTopkRowThreads = 128;
template <int N>     // N_b rounded up
__global__ void __launch_bounds__(kTopkRowThreads)
select_topk_rows_kernel(const float* __restrict__ scores, int S, int Nb, int k, int own_sb,
                        uint32_t* __restrict__ mask_bits, HeadState* __restrict__ st, long long n_rows) {
  if (!grid_begin()) return;
  __shared__ float tile[kTopkRowThreads * (N | 1)];
  const int pitch = Nb | 1;
  const float inv_nb = 1.0f / (float)Nb;
  for (long long row0 = (long long)blockIdx.x * kTopkRowThreads; row0 < n_rows; row0 += (long long)gridDim.x * kTopkRowThreads) {
    const int rows = (int)min((long long)kTopkRowThreads, n_rows - row0);
    const float* src = scores + row0 * Nb;
    __syncthreads();
    for (int i = threadIdx.x; i < rows * Nb; i += kTopkRowThreads) {
      const int r = (int)(((float)i + 0.5f) * inv_nb);          // exact: i < 4096
      tile[r * pitch + (i - r * Nb)] = __ldg(src + i);
    }
    __syncthreads();
    const bool live = (int)threadIdx.x < rows;
    float x[N];
    float lo = INFINITY, hi = -INFINITY;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      x[j] = (live && j < Nb) ? tile[threadIdx.x * pitch + j] : -INFINITY;
      if (j < Nb) { lo = fminf(lo, x[j]); hi = max_nan(hi, x[j]); }
    }
    auto count_ge = [&](float c) {
      int n = 0;
#pragma unroll
      for (int j = 0; j < N; ++j) n += (j < Nb && x[j] >= c) ? 1 : 0;
      return n;
    };
    const bool on_keys = live && hi != hi;
    if (live && k < Nb && !on_keys) {
      float mid;
      if (count_ge(hi) >= k) lo = hi;
      while (split_interval(lo, hi, mid)) {
        const int n = count_ge(mid);
        if (n >= k) lo = mid; else hi = mid;
        if (n == k) break;
      }
    }
    uint32_t word = 0u, key = 0xffffffffu;      // selected blocks, smallest selected key
    if (on_keys) {
      auto key_at = [&](int j) { return key_of_bits(reinterpret_cast<const uint32_t*>(tile)[threadIdx.x * pitch + j]); };
      uint32_t c = 0u;
#pragma unroll 1
      for (uint32_t bit = 0x80000000u; bit; bit >>= 1) {
        int n = 0;
#pragma unroll 1
        for (int j = 0; j < Nb; ++j) n += key_at(j) >= (c | bit) ? 1 : 0;
        if (n >= k) c |= bit;
      }
      int need = k;
#pragma unroll 1
      for (int j = 0; j < Nb; ++j) need -= key_at(j) > c ? 1 : 0;
#pragma unroll 1
      for (int j = 0; j < Nb; ++j) {
        const uint32_t kj = key_at(j);
        if (kj > c || (kj == c && need-- > 0)) word |= 1u << j;
      }
      key = c;
    } else {
      int need = k;
#pragma unroll
      for (int j = 0; j < N; ++j) need -= (j < Nb && x[j] > lo) ? 1 : 0;
      float low = INFINITY;
#pragma unroll
      for (int j = 0; j < N; ++j) {
        const bool tie = x[j] == lo && need > 0;
        const bool sel = j < Nb && (x[j] > lo || tie);
        if (j < Nb && x[j] == lo) --need;
        if (sel) { word |= 1u << j; low = fminf(low, x[j]); }
      }
      if (live) key = float_key(low);
    }
    const long long row = row0 + threadIdx.x;
    if (live && own_sb > 0) word |= 1u << ((int)(row % S) / own_sb);
    if (live) mask_bits[row] = word;
    // smallest selected key: one atomic per warp unless its rows straddle two heads
    const int head = live ? (int)(row / S) : -1;
    const int head_lo = __reduce_min_sync(0xffffffffu, live ? head : INT32_MAX), head_hi = __reduce_max_sync(0xffffffffu, head);
    if (head_lo == head_hi) {
      const uint32_t m = __reduce_min_sync(0xffffffffu, key);
      if ((threadIdx.x & 31) == 0) atomicMin(&st[head_hi].cutoff_key, m);
    } else if (live) {
      atomicMin(&st[head].cutoff_key, key);
    }
  }
}

// Threshold per query, one warp per row: lane l holds the blocks j = l + 32 i as order-preserving keys.  Short
// selections are taken best first; otherwise the cutoff of the row, the largest key c with mass{key >= c} >= target,
// is found bit by bit from the top; blocks above it are taken, blocks tied with it in block order until the target
// is met.  A ballot IS the mask word.
// MW: compile-time bound on the mask words of a row (the loops over a lane's blocks unroll to it)
template <int MW>
__global__ void __launch_bounds__(256)
select_threshold_local_kernel(const float* __restrict__ scores, int S, int Nb, int mw, float sigma, float tau, int own_sb,
                              uint32_t* __restrict__ mask_bits, HeadState* __restrict__ st, long long n_rows) {
  if (!grid_begin()) return;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  const uint32_t lt_mask = (1u << lane) - 1u;
  // A warp takes a run of consecutive rows; the next row's scores are requested while the current row is worked on.
  const long long per_warp = (n_rows + nwarps - 1) / nwarps;
  const long long row_begin = warp * per_warp, row_end = min(n_rows, row_begin + per_warp);
  RunCutoff run;
  auto load_row = [&](long long row, uint32_t (&k)[MW]) {
    const float* sr = scores + row * Nb;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      const int j = lane + 32 * i;
      k[i] = (i < mw && j < Nb) ? float_key(__ldg(sr + j)) : 0u;     // 0 is below every real score's key
    }
  };
  uint32_t next_key[MW];
  if (row_begin < row_end) load_row(row_begin, next_key);
  for (long long row = row_begin; row < row_end; ++row) {
    const int own = own_sb > 0 ? (int)(row % S) / own_sb : -1;      // the query's own block, if it is to be kept
    const uint32_t own_bit = (own >= 0 && (own >> 5) == lane) ? 1u << (own & 31) : 0u;
    uint32_t key[MW];
    uint32_t kmax = 0u;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      key[i] = next_key[i];
      kmax = max(kmax, key[i]);
    }
    if (row + 1 < row_end) load_row(row + 1, next_key);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    double w[MW];
    const float smax = key_float(kmax);
    double z = 0.0;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      w[i] = key[i] ? (double)pair_weight(sigma, key_float(key[i]), smax) : 0.0;
      z += w[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const double target = (double)tau * z;
    auto mass_ge = [&](uint32_t c) {
      double m = 0.0;
#pragma unroll
      for (int i = 0; i < MW; ++i) m += (i < mw && key[i] >= c) ? w[i] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
      return m;
    };
    // Short selections (the usual case: a handful of blocks per query) are taken one block at a time,
    // best first, lowest block index among equals, exactly the order the rule is stated in; the
    // cumulative mass is the running sum of the winners' weights.
    {
      constexpr int kRounds = 24;
      const int rounds = tau < 1.0f ? min(kRounds, Nb) : 0;
      uint32_t taken = 0u;              // bit i: this lane's block lane + 32 i is selected
      uint32_t c_last = 0u;
      double acc = 0.0;
      bool done = false;
      for (int r = 0; r < rounds && !done; ++r) {
        uint32_t m = 0u;
#pragma unroll
        for (int i = 0; i < MW; ++i) m = max(m, ((taken >> i) & 1u) ? 0u : key[i]);
        m = __reduce_max_sync(0xffffffffu, m);
        if (m == 0u) { done = true; break; }          // every block of the row is taken
        int my_j = INT32_MAX;
#pragma unroll
        for (int i = MW - 1; i >= 0; --i)
          if (key[i] == m && !((taken >> i) & 1u)) my_j = lane + 32 * i;
        const int j_min = __reduce_min_sync(0xffffffffu, my_j);
        if ((j_min & 31) == lane) taken |= 1u << (j_min >> 5);
        c_last = m;
        acc += (double)pair_weight(sigma, key_float(m), key_float(kmax));
        done = acc >= target;
      }
      if (done) {
        uint32_t my_word = 0u;
#pragma unroll
        for (int i = 0; i < MW; ++i) {
          const uint32_t word = __ballot_sync(0xffffffffu, (taken >> i) & 1u);
          if (lane == i) my_word = word;
        }
        if (lane < mw) mask_bits[row * mw + lane] = my_word | own_bit;
        run.note(st, lane, row / S, c_last);
        continue;
      }
    }
    // General path: bitwise search for the cutoff key.
    uint32_t c = 0u;
    if (tau >= 1.0f) {
      c = 1u;                                  // everything: every real key is >= 1
    } else {
      for (int b = 31; b >= 0; --b) {
        const uint32_t cand = c | (1u << b);
        if (cand > kmax) continue;
        if (mass_ge(cand) >= target) c = cand;
      }
      if (c == 0u) c = 1u;                     // rounding kept the mass below the target: take the row
    }
    // what the blocks strictly above the cutoff already cover, and how many of the tied ones are needed
    const double above = c == 0xffffffffu ? 0.0 : mass_ge(c + 1u);
    int n_ties = 0;
    double w_tie = 0.0;
#pragma unroll
    for (int i = 0; i < MW; ++i)
      if (i < mw && key[i] == c) { n_ties += 1; w_tie = w[i]; }
    n_ties = __reduce_add_sync(0xffffffffu, n_ties);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w_tie = fmax(w_tie, __shfl_xor_sync(0xffffffffu, w_tie, o));
    int need = (tau >= 1.0f || !(w_tie > 0.0)) ? n_ties : (int)ceil((target - above) / w_tie);
    need = max(1, min(need, n_ties));
    int seen = 0;
    uint32_t my_word = 0u;
#pragma unroll
    for (int i = 0; i < MW; ++i) {
      if (i < mw) {
        const bool eq = key[i] == c;
        const uint32_t e = __ballot_sync(0xffffffffu, eq);
        const bool sel = key[i] > c || (eq && seen + __popc(e & lt_mask) < need);
        const uint32_t word = __ballot_sync(0xffffffffu, sel);
        if (lane == i) my_word = word;
        seen += __popc(e);
      }
    }
    if (lane < mw) mask_bits[row * mw + lane] = my_word | own_bit;
    run.note(st, lane, row / S, c);
  }
  run.flush(st, lane);
}

__global__ void local_cutoff_kernel(const HeadState* __restrict__ st, float* __restrict__ cutoff_per_head, int BH) {
  if (!grid_begin()) return;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < BH) cutoff_per_head[i] = key_float(st[i].cutoff_key);
}

// The mark pass of the local rules: the mask words exist already; a segment's CTA derives the
// per-block columns, the per-(segment, block) counts and the segment's pair total from them.
__global__ void __launch_bounds__(kSegThreads)
mark_from_mask_kernel(const uint32_t* __restrict__ mask_bits, int S, int Nb, int mw, int QSEG, int nseg,
                      int* __restrict__ seg_cnt, int* __restrict__ seg_total, uint32_t* __restrict__ tmask) {
  if (!grid_begin()) return;
  extern __shared__ uint32_t sm[];
  const int TW = QSEG >> 5;
  int* s_cnt = reinterpret_cast<int*>(sm);            // [Nb]
  uint32_t* s_tm = sm + Nb;                           // [TW][Nb]
  __shared__ int s_total;
  const int seg = blockIdx.x, bh = blockIdx.y;
  const int q0 = seg * QSEG;
  const int nq = min(QSEG, S - q0);
  for (int i = threadIdx.x; i < Nb; i += blockDim.x) s_cnt[i] = 0;
  for (int i = threadIdx.x; i < Nb * TW; i += blockDim.x) s_tm[i] = 0u;
  if (threadIdx.x == 0) s_total = 0;
  __syncthreads();
  const uint32_t* gm = mask_bits + ((long long)bh * S + q0) * mw;
  int local = 0;
  for (int i = threadIdx.x; i < nq * mw; i += blockDim.x) {
    uint32_t word = gm[i];
    const int ql = i / mw, wj = i - ql * mw;
    local += __popc(word);
    while (word) {
      const int j = 32 * wj + __ffs(word) - 1;
      word &= word - 1;
      atomicOr(&s_tm[(ql >> 5) * Nb + j], 1u << (ql & 31));
      atomicAdd(&s_cnt[j], 1);
    }
  }
  local = __reduce_add_sync(0xffffffffu, local);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(&s_total, local);
  __syncthreads();
  int* sc = seg_cnt + ((long long)bh * nseg + seg) * Nb;
  for (int i = threadIdx.x; i < Nb; i += blockDim.x) sc[i] = s_cnt[i];
  uint32_t* tm = tmask + ((long long)bh * nseg + seg) * Nb * TW;
  for (int i = threadIdx.x; i < Nb * TW; i += blockDim.x) tm[i] = s_tm[i];
  if (threadIdx.x == 0) seg_total[bh * nseg + seg] = s_total;
}

// ------------------------------------------------------------------------------------------
// Small pools: one cluster of up to eight CTAs per head does the whole of the selection up to the offsets of its own pairs;
// fill_kernel adds the pairs of the heads before.  Two launches take the place of eleven, each of which waited two to five
// microseconds for the one before it: 12 heads x 1,872 queries x 8 blocks 40 -> 18 us, x 13,440 x 16 57 -> 38.  A CTA takes
// whole segments of QSEG queries and keeps their scores in shared memory.  The search is the one of the kernels above in other
// steps, bound by the latency of each:
//   * 32 bins of the head's range, a set for every thread (one bank each, plain additions; with 512 bins shared by the
//     CTA, the compare-and-swap loops that fp32 additions in shared memory are took 14 us for 27,000 scores);
//   * the scores of the crossing bin, put together in a list, in a bin of it per thread (again, where they are alike);
//   * the up to kPoolFinal scores of the crossing bin of those, each against all others.
// What the CTAs of a cluster have to tell one another they write into each other's shared memory ahead of a barrier (the
// finer bins are read from there), and all of them come to the same state.
// SRC = kPoolMask: the per-query rules, whose mask words exist already.
enum PoolSrc { kPoolScores, kPoolMask };
constexpr int kPoolCtas = 8;                  // what every device schedules as one cluster
constexpr int kPoolBins0 = 32, kPoolLevels = 3, kPoolFinal = 256;
constexpr int kPoolSmemMax = 224 * 1024;
// A second (fourth, eighth) CTA shares a head from more than 4,096 scores per CTA on, as long as there is an SM for each: 12 heads x
// 15,000 scores 19.0 us (one CTA 25), x 33,000 21.2 (16,384 per CTA 26; whole selection, 37.7 by the passes over the matrix).
constexpr long long kPoolSlice = 4096;
constexpr long long kPoolSecond[2] = {28672, 22528};      // scores per CTA of a cluster of four, of eight: see pool_plan()
// Up to 2,048 scores a CTA has 256 threads, else 512: a step that every thread takes costs their number (x 1,024 scores 14.8
// us with 256, 15.2 with 512, 16.7 with 1,024; x 15,000 in two CTAs 24.1, 21.6, 23.0).
constexpr long long kPoolShort = 2048;
// bytes of shared memory: the first bins of T threads; then, in their place, masses and counts of the levels' bins and the list
constexpr int kPoolFront = kPoolBins0 * 4;      // (per thread)

struct PoolArgs {
  const float* scores;
  const float* range;          // or null: looked for here
  const HeadState* state;      // kPoolMask: smallest selected key of each head
  int S, Nb, mw, QSEG, nseg, segs_per, own_sb, unit_w;
  float sigma, tau;
  double count_target;
  uint32_t* mask_bits;
  uint32_t* tmask;
  int* seg_cnt;
  int* seg_qoff;
  int* kb_excl;                // [BH][Nb + 1] pairs of the head in front of each block
  int64_t* k_per_head;
  float* cutoff_per_head;
};

// exclusive sum over the threads of the CTA (s_warp: a word per warp; the caller keeps calls apart by barriers)
template <typename T>
__device__ __noinline__ T pool_exclusive(T x, T* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  T before = lane < warp ? s_warp[lane] : T(0);      // (at most sixteen warps)
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o, 16);
  return __shfl_sync(0xffffffffu, before, 0) + (inc - x);
}

// The search for a head's cutoff among the scores src[0 .. n) of every CTA of a cluster, in shared memory, which lie in [lo, lo +
// span].  target(total): the mass to be covered, given that of all these scores.  front: kPoolFront * T bytes of shared memory.
template <int T, typename Meet, typename Weight, typename Target>
__device__ __forceinline__ uint32_t pool_search(cooperative_groups::cluster_group& cluster, Meet meet, unsigned char* front, const float* src,
                                                int n, float lo, float span, Weight weight, Target target) {
  constexpr int kLevelBytes = 8 * T, kList = (kPoolFront * T - kPoolLevels * kLevelBytes) / 4;
  __shared__ double s_w0[kPoolCtas][kPoolBins0], s_dsum[32], s_above;
  __shared__ uint32_t s_key[kPoolCtas][2], s_final[kPoolFinal], s_best, s_least;
  __shared__ int s_crossed, s_lowest, s_n, s_at, s_k, s_cross[kPoolLevels];
  __shared__ int s_sum[32], s_listed;
  __shared__ float s_anchor[kPoolLevels], s_inv[kPoolLevels];
  uint32_t cutoff = 0u;
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  float* s_own = reinterpret_cast<float*>(front);        // [kPoolBins0][threads]
#pragma unroll
  for (int b = 0; b < kPoolBins0 / 4; ++b) reinterpret_cast<float4*>(s_own)[b * T + t] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const float inv0 = span > 0.f ? (float)kPoolBins0 / span : 0.f, off0 = -lo * inv0;
  // smallest and largest of a value over the cluster
  auto exchange = [&](uint32_t& least, uint32_t& most) {
    least = __reduce_min_sync(0xffffffffu, least);
    most = __reduce_max_sync(0xffffffffu, most);
    if (lane == 0) { atomicMin(&s_least, least); atomicMax(&s_best, most); }
    __syncthreads();
    if (t < C) {
      uint32_t* to = cluster.map_shared_rank(s_key[rank], t);
      to[0] = s_least; to[1] = s_best;
    }
    meet();
    for (int c = 0; c < C; ++c) { least = min(least, s_key[c][0]); most = max(most, s_key[c][1]); }
  };
  auto stream = [&](const float* from, int count, auto f) {
    int i = t;
#pragma unroll 4
    for (; i < count; i += T) f(from[i]);
  };
  // ---- the first bins: floor(s * inv0 + off0) by an addition that rounds down, NaN to bin 0
  stream(src, n, [&](float s) {
    const float x = fminf(fmaxf(fmaf(s, inv0, off0), 0.f), (float)(kPoolBins0 - 1));
    const int b = __float_as_int(__fadd_rd(x, 8388608.f)) & (kPoolBins0 - 1);
    s_own[b * T + t] += weight(s);
  });
  __syncthreads();
  {
    constexpr int kMine = kPoolBins0 / (T / 32);       // bins of a warp, worked out side by side
    double x[kMine];
#pragma unroll
    for (int m = 0; m < kMine; ++m) {
      const float* own = s_own + (warp + m * (T / 32)) * T + lane;
      float w = 0.f;
#pragma unroll
      for (int r = 0; r < T / 32; ++r)
        if (own[32 * r] > 0.f) w += own[32 * r];
      x[m] = (double)w;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int m = 0; m < kMine; ++m) x[m] += __shfl_xor_sync(0xffffffffu, x[m], o);
    if (lane < C)
#pragma unroll
      for (int m = 0; m < kMine; ++m) cluster.map_shared_rank(s_w0[rank], lane)[warp + m * (T / 32)] = x[m];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 2 * kPoolLevels; ++i) reinterpret_cast<uint32_t*>(front)[i * T + t] = 0u;
  meet();
  double need;                           // mass still to be covered from the crossing bin down
  int cross0;
  {
    double x = 0.0;                      // lane l: bin 31 - l
    for (int c = 0; c < C; ++c) x += s_w0[c][kPoolBins0 - 1 - lane];
    double inc = x;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
      const double v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const double total = __shfl_sync(0xffffffffu, inc, 31), excl = inc - x;
    need = target(total);
    const unsigned int hit = __ballot_sync(0xffffffffu, x > 0.0 && excl < need && inc >= need);
    const unsigned int occupied = __ballot_sync(0xffffffffu, x > 0.0);
    const int e = hit ? __ffs(hit) - 1 : occupied ? 31 - __clz(occupied) : kPoolBins0 - 1;
    cross0 = kPoolBins0 - 1 - e;
    need -= __shfl_sync(0xffffffffu, excl, e);
  }
  {
    // ---- the list of the crossing bin's scores (the last bin has no end), if it has room for them
    const float y_lo = (float)cross0, y_hi = cross0 == kPoolBins0 - 1 ? NAN : (float)(cross0 + 1);
    auto inside = [&](float s) {
      const float y = fmaf(s, inv0, off0);
      return (cross0 == 0 || y >= y_lo) && !(y >= y_hi);
    };
    float* s_list = reinterpret_cast<float*>(front + kPoolLevels * kLevelBytes);
    int mine = 0;
    stream(src, n, [&](float s) { mine += inside(s) ? 1 : 0; });
    int at = pool_exclusive(mine, s_sum);
    if (t == T - 1) s_listed = at + mine;
    if (mine && at + mine <= kList)
      stream(src, n, [&](float s) { if (inside(s)) s_list[at++] = s; });
    if (t == 0) {
      s_anchor[0] = inv0 > 0.f ? lo + (float)cross0 / inv0 : lo;
      s_inv[0] = fminf(inv0 * (float)T, 1e30f);
    }
    __syncthreads();
    const bool over = s_listed > kList;
    const float* in_bin = over ? src : s_list;
    const int n_in = over ? n : s_listed;
    auto bin_of = [&](int L, float s) {
      const float x = (s - s_anchor[L]) * s_inv[L];
      return x > 0.f ? (int)fminf(x, (float)(T - 1)) : 0;
    };
    auto each = [&](int levels, auto f) {          // the scores inside the crossing bins of so many levels
      auto look = [&](float s) {
        bool in = !over || inside(s);
#pragma unroll 1
        for (int l = 0; l < levels; ++l) in = in && bin_of(l, s) == s_cross[l];
        if (in) f(s);
      };
#pragma unroll 1
      for (int i = t; i < n_in; i += T) look(in_bin[i]);
    };
    // ---- a bin of it per thread; thread t looks after bin T - 1 - t
#pragma unroll 1
    for (int L = 0; L < kPoolLevels; ++L) {
      float* w = reinterpret_cast<float*>(front + L * kLevelBytes);
      unsigned int* cnt = reinterpret_cast<unsigned int*>(w + T);
      each(L, [&](float s) {
        const int b = bin_of(L, s);
        // lanes that are at the same score go in one update: scores that are all alike would queue for one bin
        const uint32_t key = pool_key(s);
        const unsigned int here = __activemask();
        int lanes = 1;
        if (__reduce_min_sync(here, key) == __reduce_max_sync(here, key)) {
          if (lane != __ffs(here) - 1) return;
          lanes = __popc(here);
        }
        atomicAdd(&cnt[b], (unsigned int)lanes);
        atomicAdd(&w[b], (float)lanes * weight(s));
      });
      if (t == 0) { s_crossed = INT32_MAX; s_lowest = -1; s_k = 0; s_n = 0; s_best = 0u; s_least = 0xffffffffu; s_above = 0.0; }
      meet();
      const int b = T - 1 - t;
      double x = 0.0;
      int k = 0, before = 0;
#pragma unroll
      for (int c0 = 0; c0 < kPoolCtas; c0 += 4) {
        if (c0 >= C) break;
        unsigned int ks[4];
        float ws[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int from = min(c0 + c, C - 1);
          ks[c] = *cluster.map_shared_rank(cnt + b, from);
          ws[c] = *cluster.map_shared_rank(w + b, from);
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (c0 + c < C) {
            x += (double)ws[c];
            if (c0 + c < rank) before += (int)ks[c];
            k += (int)ks[c];
          }
      }
      const double excl = pool_exclusive(x, s_dsum);
      if (k && excl < need && excl + x >= need) atomicMin(&s_crossed, t);
      const unsigned int some = __ballot_sync(0xffffffffu, k != 0);
      if (lane == 0 && some) atomicMax(&s_lowest, 32 * warp + 31 - __clz(some));      // where rounding keeps the sum below `need`
      __syncthreads();
      const int e = s_crossed != INT32_MAX ? s_crossed : s_lowest >= 0 ? s_lowest : T - 1;
      if (t == e) {
        s_above = excl; s_k = k; s_at = before; s_cross[L] = T - 1 - e;
        if (L + 1 < kPoolLevels) {
          s_anchor[L + 1] = s_inv[L] > 0.f ? s_anchor[L] + (float)(T - 1 - e) / s_inv[L] : s_anchor[L];
          s_inv[L + 1] = fminf(s_inv[L] * (float)T, 1e30f);
        }
      }
      __syncthreads();
      need -= s_above;
      const int K = s_k;
      if (K <= kPoolFinal) {
        // ---- the last few, each against all others: the largest key whose mass and that of those above reach the target
        each(L + 1, [&](float s) {
          const int to = s_at + atomicAdd(&s_n, 1);
          const uint32_t key = pool_key(s);
          for (int c = 0; c < C; ++c) cluster.map_shared_rank(s_final, c)[to] = key;
        });
        meet();
        int G = 32;                      // threads per score
        while (G * K > T) G >>= 1;
        const int i = t / G, r = t & (G - 1);
        double mass = 0.0;
        const uint32_t key = i < K ? s_final[i] : 0u;
        if (i < K)
#pragma unroll 1
          for (int j = r; j < K; j += G) {
            const uint32_t other = s_final[j];
            if (other >= key) mass += (double)weight(key_float(other));
          }
#pragma unroll 1
        for (int o = G >> 1; o > 0; o >>= 1) mass += __shfl_xor_sync(0xffffffffu, mass, o);
        const uint32_t best = __reduce_max_sync(0xffffffffu, i < K && mass >= need ? key : 0u);
        const uint32_t least = __reduce_min_sync(0xffffffffu, i < K ? key : 0xffffffffu);
        if (lane == 0) {
          if (best) atomicMax(&s_best, best);
          atomicMin(&s_least, least);
        }
        __syncthreads();
        cutoff = s_best ? s_best : s_least;
        break;
      }
      uint32_t kmin = 0xffffffffu, kmax = 0u;
      each(L + 1, [&](float s) {
        kmin = min(kmin, pool_key(s));
        kmax = max(kmax, pool_key(s));
      });
      exchange(kmin, kmax);
      cutoff = kmin;
      if (kmin == kmax) break;
    }
  }
  return cutoff;
}

template <PoolSrc SRC, int T>
__global__ void __launch_bounds__(T, 1)
select_pool_kernel(const PoolArgs a) {
  if (!grid_begin()) return;
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // a barrier of the cluster (a head with one CTA: its own, at a third of the price)
  auto meet = [&]() { if (cluster.num_blocks() > 1) cluster.sync(); else __syncthreads(); };
  // before the first look into another CTA's shared memory: all of them have started
  auto all_there = []() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); };
  constexpr int kFront = SRC == kPoolScores ? kPoolFront * T : 0;
  extern __shared__ __align__(16) unsigned char pool_smem[];
  __shared__ int s_pairs[kPoolCtas], s_mine;      // pairs of the cluster's CTAs
  __shared__ int s_sum[32];
  if (threadIdx.x == 0) s_mine = 0;
  const int C = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), bh = (int)blockIdx.x / C;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int Nb = a.Nb, mw = a.mw, TW = a.QSEG >> 5;
  const int seg0 = rank * a.segs_per, segs = max(0, min(a.segs_per, a.nseg - seg0));      // (none, for the last CTAs of some)
  const int q0 = seg0 * a.QSEG, nq = max(0, min(a.S - q0, a.segs_per * a.QSEG));
  const int n = nq * Nb;
  int* s_tot = reinterpret_cast<int*>(pool_smem + kFront);      // [C][Nb] pairs of the CTAs
  int* s_seg = s_tot + C * Nb;                                  // [segs_per][Nb]
  int* s_segp = s_seg + a.segs_per * Nb;                        // [segs_per] pairs of a segment
  for (int i = t; i < a.segs_per * (Nb + 1); i += T) s_seg[i] = 0;      // (s_segp follows)
  uint32_t* gmask = a.mask_bits + ((long long)bh * a.S + q0) * mw;
  uint32_t* gtm = a.tmask + ((long long)bh * a.nseg + seg0) * TW * Nb;      // [segs][TW][Nb]

  uint32_t cutoff = 0u;
  float* s_src = nullptr;
  if constexpr (SRC == kPoolScores) {
    __shared__ uint32_t s_key[kPoolCtas][2], s_least, s_most;
    s_src = reinterpret_cast<float*>(pool_smem + kFront + ((4 * (C * Nb + a.segs_per * (Nb + 1)) + 15) & ~15));
    uint32_t min_key = 0xffffffffu, max_key = 0u;
    if (t == 0) { s_least = min_key; s_most = max_key; }
    if (a.range) { min_key = float_key(__ldg(a.range + 2 * bh)); max_key = float_key(__ldg(a.range + 2 * bh + 1)); }
    {
      const float* g_src = a.scores + ((long long)bh * a.S + q0) * Nb;
      if ((reinterpret_cast<uintptr_t>(g_src) & 15u) == 0) {
        const int n4 = n >> 2;
#pragma unroll 8
        for (int i = t; i < n4; i += T) reinterpret_cast<float4*>(s_src)[i] = __ldg(reinterpret_cast<const float4*>(g_src) + i);
        if (t < n - (n4 << 2)) s_src[(n4 << 2) + t] = __ldg(g_src + (n4 << 2) + t);
      } else {
#pragma unroll 8
        for (int i = t; i < n; i += T) s_src[i] = __ldg(g_src + i);
      }
    }
    all_there();
    if (!a.range) {
      __syncthreads();
#pragma unroll 2
      for (int i = t; i < n; i += T) {
        const uint32_t key = pool_key(s_src[i]);
        min_key = min(min_key, key);
        max_key = max(max_key, key);
      }
      min_key = __reduce_min_sync(0xffffffffu, min_key);
      max_key = __reduce_max_sync(0xffffffffu, max_key);
      if (lane == 0) { atomicMin(&s_least, min_key); atomicMax(&s_most, max_key); }
      __syncthreads();
      if (t < C) {
        uint32_t* to = cluster.map_shared_rank(s_key[rank], t);
        to[0] = s_least; to[1] = s_most;
      }
      meet();
      for (int c = 0; c < C; ++c) { min_key = min(min_key, s_key[c][0]); max_key = max(max_key, s_key[c][1]); }
    }
    const float lo = key_float(min_key), smax = key_float(max_key);
    const bool unit_w = a.unit_w != 0;
    cutoff = min_key;                      // everything, where tau = 1
    if (a.tau < 1.0f) {
      cutoff = pool_search<T>(cluster, meet, pool_smem, s_src, n, lo, smax - lo,
                              [&](float s) { return unit_w ? 1.0f : pair_weight(a.sigma, s, smax); },
                              [&](double total) { return a.count_target >= 0.0 ? a.count_target : (double)a.tau * total; });
    } else {
      __syncthreads();
    }
    if (rank == 0 && t == 0) a.cutoff_per_head[bh] = key_float(cutoff);
  } else {
    if (rank == 0 && t == 0) a.cutoff_per_head[bh] = key_float(a.state[bh].cutoff_key);
    __syncthreads();
    all_there();
  }

  // ---- mark: a warp takes 32 queries x 32 blocks at a time.  Lane = query puts its mask word together (the lanes start at
  // different blocks: rows a power of two apart would meet in a few banks); ballots of its bits are the column words.
#pragma unroll 1
  for (int sg = 0; sg < segs; ++sg)
#pragma unroll 1
    for (int g = sg * TW + ((warp - sg * TW) & (T / 32 - 1)); g < (sg + 1) * TW; g += T / 32) {
      const int rows = nq - g * 32;         // (< 1 beyond the head's last query)
      const bool live = lane < rows;
#pragma unroll 1
      for (int i = 0; i < mw; ++i) {
        const int width = min(32, Nb - 32 * i);
        uint32_t word = 0u, col = 0u;
        uint32_t* to = gmask + (g * 32 + lane) * mw + i;
        if constexpr (SRC == kPoolMask) {
          if (live) word = *to;
        } else {
          if (live) {
            const float* s = s_src + (g * 32 + lane) * Nb + 32 * i;
            int j = lane & ((1 << (31 - __clz(width))) - 1);
#pragma unroll 4
            for (int r = 0; r < width; ++r) {
              if (pool_key(s[j]) >= cutoff) word |= 1u << j;
              if (++j == width) j = 0;
            }
            if (a.own_sb > 0) {             // the query's own block, if it is to be kept
              const int own = (q0 + g * 32 + lane) / a.own_sb;
              if ((own >> 5) == i) word |= 1u << (own & 31);
            }
            *to = word;
          }
          __syncwarp();
        }
#pragma unroll 4
        for (int r = 0; r < width; ++r) {
          const uint32_t c = __ballot_sync(0xffffffffu, (word >> r) & 1u);
          if (lane == r) col = c;
        }
        if (lane < width) {
          gtm[g * Nb + 32 * i + lane] = col;
          if (col) atomicAdd(&s_seg[sg * Nb + 32 * i + lane], __popc(col));
        }
      }
    }
  __syncthreads();
  // ---- places of the segments' pairs, from the head's first pair on: by key block, by query, and of the blocks
  int pairs = 0;
  for (int j = t; j < Nb; j += T) {
    int sum = 0;
    for (int sg = 0; sg < segs; ++sg) {
      const int x = s_seg[sg * Nb + j];
      if (x) atomicAdd(&s_segp[sg], x);
      sum += x;
    }
    for (int c = 0; c < C; ++c) cluster.map_shared_rank(s_tot + rank * Nb, c)[j] = sum;
    pairs += sum;
  }
  if (pairs) atomicAdd(&s_mine, pairs);
  __syncthreads();
  if (t < C) cluster.map_shared_rank(s_pairs, t)[rank] = s_mine;
  meet();      // (what is read from here on is the CTA's own: it may leave when it is done)
  const int per = (Nb + T - 1) / T, j0 = min(t * per, Nb), j1 = min(j0 + per, Nb);
  int run_all = 0;
  for (int j = j0; j < j1; ++j) {
    int run = 0;
    for (int c = 0; c < C; ++c) {
      const int x = s_tot[c * Nb + j];
      if (c < rank) run += x;
      run_all += x;
    }
    for (int sg = 0; sg < segs; ++sg) {
      a.seg_cnt[((long long)bh * a.nseg + seg0 + sg) * Nb + j] = run;
      run += s_seg[sg * Nb + j];
    }
  }
  if (t == T - 1) {
    int run = 0;
    for (int c = 0; c < rank; ++c) run += s_pairs[c];
    for (int sg = 0; sg < segs; ++sg) {
      a.seg_qoff[bh * a.nseg + seg0 + sg] = run;
      run += s_segp[sg];
    }
  }
  if (rank == 0) {
    int at = pool_exclusive(run_all, s_sum);
    int* kb = a.kb_excl + (long long)bh * (Nb + 1);
    for (int j = j0; j < j1; ++j) {
      kb[j] = at;
      for (int c = 0; c < C; ++c) at += s_tot[c * Nb + j];
    }
    if (t == T - 1) a.k_per_head[bh] = at;
  }
}

// Row normalisation for the second reading of Eq. 4: out[i][j] = sigma * s[i][j] - logsumexp_j(sigma * s[i][:]),
// the logarithm of S times the pair's probability when every query is normalised on its own.  One
// warp per query row; the head-wide quantile search then runs on `out` with unit temperature.
__global__ void __launch_bounds__(256)
rownorm_kernel(const float* __restrict__ scores, float* __restrict__ out, int Nb, float sigma, long long n_rows) {
  if (!grid_begin()) return;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long row = warp; row < n_rows; row += nwarps) {
    const float* sr = scores + row * Nb;
    float mx = -INFINITY;
    for (int j = lane; j < Nb; j += 32) mx = fmaxf(mx, sigma * __ldg(sr + j));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float z = 0.f;
    for (int j = lane; j < Nb; j += 32) z += expf(sigma * __ldg(sr + j) - mx);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
    const float lse = mx + logf(z);
    float* orow = out + row * Nb;
    for (int j = lane; j < Nb; j += 32) orow[j] = sigma * __ldg(sr + j) - lse;
  }
}

static int seg_queries(int mw) {
  int q = 4096 / mw;            // keep the shared mask tile <= 16 KB
  q = q / 32 * 32;
  if (q > kSegThreads) q = kSegThreads;
  if (q < 32) q = 32;
  return q;
}

// How select_pool_kernel divides a head (C = 0: it does not take it, the passes over the matrix do).
//
// One CTA of 512 threads or two of 256 fit an SM by their registers, and 148 SMs hold 148 clusters of one, 74 of two, 33 of four and 15
// of eight (a cluster lies within one GPC).  What runs in one wave is taken (us, small route / passes: 15 heads x 131,072 scores
// 34 / 58, x 299,776 52 / 71; 148 x 19,968 38 / 75), and of what takes more
//   * as many CTAs as shared memory and 2,048 threads per SM would let run: 296 heads x 1,024 scores 21 / 60, 740, in three waves,
//     38 / 95, 296 x 7,488 48 / 83;
//   * a second wave of clusters of four or eight while their slices are short (kPoolSecond): 18 heads x 162,816 60 / 65, but 16 x
//     215,040 71 / 67 and x 299,776 83 / 73; 37 x 107,520 69 / 73, but x 149,760 83 / 79.
// The per-query rules' masks (`scores` false) have no slice to search: 18 heads x 299,776 49 / 50, 37 x 149,760 49 / 52.
struct PoolPlan { int C, T, QSEG, nseg, segs_per; size_t smem, smem_mask; };
static PoolPlan pool_plan(const Dims& D, bool scores) {
  PoolPlan p = {};
  const long long P = (long long)D.S * D.Nb;
  if (P > kPoolCtas * (long long)kPoolSmemMax / 4 || D.Nb > 1024) return p;
  auto divide = [&](int C) {
    const int most = seg_queries(D.mask_words);
    p.C = C;
    p.segs_per = (int)(((long long)D.S + (long long)most * C - 1) / ((long long)most * C));
    p.QSEG = (D.S + C * p.segs_per - 1) / (C * p.segs_per);
    p.QSEG = (p.QSEG + 31) / 32 * 32;
    p.nseg = (D.S + p.QSEG - 1) / p.QSEG;
    p.segs_per = (p.nseg + C - 1) / C;
    p.smem_mask = 4 * ((size_t)C * D.Nb + (size_t)p.segs_per * (D.Nb + 1)) + 16;
    p.T = P / C <= kPoolShort ? 256 : 512;
    p.smem = kPoolFront * p.T + p.smem_mask + 4 * (size_t)p.segs_per * p.QSEG * D.Nb;
    return p.smem <= (size_t)kPoolSmemMax;
  };
  auto takes = [&](int C) {
    const long long per_sm = std::min<long long>((227 * 1024) / (long long)(p.smem + 5 * 1024), 2048 / p.T), sms = sm_count();
    const long long whole = C == 8 ? sms * 5 / 6 : C == 4 ? sms * 9 / 10 : sms;      // SMs that clusters of C come to fill
    if (scores && C >= 4 && (long long)D.BH * C > whole && P / C > kPoolSecond[C == 8]) return false;
    return (long long)D.BH * C <= sms * per_sm;
  };
  int C = 1;
  while (C < kPoolCtas && P / C > kPoolSlice && (long long)D.BH * 2 * C <= sm_count()) C *= 2;
  while (!divide(C)) {
    if (C == kPoolCtas) { p.C = 0; return p; }
    C *= 2;
  }
  if (!takes(C)) p.C = 0;
  return p;
}

struct SelectWs {
  HeadState* state;
  unsigned int* g_cnt;
  double* g_w;
  uint32_t* g_minkey;
  uint32_t* g_maxkey;
  uint32_t* tmask;
  int* seg_cnt;
  int* seg_total;
  int* seg_qoff;
  int* kb_total;        // pairs of a block; from select_pool_kernel: [BH][Nb + 1] pairs of the head in front of it
  PoolPlan pool;
  int QSEG, nseg;       // queries of a segment, segments of a head
  float* cand;          // [BH][ccap] scores copied aside by the level-0 pass (optional: the last slice)
  long long ccap;
  size_t base_bytes;    // without the candidate lists
  size_t bytes;
  Guards guards;
};

// Room for the list of one head: the pairs of one of the 512 level-0 bins.
static long long cand_capacity(const Dims& D) {
  const long long P = (long long)D.S * D.Nb;
  return std::max<long long>(4096, ((P / 32 + 3) / 4) * 4);
}

static SelectWs lay_out_select(const Dims& D, const PoolPlan& pool, void* ws) {
  SelectWs w;
  Carver c(ws);
  w.pool = pool;
  const int QSEG = w.QSEG = w.pool.C ? w.pool.QSEG : seg_queries(D.mask_words);
  const long long nseg = w.nseg = (D.S + QSEG - 1) / QSEG;
  w.state = c.take<HeadState>(D.BH);
  const size_t bins = w.pool.C ? 0 : (size_t)D.BH * kBins;      // (select_pool_kernel keeps its bins to itself)
  w.g_cnt = c.take<unsigned int>(bins);
  w.g_w = c.take<double>(bins);
  w.g_minkey = c.take<uint32_t>(bins);
  w.g_maxkey = c.take<uint32_t>(bins);
  w.tmask = c.take<uint32_t>((size_t)D.BH * nseg * D.Nb * (QSEG >> 5));
  w.seg_cnt = c.take<int>((size_t)D.BH * nseg * D.Nb);
  w.seg_total = c.take<int>((size_t)D.BH * nseg);
  w.seg_qoff = c.take<int>((size_t)D.BH * nseg + 1);
  w.kb_total = c.take<int>((size_t)D.BH * (D.Nb + (w.pool.C ? 1 : 0)));
  w.base_bytes = c.total();
  w.ccap = w.pool.C ? 0 : cand_capacity(D);
  w.cand = c.take<float>((size_t)D.BH * w.ccap);
  w.bytes = c.total();
  w.guards = c.guards;
  return w;
}

// The scratch that a call needs is that of the passes over the matrix, whichever route it takes: how many heads go to
// select_pool_kernel depends on the GPU, and a size that was asked for on one (or without one) holds on another.  The small route
// lives in the same bytes, without the bins, which leaves it room to spare.
static SelectWs carve_select(const Dims& D, bool scores, void* ws) {
  const SelectWs passes = lay_out_select(D, PoolPlan(), ws);
  const PoolPlan plan = pool_plan(D, scores);
  if (!plan.C) return passes;
  SelectWs w = lay_out_select(D, plan, ws);
  if (w.bytes > passes.base_bytes) return passes;
  w.base_bytes = passes.base_bytes;
  w.bytes = passes.bytes;
  return w;
}

size_t select_ws_bytes(const Dims& D) { return lay_out_select(D, PoolPlan(), nullptr).bytes; }
// the least the selection can work with (no candidate lists: levels 1 and 2 read the score matrix)
size_t select_base_ws_bytes(const Dims& D) { return lay_out_select(D, PoolPlan(), nullptr).base_bytes; }
// the row-normalised rule also keeps a transformed copy of the score matrix behind the common scratch
size_t select_rownorm_ws_bytes(const Dims& D) {
  return ((select_ws_bytes(D) + 255) / 256) * 256 + (size_t)D.BH * D.S * D.Nb * sizeof(float);
}

}  // namespace vmoba

using namespace vmoba;

static int select_impl(const vmoba_shape* shape, const float* scores, const float* range, int rule, float tau, int topk, uint32_t* mask_bits,
                       int32_t* kb_ptr, int32_t* q_idx, int32_t* q_ptr, int32_t* q_pairs, int64_t capacity,
                       int64_t* k_per_head, float* cutoff_per_head, int32_t* dev_status, void* ws, size_t ws_bytes,
                       void* stream, bool allow_base_ws = false) {
  Dims D;
  int rc = make_dims(shape, &D);
  if (rc) return rc;
  // D is known here: a query at block-major position p lies in key block p / s_b
  const int own_sb = (rule & VMOBA_SELECT_KEEP_OWN_BLOCK) ? D.sb : 0;
  rule &= ~VMOBA_SELECT_KEEP_OWN_BLOCK;
  const bool rownorm = rule == VMOBA_SELECT_THRESHOLD_GLOBAL_ROWNORM;
  if (rownorm) rule = VMOBA_SELECT_THRESHOLD_GLOBAL;
  const bool by_topk = rule == VMOBA_SELECT_TOPK_GLOBAL || rule == VMOBA_SELECT_TOPK_LOCAL;
  const bool local = rule == VMOBA_SELECT_THRESHOLD_LOCAL || rule == VMOBA_SELECT_TOPK_LOCAL;
  if (rule < VMOBA_SELECT_THRESHOLD_GLOBAL || rule > VMOBA_SELECT_TOPK_LOCAL) return VMOBA_ERR_ARG;
  if (by_topk ? topk < 1 : (!(tau > 0.0f) || tau > 1.0f)) return VMOBA_ERR_ARG;
  if (!scores || !mask_bits || !kb_ptr || !q_idx || !q_ptr || !q_pairs || !k_per_head || !cutoff_per_head ||
      !dev_status || !ws)
    return VMOBA_ERR_ARG;
  if (!aligned16(scores) || !aligned16(ws)) return VMOBA_ERR_ARG;
  if (capacity <= 0 || capacity > (int64_t)INT32_MAX) return VMOBA_ERR_ARG;
  if (D.Nb > 8192 || (local && D.Nb > 32 * kLocalMaxWords)) return VMOBA_ERR_SHAPE;
  SelectWs w = carve_select(D, !local, ws);
  if (ws_bytes < (rownorm ? select_rownorm_ws_bytes(D) : (allow_base_ws ? w.base_bytes : w.bytes))) return VMOBA_ERR_WORKSPACE;
  // the candidate lists are the last slice: a caller with a fixed scratch area may have no room for them
  const bool use_cand = ws_bytes >= w.bytes;
  if (!use_cand && !w.pool.C) { w.cand = nullptr; w.ccap = -1; if (w.guards.n > 0) w.guards.n -= 1; }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const long long P = (long long)D.S * D.Nb;
  float sigma = D.scale;
  if (rownorm) {
    // search on the row-normalised log-probabilities with unit temperature
    float* lp = reinterpret_cast<float*>(static_cast<char*>(ws) + ((w.bytes + 255) / 256) * 256);
    const long long n_rows = (long long)D.BH * D.S;
    launch_kernel(rownorm_kernel, (int)std::min<long long>((n_rows + 7) / 8, sm_count() * 8), 256, 0, st, scores, lp,
                  D.Nb, D.scale, n_rows);
    VMOBA_LAUNCH_OK(1);
    scores = lp;
    sigma = 1.0f;
    range = nullptr;      // the range of the raw scores says nothing about the transformed matrix
  }
  VMOBA_GUARDS_ARM(w.guards, st);
  const int QSEG = w.QSEG, nseg = w.nseg;
  const bool pool = w.pool.C > 0;
  auto pool_launch = [&](auto tag, const float* pool_range, int unit_w, double count_target) -> int {
    const size_t pool_smem = decltype(tag)::value == kPoolMask ? w.pool.smem_mask : w.pool.smem;
    PoolArgs a;
    a.scores = scores; a.range = pool_range; a.state = w.state;
    a.S = D.S; a.Nb = D.Nb; a.mw = D.mask_words; a.QSEG = QSEG; a.nseg = nseg; a.segs_per = w.pool.segs_per;
    a.own_sb = own_sb; a.unit_w = unit_w; a.sigma = sigma; a.tau = tau; a.count_target = count_target;
    a.mask_bits = mask_bits; a.tmask = w.tmask; a.seg_cnt = w.seg_cnt; a.seg_qoff = w.seg_qoff; a.kb_excl = w.kb_total;
    a.k_per_head = k_per_head; a.cutoff_per_head = cutoff_per_head;
    auto kernel = w.pool.T == 256 ? select_pool_kernel<decltype(tag)::value, 256> : select_pool_kernel<decltype(tag)::value, 512>;
    VMOBA_CUDA_OK(allow_smem(kernel, kSmemMost));
    launch_cluster(true, w.pool.C, kernel, (unsigned)(D.BH * w.pool.C), w.pool.T, pool_smem, st, a);
    VMOBA_LAUNCH_OK(1);
    return VMOBA_OK;
  };
#define VMOBA_POOL(src) std::integral_constant<PoolSrc, src>()
  const size_t smem = (size_t)QSEG * D.mask_words * 4 + (size_t)std::max(D.Nb, QSEG) * 4 + (size_t)D.Nb * (QSEG >> 5) * 4;
  const dim3 sgrid(nseg, D.BH);

  if (local) {
    launch_kernel(init_state_kernel, (D.BH + 127) / 128, 128, 0, st, w.state, D.BH, nullptr, nullptr, nullptr,
                  nullptr, nullptr);
    // per-query rules: the mask comes straight from the rows; cutoff_key collects the smallest selected key
    const long long n_rows = (long long)D.BH * D.S;
    const int blocks = (int)std::min<long long>((n_rows + 7) / 8, sm_count() * 8);
    const int mw = D.mask_words;
    const int k = std::min(topk, D.Nb);
    auto topk_words = [&](auto tag) {
      launch_kernel(select_topk_kernel<decltype(tag)::value>, blocks, 256, 0, st, scores, D.S, D.Nb, mw, k, own_sb,
                    mask_bits, w.state, n_rows);
    };
    auto topk_rows = [&](auto tag) {
      const int g = (int)std::min<long long>((n_rows + kTopkRowThreads - 1) / kTopkRowThreads, sm_count() * 32LL);
      launch_kernel(select_topk_rows_kernel<decltype(tag)::value>, g, kTopkRowThreads, 0, st, scores, D.S, D.Nb, k,
                    own_sb, mask_bits, w.state, n_rows);
    };
    auto threshold_words = [&](auto tag) {
      launch_kernel(select_threshold_local_kernel<decltype(tag)::value>, blocks, 256, 0, st, scores, D.S, D.Nb, mw,
                    D.scale, tau, own_sb, mask_bits, w.state, n_rows);
    };
#define VMOBA_INT(n) std::integral_constant<int, n>()
    if (by_topk) {
      // a word that a row does not have still costs its compares in every step: the instantiations are close together
      if (D.Nb <= 8) topk_rows(VMOBA_INT(8));
      else if (D.Nb <= 16) topk_rows(VMOBA_INT(16));
      else if (D.Nb <= 24) topk_rows(VMOBA_INT(24));
      else if (D.Nb <= 32) topk_rows(VMOBA_INT(32));
      else if (mw <= 2) topk_words(VMOBA_INT(2));
      else if (mw <= 3) topk_words(VMOBA_INT(3));
      else if (mw <= 4) topk_words(VMOBA_INT(4));
      else if (mw <= 5) topk_words(VMOBA_INT(5));
      else if (mw <= 6) topk_words(VMOBA_INT(6));
      else if (mw <= 7) topk_words(VMOBA_INT(7));
      else if (mw <= 8) topk_words(VMOBA_INT(8));
      else if (mw <= 9) topk_words(VMOBA_INT(9));
      else if (mw <= 10) topk_words(VMOBA_INT(10));
      else if (mw <= 12) topk_words(VMOBA_INT(12));
      else if (mw <= 14) topk_words(VMOBA_INT(14));
      else if (mw <= 16) topk_words(VMOBA_INT(16));
      else if (mw <= 24) topk_words(VMOBA_INT(24));
      else topk_words(VMOBA_INT(kLocalMaxWords));
    } else {
      if (mw <= 1) threshold_words(VMOBA_INT(1));
      else if (mw <= 2) threshold_words(VMOBA_INT(2));
      else if (mw <= 4) threshold_words(VMOBA_INT(4));
      else if (mw <= 8) threshold_words(VMOBA_INT(8));
      else if (mw <= 16) threshold_words(VMOBA_INT(16));
      else threshold_words(VMOBA_INT(kLocalMaxWords));
    }
#undef VMOBA_INT
    VMOBA_LAUNCH_OK(2);
    if (pool) {
      if ((rc = pool_launch(VMOBA_POOL(kPoolMask), nullptr, 0, -1.0))) return rc;
    } else {
      launch_kernel(local_cutoff_kernel, (D.BH + 127) / 128, 128, 0, st, w.state, cutoff_per_head, D.BH);
      VMOBA_CUDA_OK(allow_smem(mark_from_mask_kernel, kSmemMost));
      launch_kernel(mark_from_mask_kernel, sgrid, kSegThreads, smem, st, mask_bits, D.S, D.Nb, D.mask_words, QSEG, nseg,
                    w.seg_cnt, w.seg_total, w.tmask);
      VMOBA_LAUNCH_OK(2);
    }
  } else {
    // head-wide rules: weighted quantile of the pool (unit weights and a pair budget for top-k)
    double count_target = -1.0;
    if (by_topk) {
      count_target = (double)std::min<long long>((long long)topk * D.S, P);
      tau = count_target >= (double)P ? 1.0f : 0.5f;      // tau only tells the scan whether everything is taken
    }
    const int unit_w = by_topk ? 1 : 0;
    if (pool) {
      if ((rc = pool_launch(VMOBA_POOL(kPoolScores), range, unit_w, count_target))) return rc;
    } else {
      // enough CTAs per head to fill the machine, few enough that the per-CTA flush stays small
      long long per_head = (P / 4 + 255) / 256;
      int gx = (int)std::min<long long>(std::max<long long>(per_head / 8, 1), std::max(1, sm_count() * 8 / D.BH));
      dim3 grid(gx, D.BH);
      launch_kernel(init_state_kernel, (unsigned)(((long long)D.BH * kBins + 255) / 256), 256, 0, st, w.state, D.BH,
                    range, w.g_cnt, w.g_w, w.g_minkey, w.g_maxkey);

      if (!range) {
        launch_kernel(minmax_kernel, grid, 256, 0, st, scores, P, w.state);
        launch_kernel(setup_level0_kernel, (D.BH + 127) / 128, 128, 0, st, w.state, D.BH);
        count_launches(2);
      }
      {
        constexpr int smem0 = kBins0 * kRep * (int)sizeof(float);
        VMOBA_CUDA_OK(allow_smem(hist0_kernel, smem0));
        // three 512-thread CTAs per SM hold their replicated bins side by side
        int gx0 = (int)std::min<long long>(std::max<long long>(per_head / 16, 1), std::max(1, sm_count() * 3 / D.BH));
        launch_kernel(early_rows(D), hist0_kernel, dim3(gx0, D.BH), 512, smem0, st, scores, P, w.state, sigma, unit_w,
                      w.g_w);
      }
      launch_kernel(scan_kernel<0>, D.BH, 1024, 0, st, w.state, tau, count_target, w.g_cnt, w.g_w, w.g_minkey,
                    w.g_maxkey, k_per_head, cutoff_per_head, w.ccap);
      launch_kernel(hist_kernel<1>, grid, 256, 0, st, scores, P, w.state, sigma, unit_w, w.g_cnt, w.g_w, w.g_minkey,
                    w.g_maxkey, w.cand, w.ccap, &w.state->cand_cnt);
      launch_kernel(scan_kernel<1>, D.BH, 1024, 0, st, w.state, tau, count_target, w.g_cnt, w.g_w, w.g_minkey,
                    w.g_maxkey, k_per_head, cutoff_per_head, w.ccap);
      launch_kernel(hist_kernel<2>, grid, 256, 0, st, scores, P, w.state, sigma, unit_w, w.g_cnt, w.g_w, w.g_minkey,
                    w.g_maxkey, w.cand, w.ccap, &w.state->cand_cnt);
      launch_kernel(scan_kernel<2>, D.BH, 1024, 0, st, w.state, tau, count_target, w.g_cnt, w.g_w, w.g_minkey,
                    w.g_maxkey, k_per_head, cutoff_per_head, w.ccap);
      VMOBA_LAUNCH_OK(7);
      VMOBA_CUDA_OK(allow_smem(mark_kernel, kSmemMost));
      launch_kernel(mark_kernel, sgrid, kSegThreads, smem, st, scores, w.state, D.S, D.Nb, D.mask_words, QSEG, nseg,
                    own_sb, mask_bits, w.seg_cnt, w.seg_total, w.tmask);
      VMOBA_LAUNCH_OK(1);
    }
  }
#undef VMOBA_POOL

  // (the top-k rule's segments have so many pairs and no more)
  const int stage = rule == VMOBA_SELECT_TOPK_LOCAL
                        ? (int)std::min<long long>(kStage, (long long)QSEG * (std::min(topk, D.Nb) + (own_sb > 0 ? 1 : 0)) + 1 & ~1ll)
                        : kStage;
  const size_t cols = (size_t)D.Nb * (QSEG >> 5);
  const size_t smem_fill = ((size_t)QSEG * D.mask_words + cols + 2 * (size_t)D.Nb + 1 + stage) * 4 + (stage + cols) * 2;
  VMOBA_CUDA_OK(allow_smem(fill_kernel, kSmemMost));
  long long nkb = (long long)D.BH * D.Nb;
  if (!pool) {
    launch_kernel(seg_prefix_kernel, (unsigned)(D.BH * ((D.Nb + 31) / 32)), 32 * std::min(32, (nseg + 7) / 8), 0, st,
                  w.seg_cnt, w.kb_total, D.Nb, nseg);
    launch_kernel(offsets_kernel, 1, 1024, 0, st, w.kb_total, kb_ptr, nkb, w.seg_total, w.seg_qoff,
                  (long long)D.BH * nseg, D.BH, D.Nb, k_per_head, capacity, q_ptr + (long long)D.BH * D.S, dev_status);
    VMOBA_LAUNCH_OK(2);
  }
  // A thread per query of the segment; many blocks leave short segments (32 queries from 2,049 blocks on), whose columns and
  // runs want the threads all the same: 2,100 blocks x 33,600 queries 1001 -> 432 us (whole selection, threshold rule), 8,192 x
  // 16,384 3376 -> 1053.
  const int fill_threads = QSEG >= 128 ? QSEG : kSegThreads;
  launch_kernel(fill_kernel, sgrid, fill_threads, smem_fill, st, mask_bits, w.tmask, D.S, D.Nb, D.mask_words, QSEG, nseg,
                kb_ptr, w.seg_cnt, w.seg_qoff, q_idx, q_ptr, q_pairs, capacity, pool ? w.kb_total : nullptr, k_per_head,
                dev_status, stage);
  VMOBA_LAUNCH_OK(1);
  VMOBA_GUARDS_CHECK(w.guards, dev_status, st);
  return VMOBA_OK;
}

extern "C" int vmoba_select(const vmoba_shape* shape, const float* scores, float tau, uint32_t* mask_bits,
                            int32_t* kb_ptr, int32_t* q_idx, int32_t* q_ptr, int32_t* q_pairs,
                            int64_t capacity, int64_t* k_per_head, float* cutoff_per_head,
                            int32_t* dev_status, void* ws, size_t ws_bytes, void* stream) {
  return select_impl(shape, scores, nullptr, VMOBA_SELECT_THRESHOLD_GLOBAL, tau, 0, mask_bits, kb_ptr, q_idx, q_ptr, q_pairs,
                     capacity, k_per_head, cutoff_per_head, dev_status, ws, ws_bytes, stream);
}

extern "C" int vmoba_select_ranged(const vmoba_shape* shape, const float* scores, const float* score_range, int32_t rule,
                                   float tau, int32_t topk, uint32_t* mask_bits, int32_t* kb_ptr, int32_t* q_idx,
                                   int32_t* q_ptr, int32_t* q_pairs, int64_t capacity, int64_t* k_per_head,
                                   float* cutoff_per_head, int32_t* dev_status, void* ws, size_t ws_bytes, void* stream) {
  if (!score_range) return VMOBA_ERR_ARG;
  return select_impl(shape, scores, score_range, rule, tau, topk, mask_bits, kb_ptr, q_idx, q_ptr, q_pairs, capacity,
                     k_per_head, cutoff_per_head, dev_status, ws, ws_bytes, stream);
}

extern "C" int vmoba_select_rule_apply(const vmoba_shape* shape, const float* scores, int32_t rule, float tau, int32_t topk,
                                       uint32_t* mask_bits, int32_t* kb_ptr, int32_t* q_idx, int32_t* q_ptr,
                                       int32_t* q_pairs, int64_t capacity, int64_t* k_per_head, float* cutoff_per_head,
                                       int32_t* dev_status, void* ws, size_t ws_bytes, void* stream) {
  return select_impl(shape, scores, nullptr, rule, tau, topk, mask_bits, kb_ptr, q_idx, q_ptr, q_pairs, capacity, k_per_head,
                     cutoff_per_head, dev_status, ws, ws_bytes, stream);
}

// ------------------------------------------------------------------------------------------
// Selection without a caller-provided workspace.
//
// Some callers of this library are not allowed to allocate device memory at the point where
// they run the layer: code running inside a memory-planned inference engine or a framework
// plug-in that was handed fixed input/output buffers and nothing else, or a latency-critical
// loop in which cudaMalloc (which synchronises the device) is forbidden.  For them the scratch
// of the selection stage lives in the array below, which is part of the library image: every
// GPU that loads the library holds these bytes until the process exits.
namespace vmoba {
constexpr size_t kStaticSelectScratchBytes = 16u << 20;   // 16 MiB
static __device__ __align__(256) unsigned char g_select_scratch[kStaticSelectScratchBytes];

constexpr int kMaxDevices = 64;
static void* g_select_scratch_addr[kMaxDevices] = {nullptr};
}  // namespace vmoba

extern "C" size_t vmoba_select_static_scratch_bytes(void) { return vmoba::kStaticSelectScratchBytes; }

extern "C" int vmoba_select_static(const vmoba_shape* shape, const float* scores, float tau, uint32_t* mask_bits,
                                   int32_t* kb_ptr, int32_t* q_idx, int32_t* q_ptr, int32_t* q_pairs,
                                   int64_t capacity, int64_t* k_per_head, float* cutoff_per_head,
                                   int32_t* dev_status, void* stream) {
  Dims D;
  int rc = make_dims(shape, &D);
  if (rc) return rc;
  if (D.Nb > 8192) return VMOBA_ERR_SHAPE;
  // The shape's scratch need must fit the fixed array; larger problems have to use vmoba_select.
  if (select_base_ws_bytes(D) > kStaticSelectScratchBytes) return VMOBA_ERR_WORKSPACE;
  int dev = -1;
  VMOBA_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return VMOBA_ERR_CUDA;
  if (!g_select_scratch_addr[dev]) {
    // In host code the array's name is only a handle for the symbol, not a device address: ask the
    // runtime for the address on the current device, once per device.
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_select_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return VMOBA_ERR_CUDA;
    }
    g_select_scratch_addr[dev] = p;
  }
  // vmoba_select clears everything in its scratch that has to start at zero, so the contents
  // left by an earlier call do not matter.
  return select_impl(shape, scores, nullptr, VMOBA_SELECT_THRESHOLD_GLOBAL, tau, 0, mask_bits, kb_ptr, q_idx, q_ptr, q_pairs,
                     capacity, k_per_head, cutoff_per_head, dev_status, g_select_scratch_addr[dev], kStaticSelectScratchBytes,
                     stream, /*allow_base_ws=*/true);
}
