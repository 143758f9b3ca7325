// Tensor-core attention forward for bf16, head_dim 128 (Step 3 of VMoBA and its dense limit).
//
// One persistent CTA per SM walks the work items.  An item is up to 256 query rows (sparse: a chunk of
// the queries that selected key block j, gathered by index; dense: 256 consecutive rows) against a
// contiguous key range (the block, or the whole sequence), streamed in tiles of 128 keys.
// With 128 query rows per CTA every 128-key tile of K and V (64 KB) feeds only 1024 tensor-pipe
// cycles, and the L2-to-SM path, not the tensor pipe, sets the pace.  Here a CTA owns TWO 128-row
// query tiles (A and B) that share each K/V tile, which halves the bytes per MMA.
//
//   warp 0        TMA producer: K tiles into a ring of two stages, V tiles into one of three
//   warps 1, 2    MMA issuers: Q K^T, P V
//   warps 4-7     softmax of tile A: thread = one query row, all 128 keys of the tile
//   warps 8-11    softmax of tile B
//   warps 12-15   gather the 256 Q rows of the NEXT item and write the rows of o of the one before
//
// TMEM: ONE score buffer S (128 columns) that A and B use in turn, P_A and P_B (64 columns each, bf16), the accumulators
// O_A and O_B (128 columns each).  A softmax thread (200 registers) takes its whole row of 128 scores out of S at once and
// frees the buffer; the tensor pipe goes on with the other tile's Q K^T while the exponentials are worked out of
// registers, and P goes to columns of its own.  So Q K^T(t+1) of a tile waits neither for its own P(t) nor for its
// P V(t): a tile's pace is the softmax alone (128 scores per thread: 1024 cycles of the exponential unit per warp, two
// warps to a unit, 2048 per pair of tiles, as many as the four matrix products take).  With a score buffer per tile and P
// written over it, the chain Q K^T -> softmax -> P V -> Q K^T of a tile took 4490 cycles per pair of tiles.
#include <algorithm>

#include <cuda_fp16.h>

#include "attn_simt.cuh"
#include "sm100.cuh"

namespace vmoba {
namespace tcw {

using namespace sm100;

constexpr int BM = 128;              // rows per query tile
constexpr int IM = 2 * BM;           // query rows per item
constexpr int BN = 128;              // keys per tile
constexpr int DH = 128;              // head dim
// K and V ring depths.  A V tile is needed by A and, half a period later, by B, and is reloaded after that: with two
// stages the MMA warp waited for V tiles (700 of 4550 cycles per pair of tiles).
constexpr int KST = 2, VST = 3;
constexpr int PANEL = BM * 128;      // bytes of one 64-column panel of a 128-row tile (16 KB)
constexpr int TILE = 2 * PANEL;      // bytes of a [128 x 128] bf16 tile (32 KB)
constexpr int THREADS = 512;         // warp groups {TMA, MMA, MMA, -}, A, B, loaders; registers 56, 200, 200, 56 (= 4 x 128)
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t P_COL = 128, O_COL = 256;      // S at 0, P_X at 128 + 64 X, O_X at 256 + 128 X
constexpr float RESCALE_LOG2 = 8.0f;

struct Smem {
  uint64_t k_full[KST], k_empty[KST], v_full[VST], v_empty[VST];
  uint64_t s_full[2], p_ready[2];    // per query tile: scores written (commit) / P written (128 arrivals)
  uint64_t s_free;                   // the score buffer has been read (128 arrivals of whichever tile used it)
  uint64_t o_done[2];                // per query tile: P V of a key tile complete (commit)
  uint64_t ep_ready[2];              // per query tile: an item's normalisers are in ep_inv / ep_lse (128 softmax arrivals)
  uint64_t o_free[2];                // per query tile: epilogue has read them and the accumulator (128 arrivals)
  uint64_t q_full, q_empty;          // Q tiles of an item gathered (128 arrivals) / no longer needed (commit)
  uint32_t tmem_base;
  int abort_flag;
  float ep_inv[2][BM], ep_lse[2][BM];   // 1 / sum of the rounded weights, natural-log lse
};
// no alignment slack: the kernel checks that its dynamic shared memory starts on a 1024-byte boundary
constexpr size_t SMEM_BYTES = (2 /*Q*/ + KST + VST) * TILE + sizeof(Smem) + 32;
static_assert(SMEM_BYTES <= 232448, "wide forward: shared memory");

struct Params {
  const __nv_bfloat16* q;
  const int* q_idx;
  const int* q_ptr;
  const int* item_ptr;
  const int4* item_desc;   // per item {list index, first list position, rows, 0}
  int n_kb, S, Nb, sb, BH;
  float scale_log2;      // softmax scale * log2(e)
  __nv_bfloat16* o;
  __nv_bfloat16* o_resid;
  RowMap o_map;          // where the rows of o go (block-major, or raster order through perm); o_resid is block-major
  float* lse;
  __half* part_o;        // partial rows: fp16 values times part_scale[row]
  float* part_lse;
  float* part_scale;
  int part_o_32;         // part_o is 32-byte aligned: rows go out with 32-byte stores
  int32_t* status;
  unsigned long long* prof;   // optional per-section cycle counters (diagnostics), or null
};

struct FwdItem {
  int bh, key_begin, n_keys, list_lo, n_rows, ntiles, nx;   // nx: query tiles in use (1 or 2)
  long long head_off;
};

template <bool DENSE>
__device__ __forceinline__ FwdItem decode_item(const Params& p, int item) {
  FwdItem it;
  if (DENSE) {
    const int tiles = (p.S + IM - 1) / IM;
    it.bh = item / tiles;
    const int t = item - it.bh * tiles;
    it.key_begin = 0; it.n_keys = p.S; it.list_lo = t * IM; it.n_rows = min(IM, p.S - it.list_lo);
  } else {
    const int4 d = __ldg(p.item_desc + item);
    const int kbi = checked_index(d.x, p.n_kb, p.status);
    it.bh = kbi / p.Nb;
    it.key_begin = (kbi - it.bh * p.Nb) * p.sb; it.n_keys = p.sb;
    it.list_lo = d.y; it.n_rows = d.z;
  }
  it.ntiles = (it.n_keys + BN - 1) / BN;
  it.nx = it.n_rows > BM ? 2 : 1;
  it.head_off = (long long)it.bh * p.S;
  return it;
}

__device__ __forceinline__ constexpr uint32_t koff(int ks) { return (uint32_t)(((ks >> 2) * PANEL + (ks & 3) * 32) >> 4); }
__device__ __forceinline__ constexpr uint32_t mnoff(int ks) { return (uint32_t)((ks * 2048) >> 4); }

// p = 2^(s * scale - m) for 32 scores; bf16 pairs (keys 2i, 2i+1 -> word i); s0/s1 collect the exact
// weights, r0/r1 the bf16-rounded ones (the tensor core multiplies the ROUNDED weights: O is
// normalised by their sum, so that the rounding perturbs the weights but never their total).
__device__ __forceinline__ void exp_pack32(const uint32_t* sv, float scale, float neg_m, uint32_t (&pk)[16], float& s0, float& s1,
                                           float& r0, float& r1) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    float p0, p1;
    fma2(p0, p1, __uint_as_float(sv[2 * i]), __uint_as_float(sv[2 * i + 1]), scale, scale, neg_m, neg_m);
    p0 = ex2(p0);
    p1 = ex2(p1);
    add2(s0, s1, s0, s1, p0, p1);
    pk[i] = pack_bf16(p0, p1);
    add_bf16_pair(r0, r1, pk[i]);
  }
}

// Partial rows are stored as fp16 times a power of two per row: the smallest one at or above the row's largest
// magnitude (1 for a row of zeros), so that the values use the format's full precision whatever the scale of V.
__device__ __forceinline__ float pow2_at_or_above(float x) {
  const uint32_t u = (__float_as_uint(x) + 0x007fffffu) & 0x7f800000u;
  return u ? __uint_as_float(u) : 1.0f;
}
__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Eight consecutive outputs as bf16 (one 16-byte store) and, if asked for, their rounding residuals bf16(v - bf16(v)),
// computed in registers.
__device__ __forceinline__ void store8_resid(__nv_bfloat16* dst, __nv_bfloat16* rdst, const float (&v)[8]) {
  uint32_t h[4], r[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    h[k] = pack_bf16(v[2 * k], v[2 * k + 1]);
    r[k] = pack_bf16(v[2 * k] - __uint_as_float(h[k] << 16), v[2 * k + 1] - __uint_as_float(h[k] & 0xffff0000u));
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(h[0], h[1], h[2], h[3]);
  if (rdst) *reinterpret_cast<uint4*>(rdst) = make_uint4(r[0], r[1], r[2], r[3]);
}

// RASTER: the directly written rows of o go through p.o_map (a kernel of its own: with the map's address
// arithmetic compiled into the one kernel, the block-major case ran 6 % slower on the 720p-shaped layers).
template <bool DENSE, bool RASTER, bool PROF>
__global__ void __launch_bounds__(THREADS, 1)
attn_fwd_wide_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                     const __grid_constant__ CUtensorMap tmQ, const Params p) {
  if (!grid_begin()) return;
  extern __shared__ uint8_t smem_raw[];
  // the swizzled tiles need 1024-byte alignment and there is no room for alignment slack
  if ((smem_u32(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) set_status(p.status, VMOBA_ERR_CUDA);
    return;
  }
  uint8_t* sQ = smem_raw;                  // [2 query tiles][TILE]
  uint8_t* sK = sQ + 2 * TILE;             // [KST][TILE]
  uint8_t* sV = sK + KST * TILE;           // [VST][TILE]
  Smem* sm = reinterpret_cast<Smem*>(sV + VST * TILE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &sm->abort_flag;
  // diagnostics: cycles one representative thread per role spends in each section
  unsigned long long wp[6] = {0, 0, 0, 0, 0, 0};
  long long t_mark = PROF ? clock64() : 0;
  const long long t_begin = t_mark;
  auto lap = [&](int site) {
    if constexpr (PROF) {
      const long long now = clock64();
      wp[site] += (unsigned long long)(now - t_mark);
      t_mark = now;
    }
  };
  auto tflush = [&](int base_site) {
    if constexpr (PROF) {
      for (int i = 0; i < 6; ++i) atomicAdd(p.prof + base_site + i, wp[i]);
      atomicAdd(p.prof + base_site + 6, (unsigned long long)(clock64() - t_begin));
    }
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < KST; ++s) { mbar_init(&sm->k_full[s], 1); mbar_init(&sm->k_empty[s], 1); }
    for (int s = 0; s < VST; ++s) { mbar_init(&sm->v_full[s], 1); mbar_init(&sm->v_empty[s], 1); }
    for (int x = 0; x < 2; ++x) {
      mbar_init(&sm->s_full[x], 1); mbar_init(&sm->p_ready[x], 128);
      mbar_init(&sm->o_done[x], 1); mbar_init(&sm->o_free[x], 128); mbar_init(&sm->ep_ready[x], 128);
    }
    mbar_init(&sm->s_free, 128);
    mbar_init(&sm->q_full, 128); mbar_init(&sm->q_empty, 1);
    sm->abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
  }
  if (warp == 1) {
    tmem_alloc(&sm->tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem_base;
  const int n_items = DENSE ? p.BH * ((p.S + IM - 1) / IM) : p.item_ptr[p.n_kb];
  constexpr uint32_t IDESC_PV = make_idesc_bf16(BM, DH, false, true);

  if (warp < 4) asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t ks = 0, kp = 1, vs = 0, vp = 1;       // ring slots and the parities of their `empty` waits (the first pass at once)
      for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
        const FwdItem it = decode_item<DENSE>(p, item);
        const int row0 = (int)it.head_off + it.key_begin;
        for (int t = 0; t < it.ntiles; ++t) {
          const int y = row0 + t * BN;
          // a K stage is free once both query tiles' Q K^T of the key tile have run, a V stage only
          // after both P V
          mbar_wait(&sm->k_empty[ks], kp, abort_flag, p.status);
          mbar_expect_tx(&sm->k_full[ks], TILE);
          tma_load_2d(sK + ks * TILE, &tmK, &sm->k_full[ks], 0, y);
          tma_load_2d(sK + ks * TILE + PANEL, &tmK, &sm->k_full[ks], 64, y);
          mbar_wait(&sm->v_empty[vs], vp, abort_flag, p.status);
          mbar_expect_tx(&sm->v_full[vs], TILE);
          tma_load_2d(sV + vs * TILE, &tmV, &sm->v_full[vs], 0, y);
          tma_load_2d(sV + vs * TILE + PANEL, &tmV, &sm->v_full[vs], 64, y);
          // drain: every issued load must have landed before the CTA may exit (only matters after a timeout)
          if (*abort_flag) {
            mbar_wait(&sm->k_full[ks], kp ^ 1, abort_flag, p.status);
            mbar_wait(&sm->v_full[vs], vp ^ 1, abort_flag, p.status);
          }
          if (++ks == KST) { ks = 0; kp ^= 1; }
          if (++vs == VST) { vs = 0; vp ^= 1; }
        }
      }
    }
  } else if (warp <= 2) {
    // ------------------------------------------------------------------ MMA issuers: warp 1 the Q K^T, warp 2 the P V; the
    // whole warp walks the loop, one elected lane issues (warp-uniform control flow; see elect_one).
    // Two of them, because one does not keep the tensor pipe busy: next to the softmax warps of its sub-partition a warp
    // gets an MMA out every 105 cycles (64 is the pipe's rate), and a look at a barrier takes it some 300 cycles while the
    // pipe streams its operands out of shared memory.  The lanes look at an operation's barriers at once.
    const bool leader = elect_one();
    const int n_items_u = __reduce_max_sync(0xffffffffu, n_items);
    auto wait3 = [&](uint64_t* b0, uint32_t p0, uint64_t* b1, uint32_t p1, bool third, uint64_t* b2, uint32_t p2) {
      const int which = lane & 3;
      uint32_t bar = smem_u32(b0), par = p0;
      if (which == 1) { bar = smem_u32(b1); par = p1; }
      if (which == 2 && third) { bar = smem_u32(b2); par = p2; }
      lap(5);
      mbar_wait_lanes(bar, par, abort_flag, p.status);
      __syncwarp();
      lap(0);
      tc_fence_after();
    };
    if (warp == 1) {
      uint32_t uses = 0, n = 0, slot = 0, par = 0;      // uses of the score buffer, items, K ring position
      const uint32_t lo_q = desc_lo(smem_u32(sQ), 16), lo_k = desc_lo(smem_u32(sK), 16);
      for (int item = blockIdx.x; item < n_items_u; item += gridDim.x, ++n) {
        FwdItem it = decode_item<DENSE>(p, item);
        it.nx = __reduce_max_sync(0xffffffffu, it.nx);
        for (int t = 0; t < it.ntiles; ++t) {
          const int n_mma = (min(BN, it.n_keys - t * BN) + 15) & ~15;
          const uint32_t idesc = make_idesc_bf16(BM, n_mma, false, false);
          const uint32_t dk = lo_k + slot * (uint32_t)(TILE >> 4);
          for (int x = 0; x < it.nx; ++x) {
            // the score buffer has been read (its first use waits for a phase before the first: passes at once), the K tile
            // is there, and the item's Q tiles
            wait3(&sm->s_free, (uses + 1) & 1, &sm->k_full[slot], par, t == 0 && x == 0, &sm->q_full, n & 1);
            ++uses;
            const uint32_t dq = lo_q + x * (uint32_t)(TILE >> 4);
#pragma unroll
            for (int ks = 0; ks < DH / 16; ++ks)
              if (leader) mma_ss_lo(tmem, dq + koff(ks), dk + koff(ks), idesc, ks > 0 ? 1u : 0u);
            if (leader) mma_commit(&sm->s_full[x]);
          }
          if (leader) mma_commit(&sm->k_empty[slot]);
          if (leader && t == it.ntiles - 1) mma_commit(&sm->q_empty);
          if (++slot == KST) { slot = 0; par ^= 1; }
        }
      }
      lap(5);
      if (leader) tflush(8);
    } else {
      uint32_t tcnt[2] = {0, 0}, ecnt[2] = {0, 0}, slot = 0, par = 0;      // per query tile: P V and items done; V ring position
      const uint32_t lo_v = desc_lo(smem_u32(sV), PANEL);
      for (int item = blockIdx.x; item < n_items_u; item += gridDim.x) {
        FwdItem it = decode_item<DENSE>(p, item);
        it.nx = __reduce_max_sync(0xffffffffu, it.nx);
        for (int t = 0; t < it.ntiles; ++t) {
          const int ksteps = (min(BN, it.n_keys - t * BN) + 15) >> 4;
          const uint32_t mv = lo_v + slot * (uint32_t)(TILE >> 4);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            if (x >= it.nx) continue;
            // P has been written, the V tile is there, the epilogue of the tile's previous item has read the accumulator
            wait3(&sm->p_ready[x], tcnt[x] & 1, &sm->v_full[slot], par, t == 0, &sm->o_free[x], (ecnt[x] + 1) & 1);
            tcnt[x] += 1;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              if (leader && ks < ksteps)   // P of keys 16 ks .. 16 ks + 15 sits in columns 8 ks .. of the tile's P buffer
                mma_ts_lo(tmem + O_COL + x * 128, tmem + P_COL + x * 64 + ks * 8, mv + mnoff(ks), IDESC_PV, (t > 0 || ks > 0) ? 1u : 0u);
            if (leader) mma_commit(&sm->o_done[x]);
          }
          if (leader) mma_commit(&sm->v_empty[slot]);
          if (++slot == VST) { slot = 0; par ^= 1; }
        }
        ecnt[0] += 1;
        if (it.nx == 2) ecnt[1] += 1;
      }
      lap(5);
      if (PROF && leader) { atomicAdd(p.prof + 10, wp[0]); atomicAdd(p.prof + 11, wp[5]); }
    }
  } else if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    // ------------------------------------------------------------------ loaders and epilogue: the Q rows of item n, then the
    // rows of o of item n - 1 (while the softmax warps are at work on item n: an epilogue takes about as long as one and a
    // half key tiles, a third of an item of three)
    // Q, sparse: asynchronous 16-byte copies, eight threads per 128-byte half row, asked for in the L2 ahead of time; dense:
    // consecutive rows, TMA tiles.
    const int lt = (warp - 12) * 32 + lane;   // 0..127
    const int r0 = lt >> 3, chunk = lt & 7;   // Q rows r0 + 16 k
    uint32_t n = 0;
    uint32_t tcs[2] = {0, 0}, eps[2] = {0, 0};        // per query tile: P V and items done
    auto epilogue = [&](const FwdItem& it) {
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (x >= it.nx) continue;
        const uint32_t o_tmem = tmem + ((uint32_t)((warp & 3) * 32) << 16) + O_COL + x * 128;
        const int row = x * BM + lt;                  // thread = query row
        const bool row_ok = row < it.n_rows;
        const int qpos = !row_ok ? 0 : DENSE ? it.list_lo + row : checked_index(__ldg(p.q_idx + it.list_lo + row), p.S, p.status);
        const long long G_ = it.head_off + qpos;
        // the query has a single block: final result
        const bool direct = DENSE || __ldg(p.q_ptr + G_ + 1) - __ldg(p.q_ptr + G_) == 1;
        const long long o_row_off = RASTER ? ((row_ok && direct) ? p.o_map.off(G_, DH) : 0) : G_ * DH;
        const long long pos = (long long)it.list_lo + row;
        tcs[x] += it.ntiles;
        mbar_wait(&sm->ep_ready[x], eps[x] & 1, abort_flag, p.status);
        eps[x] += 1;
        const float inv = sm->ep_inv[x][lt], row_lse = sm->ep_lse[x][lt];
        mbar_wait(&sm->o_done[x], (tcs[x] - 1) & 1, abort_flag, p.status);
        tc_fence_after();
        // a partial row goes out as fp16 times a power of two: find the row's largest magnitude first
        float mul = inv, row_scale = 1.0f;
        if constexpr (!DENSE) {
          const bool partial = row_ok && !direct;
          if (__any_sync(0xffffffffu, partial)) {
            float amax = 0.f;
#pragma unroll 1
            for (int c = 0; c < 8; ++c) {
              uint32_t ov[16];
              tmem_ld16(o_tmem + c * 16, ov);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 16; ++i) amax = fmaxf(amax, fabsf(__uint_as_float(ov[i])));
            }
            if (partial) {
              row_scale = pow2_at_or_above(amax * inv);
              mul = inv / row_scale;
            }
          }
        }
#pragma unroll 1
        for (int c = 0; c < 8; ++c) {
          uint32_t ov[16];
          tmem_ld16(o_tmem + c * 16, ov);
          tmem_ld_wait();
          if (c == 7) {
            tc_fence_before();
            mbar_arrive(&sm->o_free[x]);
          }
          if (row_ok) {
            const int col = 16 * c;
            if (direct) {
              __nv_bfloat16* dst = p.o + o_row_off + col;
              __nv_bfloat16* rdst = p.o_resid ? p.o_resid + G_ * DH + col : nullptr;
#pragma unroll
              for (int i = 0; i < 16; i += 8) {
                float v8[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) v8[k] = __uint_as_float(ov[i + k]) * inv;
                store8_resid(dst + i, rdst ? rdst + i : nullptr, v8);
              }
            } else {
              __half* dst = p.part_o + pos * DH + col;
              uint32_t h[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) h[k] = pack_half2(__uint_as_float(ov[2 * k]) * mul, __uint_as_float(ov[2 * k + 1]) * mul);
              if (p.part_o_32) {       // one 32-byte store, else two of 16 bytes
                st_global_v8(dst, h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7]);
              } else {
                reinterpret_cast<uint4*>(dst)[0] = make_uint4(h[0], h[1], h[2], h[3]);
                reinterpret_cast<uint4*>(dst)[1] = make_uint4(h[4], h[5], h[6], h[7]);
              }
            }
          }
        }
        if (row_ok) {
          if (direct) p.lse[G_] = row_lse; else { p.part_lse[pos] = row_lse; p.part_scale[pos] = row_scale; }
        }
      }
    };
    FwdItem before;
    for (int item = blockIdx.x; item < n_items; item += gridDim.x, ++n) {
      const FwdItem it = decode_item<DENSE>(p, item);
      if constexpr (DENSE) {
        if (n >= 1) mbar_wait(&sm->q_empty, (n - 1) & 1, abort_flag, p.status);
        if (lt == 0) {
          mbar_expect_tx(&sm->q_full, it.nx * TILE);
          for (int x = 0; x < it.nx; ++x) {
            tma_load_3d(sQ + x * TILE, &tmQ, &sm->q_full, 0, it.list_lo + x * BM, it.bh);
            tma_load_3d(sQ + x * TILE + PANEL, &tmQ, &sm->q_full, 64, it.list_lo + x * BM, it.bh);
          }
          if (*abort_flag) mbar_wait(&sm->q_full, n & 1, abort_flag, p.status);     // landed before the CTA may exit
        } else {
          mbar_arrive(&sm->q_full);
        }
      } else {
        const __nv_bfloat16* qh = p.q + it.head_off * DH + chunk * 8;
        int idx[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int row = r0 + 16 * k;
          idx[k] = row < it.n_rows ? checked_index(__ldg(p.q_idx + it.list_lo + row), p.S, p.status) : -1;
        }
        if (chunk == 0) {        // one request per 128-byte line
#pragma unroll
          for (int k = 0; k < 16; ++k)
            if (idx[k] >= 0) {
              asm volatile("prefetch.global.L2 [%0];" ::"l"(qh + (long long)idx[k] * DH));
              asm volatile("prefetch.global.L2 [%0];" ::"l"(qh + (long long)idx[k] * DH + 64));
            }
        }
        // both Q tiles are free once the previous item's last Q K^T has run
        if (n >= 1) mbar_wait(&sm->q_empty, (n - 1) & 1, abort_flag, p.status);
        const uint32_t dst = smem_u32(sQ) + r0 * 128 + ((chunk ^ (r0 & 7)) << 4);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          if (k >= 8 && it.nx == 1) break;
          const uint32_t to = dst + (k >> 3) * TILE + (k & 7) * 2048;
          const __nv_bfloat16* row = qh + (long long)max(idx[k], 0) * DH;
          const uint32_t bytes = idx[k] < 0 ? 0u : 16u;        // rows beyond the item's are zero-filled
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(row), "r"(bytes) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to + PANEL), "l"(row + 64), "r"(bytes) : "memory");
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        fence_async_proxy();
        mbar_arrive(&sm->q_full);
      }
      if (n >= 1) epilogue(before);
      before = it;
    }
    if (n >= 1) epilogue(before);
  } else if (warp >= 4) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 200;");
    // ------------------------------------------------------------------ softmax of one query tile
    const int x = (warp - 4) >> 2;                  // query tile of this warp group
    const int quad = warp & 3;                      // TMEM lane quarter this warp may access
    const int r = quad * 32 + lane;                 // query row inside the tile
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t s_tmem = tmem + lane_addr;
    const uint32_t p_tmem = tmem + lane_addr + P_COL + x * 64;
    const uint32_t o_tmem = tmem + lane_addr + O_COL + x * 128;
    uint32_t tc = 0, items = 0;                      // key tiles and items done on this query tile
    for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
      const FwdItem it = decode_item<DENSE>(p, item);
      if (x >= it.nx) continue;
      float m_used = -INFINITY, l = 0.f, l_r = 0.f;   // l: exact sum (for LSE); l_r: sum of the bf16-rounded weights
      for (int t = 0; t < it.ntiles; ++t, ++tc) {
        lap(3);
        mbar_wait(&sm->s_full[x], tc & 1, abort_flag, p.status);
        lap(0);
        tc_fence_after();
        const int valid = min(BN, it.n_keys - t * BN);
        uint32_t sv[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_tmem + 32 * c, *reinterpret_cast<uint32_t(*)[32]>(&sv[32 * c]));
        tmem_ld_wait();
        tc_fence_before();
        mbar_arrive(&sm->s_free);                    // the other tile's Q K^T may have the buffer
        if (valid < BN) {                            // keys beyond the range get score -inf
#pragma unroll
          for (int i = 0; i < BN; ++i)
            if (i >= valid) sv[i] = 0xff800000u;
        }
        float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
        for (int i = 0; i < BN; i += 8) {
          mx0 = max3(mx0, __uint_as_float(sv[i]), __uint_as_float(sv[i + 1]));
          mx1 = max3(mx1, __uint_as_float(sv[i + 2]), __uint_as_float(sv[i + 3]));
          mx2 = max3(mx2, __uint_as_float(sv[i + 4]), __uint_as_float(sv[i + 5]));
          mx3 = max3(mx3, __uint_as_float(sv[i + 6]), __uint_as_float(sv[i + 7]));
        }
        const float mx = fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * p.scale_log2;     // exp2 domain from here on (the scale is positive)
        lap(1);
        // lazy rescale: keep the old reference max unless the new one is more than 2^8 larger
        float factor = 1.0f;
        bool need = false;
        if (t == 0) {
          m_used = mx;
        } else if (mx > m_used + RESCALE_LOG2) {
          factor = ex2(m_used - mx);
          m_used = mx;
          need = true;
        }
        auto rescale_o = [&]() {                     // P V of the tile before is complete
#pragma unroll 1
          for (int c = 0; c < 8; ++c) {
            uint32_t ov[16];
            tmem_ld16(o_tmem + c * 16, ov);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * factor);
            tmem_st16(o_tmem + c * 16, ov);
          }
        };
        float s0 = 0.f, s1 = 0.f, r0 = 0.f, r1 = 0.f;
        const float neg_m = -m_used;
        {
          // the first half's weights stay in registers until P V of the tile before has read the P buffer
          uint32_t pk[2][16];
          exp_pack32(sv, p.scale_log2, neg_m, pk[0], s0, s1, r0, r1);
          // an early look, because the answer takes its time (33K dense forward 6.19 -> 6.10 ms); the wait follows if it was too early
          const uint32_t pv_done = mbar_test_wait(&sm->o_done[x], (tc + 1) & 1);
          if (valid > 32) exp_pack32(sv + 32, p.scale_log2, neg_m, pk[1], s0, s1, r0, r1);
          lap(3);
          if (tc > 0) {                              // (of the item before, where t is 0)
            if (!__all_sync(0xffffffffu, pv_done)) mbar_wait(&sm->o_done[x], (tc - 1) & 1, abort_flag, p.status);
            tc_fence_after();
            if (t > 0 && __any_sync(0xffffffffu, need)) {
              rescale_o();
              l *= factor;
              l_r *= factor;
            }
          }
          lap(2);
          tmem_st16(p_tmem, pk[0]);
          tmem_st16(p_tmem + 16, pk[1]);             // (whatever it holds where valid <= 32: P V does not read it)
        }
#pragma unroll
        for (int c = 2; c < 4; ++c) {
          if (32 * c < valid) {                      // (uniform; P V takes the keys up to `valid` only)
            uint32_t pk[16];
            exp_pack32(sv + 32 * c, p.scale_log2, neg_m, pk, s0, s1, r0, r1);
            tmem_st16(p_tmem + 16 * c, pk);
          }
        }
        l += s0 + s1;
        l_r += r0 + r1;
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(&sm->p_ready[x]);
      }
      // ---- hand the row's normalisers to the epilogue warps, once they are through with the tile's previous item, and go on
      lap(3);
      if (items >= 1) mbar_wait(&sm->o_free[x], (items - 1) & 1, abort_flag, p.status);
      sm->ep_inv[x][r] = 1.0f / l_r;
      sm->ep_lse[x][r] = (m_used + log2f(l)) * 0.6931471805599453f;
      mbar_arrive(&sm->ep_ready[x]);
      ++items;
      lap(4);
    }
    if (warp == 4 && lane == 0) tflush(0);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

static int grid_items(long long items) { return (int)std::max<long long>(1, std::min<long long>(items, sm_count())); }

template <bool DENSE, bool RASTER>
static int launch_wide(const Dims& D, const void* q, const void* k, const void* v, const Params& p, int grid, cudaStream_t st) {
  CUtensorMap tmK, tmV, tmQ;
  const uint64_t rows = (uint64_t)D.BH * D.S;
  if (!sm100::make_tmap_bf16_rows(&tmK, k, rows, DH, BN) || !sm100::make_tmap_bf16_rows(&tmV, v, rows, DH, BN) ||
      !sm100::make_tmap_bf16_heads(&tmQ, q, D.BH, D.S, DH, BM))      // dense: consecutive rows; sparse: not used
    return VMOBA_ERR_CUDA;
  auto kernel = p.prof ? attn_fwd_wide_kernel<DENSE, RASTER, true> : attn_fwd_wide_kernel<DENSE, RASTER, false>;
  VMOBA_CUDA_OK(allow_smem(kernel, (int)SMEM_BYTES));
  launch_kernel(kernel, grid, THREADS, SMEM_BYTES, st, tmK, tmV, tmQ, p);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

}  // namespace tcw

int tc_sparse_fwd_narrow(const Dims& D, const void* q, const void* k, const void* v, const int* kb_ptr, const int* q_idx,
                         const int* q_ptr, const int* q_pairs, long long cap, void* o, void* o_resid, float* lse,
                         int32_t* status, int* item_ptr, int* item_tab, long long max_items, float* part_o,
                         float* part_lse, float* part_scale, cudaStream_t st, const RowMap& o_map);   // attn_tc_fwd_narrow.cu

// Forward over the work lists (bf16, head_dim 128).  Key blocks of up to two 128-key tiles go to the narrow kernel (two
// CTAs of one query tile per SM), longer ones to the wide kernel of this file.  Returns VMOBA_ERR_CUDA if the tensor maps
// or the launch fail.
int tc_sparse_fwd(const Dims& D, const void* q, const void* k, const void* v, const int* kb_ptr, const int* q_idx,
                       const int* q_ptr, const int* q_pairs, long long cap, void* o, void* o_resid, float* lse,
                       int32_t* status, int* item_ptr, int* item_tab, long long max_items, float* part_o,
                       float* part_lse, float* part_scale, cudaStream_t st, const RowMap& o_map) {
  using namespace tcw;
  // Measured (forward stage, wide against narrow): 13 tiles and lists of thousands 1.91 against 2.40 ms, 6 tiles 1.19
  // against 1.46, 3 tiles 0.82 against 1.02; two tiles with lists of 200 queries (33K tokens, 3D blocks of 234 keys)
  // 0.400 against 0.365: a 256-row item is then over before its two halves have fallen into step.
  if (D.sb <= 2 * BN)
    return tc_sparse_fwd_narrow(D, q, k, v, kb_ptr, q_idx, q_ptr, q_pairs, cap, o, o_resid, lse, status, item_ptr, item_tab,
                                max_items, part_o, part_lse, part_scale, st, o_map);
  const long long n_kb = (long long)D.BH * D.Nb;
  simt::make_items(kb_ptr, n_kb, IM, cap, max_items, item_ptr, reinterpret_cast<int4*>(item_tab), st);
  Params p;
  p.q = (const __nv_bfloat16*)q; p.q_idx = q_idx; p.q_ptr = q_ptr; p.item_ptr = item_ptr;
  p.item_desc = reinterpret_cast<const int4*>(item_tab);
  p.n_kb = (int)n_kb; p.S = D.S; p.Nb = D.Nb; p.sb = D.sb; p.BH = D.BH;
  p.scale_log2 = D.scale * 1.4426950408889634f;
  p.o = (__nv_bfloat16*)o; p.o_resid = (__nv_bfloat16*)o_resid; p.lse = lse;
  p.part_o = reinterpret_cast<__half*>(part_o); p.part_lse = part_lse; p.part_scale = part_scale;
  p.status = status; p.prof = debug_wait_profile();
  p.o_map = o_map;
  p.part_o_32 = (reinterpret_cast<uintptr_t>(part_o) % 32) == 0;
  if (o_map.perm) {
    if (int rc = launch_wide<false, true>(D, q, k, v, p, grid_items(cap / IM + n_kb), st)) return rc;
  } else {
    if (int rc = launch_wide<false, false>(D, q, k, v, p, grid_items(cap / IM + n_kb), st)) return rc;
  }
  simt::merge_batched(D, q_ptr, q_pairs, p.part_o, part_lse, part_scale, cap, o, o_resid, lse, o_map, st);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

int tc_dense_fwd(const Dims& D, const void* q, const void* k, const void* v, void* o, void* o_resid, float* lse,
                      int32_t* status, cudaStream_t st) {
  using namespace tcw;
  Params p;
  p.q = (const __nv_bfloat16*)q; p.q_idx = nullptr; p.q_ptr = nullptr; p.item_ptr = nullptr; p.item_desc = nullptr;
  p.n_kb = 0; p.S = D.S; p.Nb = 1; p.sb = D.S; p.BH = D.BH;
  p.scale_log2 = D.scale * 1.4426950408889634f;
  p.o = (__nv_bfloat16*)o; p.o_resid = (__nv_bfloat16*)o_resid; p.lse = lse; p.part_o = nullptr; p.part_lse = nullptr; p.part_scale = nullptr;
  p.part_o_32 = 0; p.o_map = RowMap();
  p.status = status; p.prof = debug_wait_profile();
  const long long items = (long long)D.BH * ((D.S + IM - 1) / IM);
  return launch_wide<true, false>(D, q, k, v, p, grid_items(items), st);
}

}  // namespace vmoba
