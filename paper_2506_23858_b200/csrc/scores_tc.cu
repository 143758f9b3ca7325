// Tensor-core path of the similarity map S_hat = q b^T (Section 3.3) for bf16 queries, head_dim 128.
//
// The scores must carry fp32 accuracy (the selection cutoff is compared in fp32), but the
// centroids b are fp32.  An fp32 number is exactly the sum of three bf16 numbers (3 x 8 mantissa
// bits), so each centroid row is split b = b1 + b2 + b3 and the product runs as three bf16 MMAs
// into one fp32 TMEM accumulator; q is bf16 already, so every product is exact and only the fp32
// accumulation rounds.
//
// Persistent CTAs walk (head, block range, 128-query tile) items: the three centroid parts of
// the block range stay in shared memory, query tiles stream through a TMA ring that takes the shared memory the parts
// leave (2 tiles beside 160 centroid rows, 5 beside 32), the accumulator is double buffered in TMEM.
//
// Bound by HBM: q is read once, the fp32 [S, N_b] matrix written once.  What stood between was the epilogue (per item 128
// rows x N_b scores out of TMEM), so two sets of four warps take its 32-column slabs in turn, and no warp waits for
// another: a warp puts 32 rows x 32 columns into its own swizzled 4 KB slab and sends it with one TMA store.  Rows that are
// not multiples of 16 bytes (N_b % 4 != 0) leave the slab as one run of consecutive words per row instead.
// Before, with one set of four warps, two CTA-wide barriers per slab and 4-byte stores a row apart for N_b % 4 != 0, and now:
// 12 heads x 55,296 queries x 72 blocks 72 -> 61 us (floor 55), 32,760 x 140 70 -> 67 (49), 75,600 x 280 338 -> 315 (249),
// 75,600 x 350 2350 -> 643 (230), 40 heads x 75,600 x 21 461 -> 265 (157).  Both sets work on one item: with an item each,
// 32,760 x 140 took 71 (its rows of 560 bytes leave sectors half written for longer); boxes of 128 rows 76; staging whole
// rows and copying them in bulk 124.
#include <algorithm>

#include "sm100.cuh"

namespace vmoba {
namespace sct {

using namespace sm100;

constexpr int BM = 128, DH = 128;
constexpr int PANEL = 128 * 128;
constexpr int TILE = 2 * PANEL;
constexpr int NT_MAX = 160;              // centroid rows (key blocks) per pass
constexpr int THREADS = 320;             // TMA, MMA, two epilogue sets of four warps
constexpr int NQ_MAX = 5;
constexpr uint32_t TMEM_COLS = 512;      // two accumulators of up to 160 columns, at columns 0 and 256

struct Smem {
  uint64_t q_full[NQ_MAX], q_empty[NQ_MAX];
  uint64_t b_full, b_empty;
  uint64_t acc_full[2], acc_empty[2];
  uint64_t drain;                         // (after a time-out only)
  uint32_t tmem_base;
  int abort_flag;
};
constexpr int SLAB = 32 * 128;            // 32 rows x 32 fp32 columns, one per epilogue warp
constexpr int SLABS = 8;
constexpr int SMEM_MAX = 227 * 1024;
// query tiles [nq], 3 centroid parts of two 64-column panels (rows_pass rows x 128 bytes), slabs, barriers
inline int smem_bytes(int nq, int rows_pass) {
  return 1024 + nq * TILE + 6 * rows_pass * 128 + SLABS * SLAB + (int)sizeof(Smem) + 64;
}

struct Params {
  float* scores;
  int S, Nb, Nb_pad, BH;
  int n_pass, rows_pass;    // block ranges per head, rows per range (multiple of 16, <= NT_MAX)
  int nq;                   // query tiles in the ring
  int tma_store;            // rows are multiples of 16 bytes: the epilogue writes through tmS
  float* range;             // optional [BH][2]: smallest and largest score of each head (starts at +inf, -inf)
  int32_t* status;
};

__global__ void __launch_bounds__(THREADS, 1)
scores_tc_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmB,
                 const __grid_constant__ CUtensorMap tmS, const Params p) {
  if (!grid_begin()) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nq = p.nq;
  const int bpanel = p.rows_pass * 128, bpart = 2 * bpanel;      // multiples of 4096
  uint8_t* sQ = base;                    // [nq][TILE]
  uint8_t* sB = base + nq * TILE;        // [3][bpart]
  uint8_t* sOut = sB + 3 * bpart;        // [SLABS][SLAB]
  Smem* sm = reinterpret_cast<Smem*>(sOut + SLABS * SLAB);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &sm->abort_flag;

  if (threadIdx.x == 0) {
    for (int i = 0; i < nq; ++i) { mbar_init(&sm->q_full[i], 1); mbar_init(&sm->q_empty[i], 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm->acc_full[i], 1); mbar_init(&sm->acc_empty[i], 256);
    }
    mbar_init(&sm->b_full, 1);
    mbar_init(&sm->b_empty, 1);
    mbar_init(&sm->drain, 1);
    sm->abort_flag = 0;
    fence_barrier_init();
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmB);
  }
  if (warp == 1) {
    tmem_alloc(&sm->tmem_base, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem_base;

  // items: (bh, pass, tile), tile fastest; each CTA takes one contiguous range so that the centroid
  // parts of a (bh, pass) are loaded once per CTA
  const int tiles = (p.S + BM - 1) / BM;
  const long long n_items = (long long)p.BH * p.n_pass * tiles;
  const long long per = (n_items + gridDim.x - 1) / gridDim.x;
  const long long it0_ = (long long)blockIdx.x * per;
  const long long it0 = it0_ < n_items ? it0_ : n_items;
  const long long it1 = it0 + per < n_items ? it0 + per : n_items;
  const long long n_part_rows = (long long)p.BH * p.Nb_pad;

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t bn = 0;
      int s = 0, ph = 1, filled = 0;                  // ring slot, parity of its wait, slots ever filled
      long long cur_group = -1;
      for (long long it = it0; it < it1; ++it) {
        const int tile = (int)(it % tiles);
        const long long group = it / tiles;            // bh * n_pass + pass
        const int pass = (int)(group % p.n_pass);
        const long long bh = group / p.n_pass;
        if (group != cur_group) {
          // new centroid range: wait until the MMAs that read the old one are done
          if (bn > 0 && !mbar_wait(&sm->b_empty, (bn - 1) & 1, abort_flag, p.status)) break;      // (nothing is loaded after a time-out)
          const int y0 = (int)(bh * p.Nb_pad + (long long)pass * p.rows_pass);
          mbar_expect_tx(&sm->b_full, 3 * 2 * p.rows_pass * 128);
          for (int part = 0; part < 3; ++part) {
            const int y = (int)(part * n_part_rows) + y0;
            tma_load_2d(sB + part * bpart, &tmB, &sm->b_full, 0, y);
            tma_load_2d(sB + part * bpart + bpanel, &tmB, &sm->b_full, 64, y);
          }
          cur_group = group;
          ++bn;
        }
        if (filled < nq) ++filled;
        else if (!mbar_wait(&sm->q_empty[s], ph, abort_flag, p.status)) break;
        const int y = (int)(bh * p.S) + tile * BM;
        mbar_expect_tx(&sm->q_full[s], TILE);
        tma_load_2d(sQ + s * TILE, &tmQ, &sm->q_full[s], 0, y);
        tma_load_2d(sQ + s * TILE + PANEL, &tmQ, &sm->q_full[s], 64, y);
        if (++s == nq) { s = 0; ph ^= 1; }
      }
      if (*abort_flag) {
        // the newest load of every slot: in this lap of the ring for slots below s, in the one before for the others
        for (int f = 0; f < filled; ++f) mbar_wait(&sm->q_full[f], (f < s ? ph : ph ^ 1) ^ 1, abort_flag, p.status);
        if (bn > 0) mbar_wait(&sm->b_full, (bn - 1) & 1, abort_flag, p.status);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer: the whole warp walks the loop, one
    // elected lane issues (warp-uniform control flow; see elect_one)
    {
      const bool leader = elect_one();
      uint32_t qn = 0, bn = 0;
      int s = 0, ph = 0;
      long long cur_group = -1;
      const uint32_t idesc = make_idesc_bf16(BM, p.rows_pass, false, false);
      for (long long it = it0; it < it1; ++it, ++qn) {
        const long long group = it / tiles;
        if (group != cur_group) {
          // all MMAs on the previous range were issued before this point: release it to the producer
          if (leader && cur_group >= 0) mma_commit(&sm->b_empty);
          mbar_wait_warp(&sm->b_full, bn & 1, abort_flag, p.status);
          cur_group = group;
          ++bn;
        }
        const int e = qn & 1;
        mbar_wait_warp(&sm->q_full[s], ph, abort_flag, p.status);
        if (qn >= 2) mbar_wait_warp(&sm->acc_empty[e], ((qn >> 1) - 1) & 1, abort_flag, p.status);
        tc_fence_after();
        const uint32_t d_tmem = tmem + (e ? 256u : 0u);
        const uint32_t sQ_addr = smem_u32(sQ + s * TILE);
#pragma unroll 1
        for (int part = 0; part < 3; ++part) {
          const uint32_t sB_addr = smem_u32(sB + part * bpart);
#pragma unroll
          for (int ks = 0; ks < DH / 16; ++ks) {
            const uint64_t a = make_smem_desc(sQ_addr + (ks >> 2) * PANEL + (ks & 3) * 32, 16, 1024);
            const uint64_t b = make_smem_desc(sB_addr + (ks >> 2) * bpanel + (ks & 3) * 32, 16, 1024);
            if (leader) mma_ss(d_tmem, a, b, idesc, (part > 0 || ks > 0) ? 1u : 0u);
          }
        }
        if (leader) mma_commit(&sm->q_empty[s]);
        if (leader) mma_commit(&sm->acc_full[e]);
        if (++s == nq) { s = 0; ph ^= 1; }
      }
      if (leader && *abort_flag) mma_drain(&sm->drain);
    }
  } else {
    // ------------------------------------------------------------------ epilogue: thread = query row
    const int set = warp >= 6;                        // takes every other slab, counted on through the items
    const int quad = warp & 3;
    const int r = quad * 32 + lane;
    const uint32_t a_tmem = tmem + ((uint32_t)(quad * 32) << 16);
    uint8_t* slab = sOut + (warp - 2) * SLAB;
    uint32_t qn = 0;
    int turn = set;                                   // 1: the slab before was this set's, the next is not
    // smallest / largest score seen by this thread for the current head (the selection's first pass, taken
    // here while the scores are in registers); handed over with one atomic pair per warp when the head changes
    float rmin = INFINITY, rmax = -INFINITY;
    long long range_bh = -1;
    auto flush_range = [&]() {
      if (p.range && range_bh >= 0) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          rmin = fminf(rmin, __shfl_xor_sync(0xffffffffu, rmin, o));
          rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
        }
        if (lane == 0 && rmin <= rmax) {
          atomic_min_f32(p.range + 2 * range_bh, rmin);
          atomic_max_f32(p.range + 2 * range_bh + 1, rmax);
        }
      }
      rmin = INFINITY; rmax = -INFINITY;
    };
    for (long long it = it0; it < it1; ++it, ++qn) {
      const int tile = (int)(it % tiles);
      const long long group = it / tiles;
      const int pass = (int)(group % p.n_pass);
      const long long bh = group / p.n_pass;
      if (bh != range_bh) { flush_range(); range_bh = bh; }
      const int e = qn & 1;
      mbar_wait(&sm->acc_full[e], (qn >> 1) & 1, abort_flag, p.status);
      tc_fence_after();
      const int row = tile * BM + r, row0 = tile * BM + quad * 32;
      const int j0 = pass * p.rows_pass;
      const int ncols = min(p.rows_pass, p.Nb - j0);       // real blocks in this range
#pragma unroll 1
      for (int c0 = 0; c0 < ncols; c0 += 32) {
        turn ^= 1;
        if (turn == 0) continue;
        uint32_t v[32];
        tmem_ld32(a_tmem + (e ? 256u : 0u) + c0, v);
        tmem_ld_wait();
        const int nc = ncols - c0;                          // columns of this slab that exist, if below 32
        if (p.range && row < p.S) {
          if (nc >= 32) {
#pragma unroll
            for (int i = 0; i < 32; ++i) { rmin = fminf(rmin, __uint_as_float(v[i])); rmax = fmaxf(rmax, __uint_as_float(v[i])); }
          } else {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (i < nc) { rmin = fminf(rmin, __uint_as_float(v[i])); rmax = fmaxf(rmax, __uint_as_float(v[i])); }
          }
        }
        if (p.tma_store) {
          if (lane == 0) bulk_wait_group_read<0>();         // the slab's previous store must have read it
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<uint4*>(slab + lane * 128 + ((i ^ (lane & 7)) << 4)) = make_uint4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
          fence_async_proxy();
          __syncwarp();
          if (lane == 0 && row0 < p.S) {
            tma_store_3d(&tmS, slab, j0 + c0, row0, (int)bh);   // rows beyond S and columns beyond N_b are clipped
            bulk_commit_group();
          }
        } else {
          // word (row, column) at row * 32 + (row + column) % 32: neither side meets a bank twice
          uint32_t* words = reinterpret_cast<uint32_t*>(slab);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < 32; ++i) words[lane * 32 + ((lane + i) & 31)] = v[i];
          __syncwarp();
          uint32_t* out = reinterpret_cast<uint32_t*>(p.scores) + ((long long)bh * p.S + row0) * p.Nb + j0 + c0 + lane;
          if (lane < nc) {
            const int rows = min(32, p.S - row0);
#pragma unroll 8
            for (int i = 0; i < rows; ++i) out[(long long)i * p.Nb] = words[i * 32 + ((lane + i) & 31)];
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&sm->acc_empty[e]);
    }
    flush_range();
    if (lane == 0) bulk_wait_group<0>();      // shared memory must outlive the last stores' reads
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace sct

size_t scores_tc_ws_bytes(const Dims& D) {
  const size_t Nb_pad = (size_t)(D.Nb + 31) / 32 * 32;
  return 3 * (size_t)D.BH * Nb_pad * sct::DH * sizeof(__nv_bfloat16) + 1024;
}

// Where the centroid kernel leaves the parts: [3][BH][Nb_pad][128], rows of whole 32-column slabs (the epilogue's store unit).
CentroidParts scores_tc_parts(const Dims& D, void* ws) {
  CentroidParts c;
  c.Nb_pad = (D.Nb + 31) / 32 * 32;
  c.parts = reinterpret_cast<__nv_bfloat16*>((reinterpret_cast<uintptr_t>(ws) + 1023) & ~uintptr_t(1023));
  c.n = (long long)D.BH * c.Nb_pad * sct::DH;
  return c;
}

// scores [BH, S, Nb] fp32 from block-major bf16 q and the centroids' parts (already there; range, if given, starts at +inf, -inf).
int scores_tc(const Dims& D, const void* q_bm, const CentroidParts& cent, float* scores, float* range, int32_t* status, cudaStream_t st) {
  using namespace sct;
  const int Nb_pad = cent.Nb_pad;
  const int n_pass = (Nb_pad + NT_MAX - 1) / NT_MAX;
  const int rows_pass = ((Nb_pad + n_pass - 1) / n_pass + 31) / 32 * 32;
  CUtensorMap tmQ, tmB, tmS;
  const int tma_store = (D.Nb % 4 == 0) && (reinterpret_cast<uintptr_t>(scores) % 16 == 0);
  if (tma_store) {
    if (!sm100::make_tmap_f32_planes(&tmS, scores, (uint64_t)D.BH, (uint64_t)D.S, (uint64_t)D.Nb, 32)) return VMOBA_ERR_CUDA;
  } else {
    tmS = CUtensorMap{};
  }
  if (!sm100::make_tmap_bf16_rows(&tmQ, q_bm, (uint64_t)D.BH * D.S, DH, BM) ||
      !sm100::make_tmap_bf16_rows(&tmB, cent.parts, (uint64_t)3 * D.BH * Nb_pad, DH, rows_pass))
    return VMOBA_ERR_CUDA;
  Params p;
  p.scores = scores; p.S = D.S; p.Nb = D.Nb; p.Nb_pad = Nb_pad; p.BH = D.BH; p.n_pass = n_pass; p.rows_pass = rows_pass;
  p.tma_store = tma_store;
  p.nq = NQ_MAX;
  while (smem_bytes(p.nq, rows_pass) > SMEM_MAX) --p.nq;      // (two tiles fit beside 160 rows)
  p.range = range;
  p.status = status;
  VMOBA_CUDA_OK(allow_smem(scores_tc_kernel, SMEM_MAX));
  const long long items = (long long)D.BH * n_pass * ((D.S + BM - 1) / BM);
  launch_kernel(scores_tc_kernel, (int)std::max<long long>(1, std::min<long long>(items, sm_count())), THREADS,
                smem_bytes(p.nq, rows_pass), st, tmQ, tmB, tmS, p);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

}  // namespace vmoba
