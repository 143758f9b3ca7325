// Tensor-core attention backward for bf16, head_dim 128: the training backward of Step 3 of VMoBA (mask constant) and
// of the dense path.  One persistent kernel (one CTA per SM), key-stationary, all three gradients:
//
//   Item = 128 keys of one key block.  The K and V tiles stay in shared memory; the queries that selected the block
//   stream through in gathered units of 128 (Q and dO rows).  Per unit, with keys on the TMEM lanes:
//     S^T = K Q^T                                        (SS MMA)
//     P^T = exp2(c S^T - lse)                            (compute warps; bf16 into the S^T columns)
//     dV += P^T dO                                       (TS MMA, A = P^T)
//     dP^T = V dO^T                                      (SS)
//     dS^T = P^T (dP^T - D)                              (compute warps; bf16 into the dP^T columns and into shared memory)
//     dK += dS^T Q                                       (TS, A = dS^T)
//     dQ^T = K^T dS^T                                    (SS: K tile read MN-major as A, dS^T as the [keys][queries] tile;
//                                                         lands in the dP^T columns)
//   Every key belongs to exactly one item: dK and dV are written once, no atomics.  dQ^T is read out of TMEM by eight
//   writer warps and added into an fp32 accumulator with red.global.add.v4.f32 (per warp instruction: complete 128-byte
//   lines of four query rows).  Sparse: in whatever order the items come to it, so dQ is repeatable to rounding only.  Dense:
//   key tile after key tile, see Turns below; the whole dense backward repeats bit for bit.
//
// What bounds it is the shared-memory port (128 bytes per cycle).  A shared-memory MMA with N = 128 fetches 8 KB of
// operands in its 64 cycles, a TS one 4 KB; per 128 x 128 unit that is 2048 cycles of operands against 2560 cycles of
// tensor math, beside 512 cycles for the landing Q / dO rows and 256 for the dS^T tile.  Hence
//   * units of 128 queries: with 64 (N = 64) an SS MMA fetches 6 KB for half the math;
//   * P^T and dS^T as TMEM operands; dQ^T in the columns that dP^T and dS^T no longer need (S^T | dP^T | dV | dK fill the
//     512 columns, so nothing is double-buffered and the order of the MMAs carries the overlap, see the MMA warp);
//   * scores read and results written in the 16-row fragment shapes (16x256b in, 16x128b out, stmatrix): a thread then
//     holds 16 different queries instead of 64, and lse and D are 16 eight-byte shared-memory reads instead of 128 shuffles;
//     dQ^T read in the same shape needs no transposition before the reductions.
//
// D = rowsum(dO * O) and lse come in per query; exp runs in the exp2 domain (c = scale * log2 e).
#include <algorithm>

#include "attn_simt.cuh"
#include "sm100.cuh"

namespace vmoba {
namespace tcb {

using namespace sm100;

constexpr int BN = 128, DH = 128;
constexpr int QU = 128;                      // queries per unit
constexpr int PANEL = 128 * 128;             // bytes of one 64-column panel of a 128-row tile (16 KB)
constexpr int TILE = 2 * PANEL;              // [128 x 128] bf16 (32 KB)
constexpr uint32_t TMEM_COLS = 512;
constexpr uint32_t ST_COL = 0, DPT_COL = 128, DV_COL = 256, DK_COL = 384;
constexpr uint32_t ROW16 = 16u << 16;        // TMEM lanes 16 .. 31 of a warp's quarter
constexpr float LOG2E = 1.4426950408889634f;
// Diagnostics: when a device buffer of 16 counters is registered, the kernel adds the cycles its roles spend in each
// wait (one representative thread per role and CTA).
static unsigned long long* g_wait_profile = nullptr;

// A unit's Q tile is held from S^T, issued one unit early, to dK at its end; its dO tile only from dP^T to dV, in the
// middle.  So three Q tiles and one dO tile keep both gathers ahead (with two of each the MMA warp waited 1250 of a unit's
// 5000 cycles for Q rows).
constexpr int NQ = 3;

struct KvSmem {
  uint64_t k_full, k_empty, v_full, v_empty;                       // K / V tile of an item (TMA / commit)
  uint64_t q_full[NQ], q_empty[NQ], do_full, do_empty;             // gathered Q / dO rows of a unit (loader arrivals / commit)
  uint64_t s_full, p_ready;                                        // S^T complete (commit) / P^T written (256 arrivals)
  uint64_t dp_full, ds_ready;                                      // dP^T complete (commit) / dS^T written (256 arrivals)
  uint64_t dq_full, dq_free;                                       // dQ^T complete (commit) / read out of TMEM (256 arrivals)
  uint64_t acc_done, acc_free;                                     // dV / dK of an item complete (commit) / read (256 arrivals)
  uint64_t turn_ok, rows_out, rows_seen;                           // dense: it is this tile's turn / its dQ is on the way (256 arrivals) / and noted
  uint64_t drain;                                                  // (after a time-out only)
  uint32_t tmem_base;
  int ticket;                                // dense: the CTA's item
  int abort_flag;
  alignas(16) float lse2[NQ][QU];            // lse * log2 e, with the Q rows of a unit
  alignas(16) float negD[2][QU];             // -rowsum(dO * O), with its dO rows
};
// K, V, three Q tiles and a dO tile, the dS^T tile ([128 keys][128 queries] bf16)
// no alignment slack: the kernel checks that its dynamic shared memory starts on a 1024-byte boundary
constexpr size_t SMEM_BYTES = 7 * TILE + sizeof(KvSmem) + 32;
static_assert(SMEM_BYTES <= 232448, "backward: shared memory");
// Warp groups: {TMA, MMA, -, -}, 4 Q loaders, 4 dO loaders, 2 x 4 compute, 2 x 4 dQ writers.  896 threads start with 72
// registers each; the compute groups, which keep a unit's 64 weights per thread from the first to the second step, take
// 112, the writers (64 values of dQ) 80, the first three groups keep 40: 2 x 112 + 2 x 80 + 3 x 40 = 7 x 72.
constexpr int THREADS = 896;
constexpr uint32_t IDESC_TN = make_idesc_bf16(128, 128, false, true);    // dV, dK: A from TMEM, B MN-major

// Turns (dense).  Every unit of every head has a counter: the number of key tiles whose dQ has been added there.  Key tile t
// adds to it when it stands at t (the first one stores, so nothing has to be cleared), so the sum is taken in one order
// whatever the timing.  A CTA takes one item, by a ticket drawn when it starts: the tiles an item waits for belong to lower
// tickets, which CTAs that are running hold, so the waiting ends whatever else occupies the device.  The key tiles of a head
// follow one another about a unit apart; tickets go round `group` heads, so that a head's tiles start few units apart
// (SMs / group) and come no faster than one per unit.  Two warps that have nothing else to do look at the counter and move it
// on (a fence behind the reductions, a look at another CTA's word): the writers see shared-memory barriers only.
// Where the tiles of a head are most of what there is to run, waiting for one another takes as long as the work.  Up to four
// accumulators with counters of their own, if they fit 128 MB, shorten the row: tile t adds to accumulator t % parts, and
// cast_rows adds these up.
// Measured, against reductions in any order and tiles that start at different units (forward and backward): 12 heads x 13,440
// tokens 3796 -> 3912 us, x 8,000 1448 -> 1498, 4 heads x 32,760 7713 -> 8221 (one accumulator); 12 x 3,000 218 -> 252, 12 x 1,000
// 71 -> 81, 1 x 3,000 132 -> 158 (four; with one 275, 100, 224; with dQ in a kernel of its own 376, 118, 227).  With the
// writers looking at the counters themselves 12 x 13,440 took 4798.
struct KvParams {
  const __nv_bfloat16 *q, *d_o;
  const float *lse, *Dv;
  const int *kb_ptr, *q_idx;   // null for the dense path: every query of the head meets every key tile
  int S, Nb, sb, BH;
  float scale, scale_log2;
  long long capacity;
  __nv_bfloat16 *dk, *dv;
  int dkv_32;                  // dk and dv are 32-byte aligned: rows go out with 32-byte stores
  RowMap out_map;              // where the dK / dV rows go (block-major, or raster order through perm)
  RowMap do_map;               // where the dO rows come from (likewise)
  float* dq_acc;               // fp32 [queries][head_dim]; sparse: zeroed rows of all selecting queries; columns in the order of the
                               // dQ writers: position 32 w + 4 r + a holds column 32 w + r + 8 a (r < 8, a < 4)
  int parts;                   // dense: accumulators (dq_acc holds that many of [queries][head_dim])
  int* turns;                  // dense: [parts][BH][units], then the ticket; zero at the start
  int group;                   // dense: heads whose key tiles are taken in turn
  int32_t* status;
  unsigned long long* prof;    // optional wait-time counters (diagnostics), or null
};

struct KvItem {
  int bh, key0, valid, n_list, n_units, tile;
  int list_lo, head_off;       // positions and rows fit 31 bits (capacity, B * heads * S <= 2^30)
};

template <bool DENSE>
__device__ __forceinline__ KvItem kv_decode(const KvParams& p, int item, int tiles) {
  KvItem it;
  if constexpr (DENSE) {
    // groups of heads; in a group, the first key tile of every head, then the second ones
    const int per = p.group * tiles, first = item / per * p.group, heads = min(p.group, p.BH - first), r = item % per;
    it.tile = r / heads;
    it.bh = first + r - it.tile * heads;
    it.key0 = it.tile * BN;
    it.valid = min(BN, p.S - it.key0);
    it.head_off = it.bh * p.S;
    it.list_lo = 0;
    it.n_list = p.S;
  } else {
    const int kbi = item / tiles;
    it.tile = item - kbi * tiles;
    it.bh = kbi / p.Nb;
    it.key0 = (kbi - it.bh * p.Nb) * p.sb + it.tile * BN;
    it.valid = min(BN, p.sb - it.tile * BN);
    it.head_off = it.bh * p.S;
    long long lo = min((long long)p.kb_ptr[kbi], p.capacity), hi = min((long long)p.kb_ptr[kbi + 1], p.capacity);
#ifdef VMOBA_DEBUG
    if (lo < 0 || hi < lo) {      // offsets must be non-negative and ascending
      set_status(p.status, VMOBA_ERR_BOUNDS);
      lo = hi = 0;
    }
#endif
    it.list_lo = (int)lo;
    it.n_list = (int)(hi - lo);
  }
  it.n_units = (it.n_list + QU - 1) / QU;
  return it;
}

// Walks the units of all items of this CTA, one per next().
template <bool DENSE>
struct UnitWalk {
  KvItem it;
  int item, i, n_items, tiles, first, rows;
  __device__ __forceinline__ UnitWalk(int first_item, int n_items_, int tiles_)
      : item(first_item - (int)gridDim.x), i(0), n_items(n_items_), tiles(tiles_), first(0), rows(0) { it.n_units = 0; }
  __device__ __forceinline__ bool next(const KvParams& p) {
    while (i >= it.n_units) {
      item += gridDim.x;
      if (item >= n_items) return false;
      it = kv_decode<DENSE>(p, item, tiles);
      i = 0;
    }
    first = i * QU;
    rows = min(QU, it.n_list - first);
    ++i;
    return true;
  }
  // in-head position of the query in row `row` of the unit, -1 for a padding row
  __device__ __forceinline__ int entry(const KvParams& p, int row) const {
    if (row >= rows) return -1;
    return DENSE ? first + row : checked_index(__ldg(p.q_idx + it.list_lo + first + row), p.S, p.status);
  }
};

// Asynchronous 16-byte copy global -> shared (bypassing L1); `bytes` = 16, or 0 to write zeros.
__device__ __forceinline__ void cp_async16(uint32_t smem_dst, const void* gsrc, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gsrc), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
// 16-byte vector reduction into global memory (fp32 add)
__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// Waits (bounded) until a turn counter has reached `turn`; the reductions of other threads follow a barrier.
__device__ __forceinline__ void turn_wait(const int* addr, int turn, volatile int* abort_flag, int32_t* status) {
  constexpr uint32_t kPolls = 1u << 22;
  const uint32_t limit = *abort_flag ? 16u : kPolls;
  for (uint32_t i = 0; i < limit; ++i) {
    int at;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(at) : "l"(addr) : "memory");
    if (at >= turn) return;
    __nanosleep(32);
  }
  *abort_flag = 1;
  set_status(status, VMOBA_ERR_TIMEOUT);
}
// Passes the turn on, at device scope: behind the reductions of the threads whose barrier this one has waited for.
__device__ __forceinline__ void turn_pass(int* addr, int next) {
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(addr), "r"(next) : "memory");
}

__device__ __forceinline__ uint32_t lo_k(uint32_t tile_addr) { return desc_lo(tile_addr, 16); }
__device__ __forceinline__ uint32_t lo_mn(uint32_t tile_addr) { return desc_lo(tile_addr, PANEL); }
__device__ __forceinline__ constexpr uint32_t koff(int ks) { return (uint32_t)(((ks >> 2) * PANEL + (ks & 3) * 32) >> 4); }
__device__ __forceinline__ constexpr uint32_t mnoff(int ks) { return (uint32_t)((ks * 2048) >> 4); }

// Fragment shapes.  16x256b: of 16 TMEM lanes x 8 columns per repetition j, thread l holds lane l / 4 (registers 4j,
// 4j+1) and lane l / 4 + 8 (4j+2, 4j+3), columns 8j + 2 (l % 4) and the next.  16x128b: lane l / 4 (2j) and l / 4 + 8
// (2j+1), column 4j + l % 4: two neighbouring fp32 columns of the first, rounded and packed, are one of the second.
__device__ __forceinline__ void tmem_ld_16x256_x8(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st_16x128_x4(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.16x128b.x4.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// four 8x8 bf16 matrices; lane i gives the address of row i % 8 of matrix i / 8
__device__ __forceinline__ void stmatrix_x4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}

// MULTI (dense): several accumulators (with p.parts read in the one kernel, the case of one ran 4 % slower).
template <bool DENSE, bool MULTI, bool PROF>
__global__ void __launch_bounds__(THREADS, 1)
attn_bwd_fused_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                      const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmO, const KvParams p) {
  if (!grid_begin()) return;
  extern __shared__ uint8_t smem_raw[];
  // the swizzled tiles need 1024-byte alignment and there is no room for alignment slack
  if ((smem_u32(smem_raw) & 1023u) != 0) {
    if (threadIdx.x == 0) set_status(p.status, VMOBA_ERR_CUDA);
    return;
  }
  uint8_t* sK = smem_raw;
  uint8_t* sV = smem_raw + TILE;
  uint8_t* sQ = smem_raw + 2 * TILE;           // [NQ]
  uint8_t* sO = smem_raw + (2 + NQ) * TILE;    // dO
  uint8_t* sDS = smem_raw + 6 * TILE;
  KvSmem* sm = reinterpret_cast<KvSmem*>(smem_raw + 7 * TILE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &sm->abort_flag;
  // diagnostics: cycles spent in each wait site by one representative thread per role
  unsigned long long wp[4] = {0, 0, 0, 0};
  const long long t_begin = PROF ? clock64() : 0;
  auto twait = [&](int site, uint64_t* bar, uint32_t parity) {
    if constexpr (PROF) {
      const long long t0 = clock64();
      const bool ok = mbar_wait(bar, parity, abort_flag, p.status);
      wp[site] += (unsigned long long)(clock64() - t0);
      return ok;
    } else {
      return mbar_wait(bar, parity, abort_flag, p.status);
    }
  };
  auto tflush = [&](int base_site, int nsites) {
    if constexpr (PROF) {
      for (int i = 0; i < nsites; ++i) atomicAdd(p.prof + base_site + i, wp[i]);
      atomicAdd(p.prof + base_site + nsites, (unsigned long long)(clock64() - t_begin));
    }
  };

  if (threadIdx.x == 0) {
    mbar_init(&sm->k_full, 1); mbar_init(&sm->k_empty, 1);
    mbar_init(&sm->v_full, 1); mbar_init(&sm->v_empty, 1);
    for (int b = 0; b < NQ; ++b) { mbar_init(&sm->q_full[b], 128); mbar_init(&sm->q_empty[b], 1); }
    mbar_init(&sm->do_full, 128); mbar_init(&sm->do_empty, 1);
    mbar_init(&sm->s_full, 1); mbar_init(&sm->p_ready, 256);
    mbar_init(&sm->dp_full, 1); mbar_init(&sm->ds_ready, 256);
    mbar_init(&sm->dq_full, 1); mbar_init(&sm->dq_free, 256);
    mbar_init(&sm->acc_done, 1); mbar_init(&sm->acc_free, 256);
    mbar_init(&sm->drain, 1);
    if constexpr (DENSE) { mbar_init(&sm->turn_ok, 1); mbar_init(&sm->rows_out, 256); mbar_init(&sm->rows_seen, 1); }
    sm->abort_flag = 0;
    if constexpr (DENSE) sm->ticket = atomicAdd(p.turns + (long long)(MULTI ? p.parts : 1) * p.BH * ((p.S + QU - 1) / QU), 1);
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

  const int parts = MULTI ? p.parts : 1;
  const int tiles = ((DENSE ? p.S : p.sb) + BN - 1) / BN;
  const int n_items = p.BH * (DENSE ? 1 : p.Nb) * tiles;
  // dense: as many CTAs as items, one each
  auto first_item = [&]() { return DENSE ? sm->ticket : (int)blockIdx.x; };
  auto next_item = [&](int item) { return DENSE ? n_items : item + (int)gridDim.x; };

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    if (warp == 0) {
      // ---------------------------------------------------------------- TMA: K and V tiles, one pair per item
      if (lane == 0) {
        uint32_t n = 0;
        bool v_ahead = false;      // (nothing is loaded after a time-out)
        for (int item = first_item(); item < n_items; item = next_item(item)) {
          const KvItem it = kv_decode<DENSE>(p, item, tiles);
          if (it.n_units == 0) continue;
          const int y = it.head_off + it.key0;
          // V is free after the item's last dP^T, K only after its last dQ^T
          if (n >= 1 && !twait(0, &sm->v_empty, (n - 1) & 1)) break;
          mbar_expect_tx(&sm->v_full, TILE);
          tma_load_2d(sV, &tmV, &sm->v_full, 0, y);
          tma_load_2d(sV + PANEL, &tmV, &sm->v_full, 64, y);
          if (n >= 1 && !twait(0, &sm->k_empty, (n - 1) & 1)) { v_ahead = true; break; }
          mbar_expect_tx(&sm->k_full, TILE);
          tma_load_2d(sK, &tmK, &sm->k_full, 0, y);
          tma_load_2d(sK + PANEL, &tmK, &sm->k_full, 64, y);
          ++n;
          // the one K / V pair is reloaded when the item is over: ask the L2 for the next item's tiles now
          if (item + (int)gridDim.x < n_items) {
            const KvItem nx = kv_decode<DENSE>(p, item + gridDim.x, tiles);
            const int yn = nx.head_off + nx.key0;
            if (nx.n_units > 0) {
              tma_prefetch_2d(&tmK, 0, yn); tma_prefetch_2d(&tmK, 64, yn);
              tma_prefetch_2d(&tmV, 0, yn); tma_prefetch_2d(&tmV, 64, yn);
            }
          }
        }
        // drain: every issued load must have landed before the CTA may exit (only matters after a timeout)
        if (*abort_flag && n > 0) {
          mbar_wait(&sm->k_full, (n - 1) & 1, abort_flag, p.status);
          mbar_wait(&sm->v_full, (n - (v_ahead ? 0 : 1)) & 1, abort_flag, p.status);
        }
        tflush(0, 1);      // [0] k_empty + v_empty, [1] total
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------------- MMA issuer: the whole warp walks the loop, one
      // elected lane issues (warp-uniform control flow; see elect_one).
      //
      // The compute warps alternate between the two element-wise steps, the tensor pipe must have work during both.
      // Order per unit i, with what overlaps it:
      //   dK(i), dQ^T(i)            | P^T(i+1) from S^T(i+1), which was issued one unit early; dQ^T(i) read out
      //   dP^T(i+1)                 | rest of P^T(i+1)
      //   dV(i+1), S^T(i+2)         | dS^T(i+1)
      const bool leader = elect_one();
      auto wwait = [&](int site, uint64_t* bar, uint32_t parity) { twait(site, bar, parity); __syncwarp(); };
      uint32_t n = 0, g = 0;      // items and units done so far
      uint32_t s_slot = 0, s_par = 0, k_slot = 0;      // Q ring: next unit's slot and parity for S^T, slot of the current dK
      const uint32_t kK = lo_k(smem_u32(sK)), kV = lo_k(smem_u32(sV)), mK = lo_mn(smem_u32(sK)), mS = lo_mn(smem_u32(sDS));
      const uint32_t kQ = lo_k(smem_u32(sQ)), kO = lo_k(smem_u32(sO)), mQ = lo_mn(smem_u32(sQ)), mO = lo_mn(smem_u32(sO));
      constexpr uint32_t STAGE = TILE >> 4;
      for (int item = first_item(); item < n_items; item = next_item(item)) {
        const KvItem it = kv_decode<DENSE>(p, item, tiles);
        // the list bounds come from memory: a warp reduction marks them as warp-uniform
        const int n_list = __reduce_max_sync(0xffffffffu, it.n_list);
        const int n_units = (n_list + QU - 1) / QU;
        if (n_units == 0) continue;
        const int key_steps = (it.valid + 15) >> 4;
        auto rows16 = [&](int i) { return (min(QU, n_list - i * QU) + 15) >> 4; };   // 16-query steps of a unit
        auto issue_s = [&](int i) {
          wwait(1, &sm->q_full[s_slot], s_par);
          tc_fence_after();
          const uint32_t idesc = make_idesc_bf16(128, 16 * rows16(i), false, false);
          const uint32_t b = kQ + s_slot * STAGE;
          if (++s_slot == NQ) { s_slot = 0; s_par ^= 1; }
#pragma unroll
          for (int ks = 0; ks < DH / 16; ++ks)
            if (leader) mma_ss_lo(tmem + ST_COL, kK + koff(ks), b + koff(ks), idesc, ks > 0 ? 1u : 0u);
          if (leader) mma_commit(&sm->s_full);
        };
        auto issue_dp = [&](int i) {
          const uint32_t u = g + i;
          wwait(1, &sm->do_full, u & 1);
          if (u >= 1) wwait(3, &sm->dq_free, (u - 1) & 1);          // the columns held dQ^T of the unit before
          tc_fence_after();
          const uint32_t idesc = make_idesc_bf16(128, 16 * rows16(i), false, false);
#pragma unroll
          for (int ks = 0; ks < DH / 16; ++ks)
            if (leader) mma_ss_lo(tmem + DPT_COL, kV + koff(ks), kO + koff(ks), idesc, ks > 0 ? 1u : 0u);
          if (leader) mma_commit(&sm->dp_full);
          if (leader && i == n_units - 1) mma_commit(&sm->v_empty);
        };
        auto issue_dv = [&](int i) {
          const uint32_t u = g + i;
          wwait(2, &sm->p_ready, u & 1);
          // dV / dK still hold the previous item until its epilogue has read them
          if (i == 0 && n > 0) wwait(3, &sm->acc_free, (n - 1) & 1);
          tc_fence_after();
          const int ksteps = rows16(i);
#pragma unroll
          for (int ks = 0; ks < 8; ++ks)       // P^T of queries 64 h .. sits in columns 64 h .. 64 h + 31
            if (leader && ks < ksteps)
              mma_ts_lo(tmem + DV_COL, tmem + ST_COL + (ks >> 2) * 64 + (ks & 3) * 8, mO + mnoff(ks), IDESC_TN, (ks > 0 || i > 0) ? 1u : 0u);
          if (leader) mma_commit(&sm->do_empty);
        };
        wwait(0, &sm->k_full, n & 1);
        issue_s(0);
        wwait(0, &sm->v_full, n & 1);
        issue_dp(0);
        issue_dv(0);
        if (n_units > 1) issue_s(1);
        for (int i = 0; i < n_units; ++i) {
          const uint32_t u = g + i;
          wwait(2, &sm->ds_ready, u & 1);
          tc_fence_after();
          {
            const int ksteps = rows16(i);
            const uint32_t b = mQ + k_slot * STAGE;
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              if (leader && ks < ksteps)
                mma_ts_lo(tmem + DK_COL, tmem + DPT_COL + (ks >> 2) * 64 + (ks & 3) * 8, b + mnoff(ks), IDESC_TN, (ks > 0 || i > 0) ? 1u : 0u);
            if (leader) mma_commit(&sm->q_empty[k_slot]);
            if (++k_slot == NQ) k_slot = 0;
            // dQ^T over dP^T and dS^T: in order behind the dK MMAs that read dS^T there
            const uint32_t idesc = make_idesc_bf16(128, 16 * ksteps, true, true);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)
              if (leader && ks < key_steps) mma_ss_lo(tmem + DPT_COL, mK + mnoff(ks), mS + mnoff(ks), idesc, ks > 0 ? 1u : 0u);
            if (leader) mma_commit(&sm->dq_full);
          }
          if (i + 1 < n_units) {
            issue_dp(i + 1);
            issue_dv(i + 1);
            if (i + 2 < n_units) issue_s(i + 2);
          }
        }
        if (leader) mma_commit(&sm->k_empty);
        if (leader) mma_commit(&sm->acc_done);
        g += n_units;
        ++n;
      }
      if (leader && *abort_flag) mma_drain(&sm->drain);
      if (leader) tflush(2, 4);      // [2] k_full + v_full, [3] q_full + do_full, [4] p_ready + ds_ready, [5] dq_free + acc_free, [6] total
    } else if (DENSE && lane == 0) {
      // ---------------------------------------------------------------- turns: warp 3 waits for them, warp 2 passes them on.
      // Warp 3 lets the writers go on only when warp 2 has noted the end of the unit before: no barrier gets a phase ahead.
      const KvItem it = kv_decode<DENSE>(p, first_item(), tiles);
      const int rank = it.tile / parts;
      int* turn = p.turns + ((long long)(it.tile - rank * parts) * p.BH + it.bh) * it.n_units;
      for (int i = 0; i < it.n_units; ++i) {
        if (warp == 3) {
          if (rank > 0) turn_wait(turn + i, rank, abort_flag, p.status);
          if (i > 0) mbar_wait(&sm->rows_seen, (i - 1) & 1, abort_flag, p.status);
          mbar_arrive(&sm->turn_ok);
        } else {
          mbar_wait(&sm->rows_out, i & 1, abort_flag, p.status);
          mbar_arrive(&sm->rows_seen);
          turn_pass(turn + i, rank + 1);
        }
      }
    }
  } else if (warp < 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    // ------------------------------------------------------------------ loaders: the Q rows of the units with their lse (warps
    // 4-7), the dO rows with -rowsum(dO * O) (warps 8-11); they run ahead.
    // Sparse: the rows go from global to shared memory as asynchronous 16-byte copies, eight threads per 128-byte half
    // row; a thread keeps the list entries of its eight rows and fetches those of the next unit while the copies are in
    // flight.  Next to a busy tensor pipe a warp gets shared-memory and load instructions through at about one in 100
    // cycles, hence four warps for each tensor (six for both: the kernel waited for rows) and no shuffles.
    // Dense: consecutive rows, TMA tiles requested by one of the threads that bring the scalars.
    const bool is_q = warp < 8;
    const int lt = threadIdx.x & 127, r0 = 4 * (warp & 3) + (lane >> 3), chunk = lane & 7;      // rows r0 + 16 k
    UnitWalk<DENSE> walk(first_item(), n_items, tiles);
    const bool raster = !is_q && p.do_map.perm != nullptr;
    const long long stride = raster ? p.do_map.st : (long long)DH;
    const uint32_t tile0 = smem_u32(is_q ? sQ : sO);
    const __nv_bfloat16* src = nullptr;
    int idx[8];
    float sc = 0.f;
    auto fetch = [&]() {
      if constexpr (!DENSE) {
        const int b_ = walk.it.bh / p.do_map.heads, hd_ = walk.it.bh - b_ * p.do_map.heads;
        src = (is_q ? p.q : p.d_o) + (raster ? b_ * p.do_map.sb + hd_ * p.do_map.sh : (long long)walk.it.head_off * DH) + chunk * 8;
#pragma unroll
        for (int k = 0; k < 8; ++k) idx[k] = walk.entry(p, r0 + 16 * k);
        if (raster) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (idx[k] >= 0) idx[k] = __ldg(p.do_map.perm + idx[k]);
        }
      }
      const int mine = walk.entry(p, lt);
      sc = is_q ? INFINITY : 0.f;                          // padded queries: P = exp2(-inf) = 0
      if (mine >= 0) sc = is_q ? __ldg(p.lse + walk.it.head_off + mine) * LOG2E : -__ldg(p.Dv + walk.it.head_off + mine);
    };
    bool more = walk.next(p);
    if (more) fetch();
    uint32_t slot = 0, par = 1;
    for (uint32_t g = 0; more; ++g) {
      uint64_t* full = is_q ? &sm->q_full[slot] : &sm->do_full;
      // (the first waits pass at once: the parity of the phase before the first)
      twait(0, is_q ? &sm->q_empty[slot] : &sm->do_empty, par);
      // -rowsum(dO * O) of unit g goes to slot g % 2, which dS^T of unit g - 2 has left behind when dV of unit g - 1, which
      // follows P^T of unit g - 1, has freed the dO tile
      (is_q ? sm->lse2[slot] : sm->negD[g & 1])[lt] = sc;
      if constexpr (DENSE) {
        if (lt == 0) {
          const CUtensorMap* map = is_q ? &tmQ : &tmO;
          uint8_t* tile = is_q ? sQ + slot * TILE : sO;
          mbar_expect_tx(full, TILE);
          tma_load_3d(tile, map, full, 0, walk.first, walk.it.bh);
          tma_load_3d(tile + PANEL, map, full, 64, walk.first, walk.it.bh);
        } else {
          mbar_arrive(full);
        }
        more = walk.next(p);
        if (more) fetch();
        // drain: every issued load must have landed before the CTA may exit (only matters after a timeout)
        if (lt == 0 && *abort_flag) mbar_wait(full, par ^ 1, abort_flag, p.status);
      } else {
        const uint32_t dst = tile0 + slot * TILE + r0 * 128 + ((chunk ^ (r0 & 7)) << 4);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const __nv_bfloat16* row = src + (long long)max(idx[k], 0) * stride;
          const uint32_t bytes = idx[k] < 0 ? 0u : 16u;
          cp_async16(dst + k * 2048, row, bytes);
          cp_async16(dst + k * 2048 + PANEL, row + 64, bytes);
        }
        cp_async_commit();
        more = walk.next(p);
        if (more) fetch();
        cp_async_wait<0>();
        fence_async_proxy();
        mbar_arrive(full);
      }
      if (!is_q) par ^= 1;
      else if (++slot == NQ) { slot = 0; par ^= 1; }
    }
    if (lt == 0 && is_q) tflush(7, 1);     // [7] q_empty, [8] total
  } else if (warp >= 20) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 80;");
    // ------------------------------------------------------------------ dQ writers
    // Read dQ^T of a unit out of TMEM (lane = head-dim index, 128 query columns; two warps per TMEM lane quarter, each
    // taking 64 columns) and add it into the fp32 accumulator.  In the 16x256b shape a thread's registers hold the head-dim
    // indices r, r + 8, r + 16, r + 24 (r = lane / 4) of its quarter for the same query, so that four of them are one
    // red.global.add.v4.f32 without any exchange between lanes: the accumulator keeps a quarter's 32 columns in the order
    // 4 r + a <-> r + 8 a, and cast_rows undoes it.  A warp instruction covers four complete 128-byte lines, one in each of
    // four accumulator rows.  (Measured per SM with all SMs busy: reductions that cover whole 128-byte lines reach 23
    // B/cycle however the lines are spread over rows; 16 bytes per lane in 32 different rows reach 12.5.  With the rows
    // lane = head-dim index and shuffles between four lanes instead, the writers' own instructions were the slowest
    // part of a unit.)
    const int quad = warp & 3;
    const int qhalf = (warp - 20) >> 2;
    const uint32_t dq_tmem = tmem + ((uint32_t)(quad * 32) << 16) + DPT_COL + 64 * qhalf;
    float* acc_col = p.dq_acc + quad * 32 + (lane & ~3);
    uint32_t g = 0;
    for (int item = first_item(); item < n_items; item = next_item(item)) {
      const KvItem it = kv_decode<DENSE>(p, item, tiles);
      float* acc_head = acc_col + (long long)it.head_off * DH;
      if constexpr (MULTI) acc_head += (long long)(it.tile % parts) * p.BH * p.S * DH;
      for (int i = 0; i < it.n_units; ++i, ++g) {
        const int first = i * QU + 64 * qhalf;
        // accumulator rows of queries lane and 32 + lane of this half of the unit (-1 beyond the list)
        int row_lane[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int at = first + 32 * h + lane;
          row_lane[h] = at >= it.n_list ? -1 : DENSE ? at : checked_index(__ldg(p.q_idx + it.list_lo + at), p.S, p.status);
        }
        twait(0, &sm->dq_full, g & 1);
        tc_fence_after();
        // everything out of TMEM first: the next dP^T waits for these columns
        uint32_t x[2][32];
        tmem_ld_16x256_x8(dq_tmem, x[0]);
        tmem_ld_16x256_x8(dq_tmem + ROW16, x[1]);
        tmem_ld_wait();
        tc_fence_before();
        mbar_arrive(&sm->dq_free);
        // A reduction holds its source registers until the load/store unit has taken them, so each has its own four.
        auto write_rows = [&](auto put) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {        // query 8 j + 2 (lane % 4) + e of this half
              const int rw = __shfl_sync(0xffffffffu, row_lane[j >> 2], (8 * j + 2 * (lane & 3) + e) & 31);
              if (rw >= 0)
                put(acc_head + (long long)rw * DH, __uint_as_float(x[0][4 * j + e]) * p.scale, __uint_as_float(x[0][4 * j + 2 + e]) * p.scale,
                    __uint_as_float(x[1][4 * j + e]) * p.scale, __uint_as_float(x[1][4 * j + 2 + e]) * p.scale);
            }
        };
        auto add = [](float* to, float a, float b, float c, float d) { red_add_v4(to, a, b, c, d); };
        if constexpr (DENSE) {
          twait(1, &sm->turn_ok, g & 1);
          if (it.tile < parts)
            write_rows([](float* to, float a, float b, float c, float d) { *reinterpret_cast<float4*>(to) = make_float4(a, b, c, d); });
          else
            write_rows(add);
          mbar_arrive(&sm->rows_out);
        } else {
          write_rows(add);
        }
      }
    }
    if (warp == 20 && lane == 0) tflush(14, 1);     // [14] dq_full, [15] total
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    // ------------------------------------------------------------------ compute: warp = 32 keys x half of the unit's queries
    const int quad = warp & 3;
    const int half = (warp - 12) >> 2;
    const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
    const uint32_t st_t = tmem + lane_addr + ST_COL + 64 * half, dp_t = tmem + lane_addr + DPT_COL + 64 * half;
    // this lane's row address for stmatrix: matrices (keys 0-7, queries 8j), (keys 8-15, same), (keys 0-7, 8j + 8), ...
    const int mrow = quad * 32 + 8 * ((lane >> 3) & 1) + (lane & 7), mj = lane >> 4;
    const uint32_t ds_row = smem_u32(sDS) + half * PANEL + mrow * 128;
    uint32_t n = 0, g = 0, slot = 0, par = 0;        // items and units done; slot and parity of the Q ring
    for (int item = first_item(); item < n_items; item = next_item(item)) {
      const KvItem it = kv_decode<DENSE>(p, item, tiles);
      if (it.n_units == 0) {
        // no query selected this block: its keys get zero gradients
        const int r = quad * 32 + lane;
        if (r < it.valid) {
          const long long row_off = p.out_map.off((long long)it.head_off + it.key0 + r, DH);
          const uint4 z = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            reinterpret_cast<uint4*>(p.dk + row_off)[half * 8 + i] = z;
            reinterpret_cast<uint4*>(p.dv + row_off)[half * 8 + i] = z;
          }
        }
        continue;
      }
      // rows beyond the key range hold other blocks' keys and must not contribute to dQ
      const int key = quad * 32 + (lane >> 2);
      for (int i = 0; i < it.n_units; ++i, ++g) {
        const float2* lse2 = reinterpret_cast<const float2*>(sm->lse2[slot] + 64 * half) + (lane & 3);
        const float2* negD = reinterpret_cast<const float2*>(sm->negD[g & 1] + 64 * half) + (lane & 3);
        twait(0, &sm->q_full[slot], par);              // publishes lse2 of this unit
        if (++slot == NQ) { slot = 0; par ^= 1; }
        float2 l[8];                                   // (fetched before the wait: next to a busy tensor pipe a load takes its time)
#pragma unroll
        for (int j = 0; j < 8; ++j) l[j] = lse2[4 * j];
        twait(1, &sm->s_full, g & 1);
        tc_fence_after();
        // ---- P^T: thread holds keys key + 8 r (r = 0 .. 3) x queries 8 j + 2 (lane % 4) + {0, 1} of the half
        uint32_t pv[2][32];
        tmem_ld_16x256_x8(st_t, pv[0]);
        tmem_ld_16x256_x8(st_t + ROW16, pv[1]);
        tmem_ld_wait();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t pk[2][8];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            const int j = 4 * c + jj;
#pragma unroll
            for (int rh = 0; rh < 2; ++rh)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                float x0, x1;
                fma2(x0, x1, __uint_as_float(pv[rh][4 * j + 2 * e]), __uint_as_float(pv[rh][4 * j + 2 * e + 1]), p.scale_log2,
                     p.scale_log2, -l[j].x, -l[j].y);
                x0 = ex2(x0);
                x1 = ex2(x1);
                pv[rh][4 * j + 2 * e] = __float_as_uint(x0);
                pv[rh][4 * j + 2 * e + 1] = __float_as_uint(x1);
                pk[rh][2 * jj + e] = pack_bf16(x0, x1);
              }
          }
          tmem_st_16x128_x4(st_t + 16 * c, pk[0]);
          tmem_st_16x128_x4(st_t + ROW16 + 16 * c, pk[1]);
        }
        // negD of this unit (dV needs the dO rows anyway; asked before dV can run, so that the barrier cannot be a phase ahead)
        twait(0, &sm->do_full, g & 1);
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(&sm->p_ready);
        // ---- dS^T = P^T (dP^T - D).  The dS^T tile in shared memory is free: dP^T was issued behind the dQ^T that read it.
        float2 d[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) d[j] = negD[4 * j];
        twait(2, &sm->dp_full, g & 1);
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          uint32_t dp[2][16];
          tmem_ld_16x256_x4(dp_t + 32 * c, dp[0]);
          tmem_ld_16x256_x4(dp_t + ROW16 + 32 * c, dp[1]);
          tmem_ld_wait();
#pragma unroll
          for (int rh = 0; rh < 2; ++rh) {
            uint32_t dk_[8];
#pragma unroll
            for (int jj = 0; jj < 4; ++jj) {
              const int j = 4 * c + jj;
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                float x0, x1;
                add2(x0, x1, __uint_as_float(dp[rh][4 * jj + 2 * e]), __uint_as_float(dp[rh][4 * jj + 2 * e + 1]), d[j].x, d[j].y);
                mul2(x0, x1, x0, x1, __uint_as_float(pv[rh][4 * j + 2 * e]), __uint_as_float(pv[rh][4 * j + 2 * e + 1]));
                dk_[2 * jj + e] = key + 16 * rh + 8 * e < it.valid ? pack_bf16(x0, x1) : 0u;
              }
            }
            tmem_st_16x128_x4(dp_t + rh * ROW16 + 16 * c, dk_);
#pragma unroll
            for (int m = 0; m < 2; ++m)
              stmatrix_x4(ds_row + rh * 16 * 128 + (((4 * c + 2 * m + mj) ^ (lane & 7)) << 4), dk_[4 * m], dk_[4 * m + 1], dk_[4 * m + 2],
                          dk_[4 * m + 3]);
          }
        }
        fence_async_proxy();
        tmem_st_wait();
        tc_fence_before();
        mbar_arrive(&sm->ds_ready);
      }
      // ---- epilogue: thread = key row; each half writes 64 of its 128 dV / dK columns
      twait(3, &sm->acc_done, n & 1);
      tc_fence_after();
      const int r = quad * 32 + lane;
      const long long row_off = r < it.valid ? p.out_map.off((long long)it.head_off + it.key0 + r, DH) : 0;
#pragma unroll 1
      for (int pass = 0; pass < 4; ++pass) {      // dV columns, then dK columns, 32 at a time
        const int cgrp = half * 2 + (pass & 1);
        const bool is_dk = pass >= 2;
        uint32_t a[32];
        tmem_ld32(tmem + lane_addr + (is_dk ? DK_COL : DV_COL) + cgrp * 32, a);
        tmem_ld_wait();
        if (pass == 3) {
          tc_fence_before();
          mbar_arrive(&sm->acc_free);
        }
        if (r < it.valid) {
          const float mul = is_dk ? p.scale : 1.0f;
          __nv_bfloat16* row = (is_dk ? p.dk : p.dv) + row_off + cgrp * 32;
#pragma unroll
          for (int i = 0; i < 32; i += 16) {      // sixteen bf16 = one 32-byte store (two 16-byte stores if unaligned)
            uint32_t hv[8];
#pragma unroll
            for (int k = 0; k < 8; ++k)
              hv[k] = pack_bf16(__uint_as_float(a[i + 2 * k]) * mul, __uint_as_float(a[i + 2 * k + 1]) * mul);
            if (p.dkv_32) {
              st_global_v8(row + i, hv[0], hv[1], hv[2], hv[3], hv[4], hv[5], hv[6], hv[7]);
            } else {
              *reinterpret_cast<uint4*>(row + i) = make_uint4(hv[0], hv[1], hv[2], hv[3]);
              *reinterpret_cast<uint4*>(row + i + 8) = make_uint4(hv[4], hv[5], hv[6], hv[7]);
            }
          }
        }
      }
      ++n;
    }
    if (threadIdx.x == 384) tflush(9, 4);   // [9] q_full, [10] s_full, [11] dp_full, [12] acc_done, [13] total
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, TMEM_COLS);
}

template <bool DENSE, bool MULTI>
static int launch(const Dims& D, const void* k, const void* v, KvParams& kp, cudaStream_t st) {
  CUtensorMap tmK, tmV, tmQ, tmO;
  const uint64_t rows = (uint64_t)D.BH * D.S;
  if (!sm100::make_tmap_bf16_rows(&tmK, k, rows, DH, BN) || !sm100::make_tmap_bf16_rows(&tmV, v, rows, DH, BN))
    return VMOBA_ERR_CUDA;
  // dense: units of consecutive rows (rows beyond a head's S read as zeros); sparse: not used
  if (!sm100::make_tmap_bf16_heads(&tmQ, kp.q, D.BH, D.S, DH, QU) || !sm100::make_tmap_bf16_heads(&tmO, kp.d_o, D.BH, D.S, DH, QU))
    return VMOBA_ERR_CUDA;
  kp.S = D.S; kp.Nb = DENSE ? 1 : D.Nb; kp.sb = DENSE ? D.S : D.sb; kp.BH = D.BH;
  kp.scale = D.scale; kp.scale_log2 = D.scale * LOG2E;
  kp.prof = g_wait_profile;
  kp.dkv_32 = (reinterpret_cast<uintptr_t>(kp.dk) % 32) == 0 && (reinterpret_cast<uintptr_t>(kp.dv) % 32) == 0 &&
              (!kp.out_map.perm || (kp.out_map.sb % 16 == 0 && kp.out_map.st % 16 == 0 && kp.out_map.sh % 16 == 0));
  const long long items = (long long)D.BH * kp.Nb * ((kp.sb + BN - 1) / BN);
  if (items > (long long)INT32_MAX - 4096) return VMOBA_ERR_SHAPE;
  const int grid = DENSE ? (int)items : (int)std::max<long long>(1, std::min<long long>(items, sm_count()));
  auto kernel = kp.prof ? attn_bwd_fused_kernel<DENSE, MULTI, true> : attn_bwd_fused_kernel<DENSE, MULTI, false>;
  VMOBA_CUDA_OK(allow_smem(kernel, (int)SMEM_BYTES));
  launch_kernel(early_rows(D), kernel, grid, THREADS, SMEM_BYTES, st, tmK, tmV, tmQ, tmO, kp);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

}  // namespace tcb

// Backward over the work lists (bf16, head_dim 128).  Dv holds rowsum(dO * O) per query; dq_acc is
// an fp32 accumulator whose rows of selecting queries are zero; the caller converts it to bf16 (simt::cast_rows_kernel
// knows the order of its columns).
int tc_sparse_bwd(const Dims& D, const void* q, const void* k, const void* v, const void* d_o, const float* lse,
                  const float* Dv, const int* kb_ptr, const int* q_idx, long long cap, float* dq_acc, void* dk, void* dv,
                  int32_t* status, cudaStream_t st, const RowMap& out_map, const RowMap& do_map) {
  tcb::KvParams kp;
  kp.q = (const __nv_bfloat16*)q; kp.d_o = (const __nv_bfloat16*)d_o; kp.lse = lse; kp.Dv = Dv;
  kp.kb_ptr = kb_ptr; kp.q_idx = q_idx; kp.capacity = cap;
  kp.dk = (__nv_bfloat16*)dk; kp.dv = (__nv_bfloat16*)dv; kp.status = status;
  kp.dq_acc = dq_acc; kp.out_map = out_map; kp.do_map = do_map;
  kp.turns = nullptr; kp.group = 1; kp.parts = 1;
  return tcb::launch<false, false>(D, k, v, kp, st);
}

// Dense backward: every query of a head meets every key tile; turns holds tc_dense_bwd_turns() zeros, dq_acc anything.
int tc_dense_bwd_parts(const Dims& D) {
  const long long acc = (long long)D.BH * D.S * D.d * (long long)sizeof(float), tiles = (D.S + tcb::BN - 1) / tcb::BN;
  return (int)std::max<long long>(1, std::min<long long>(std::min<long long>(4, tiles), (128ll << 20) / acc));
}
long long tc_dense_bwd_turns(const Dims& D) {
  return (long long)tc_dense_bwd_parts(D) * D.BH * ((D.S + tcb::QU - 1) / tcb::QU) + 1;
}
int tc_dense_bwd(const Dims& D, const void* q, const void* k, const void* v, const void* d_o, const float* lse,
                 const float* Dv, float* dq_acc, int* turns, void* dk, void* dv, int32_t* status, cudaStream_t st) {
  tcb::KvParams kp;
  kp.q = (const __nv_bfloat16*)q; kp.d_o = (const __nv_bfloat16*)d_o; kp.lse = lse; kp.Dv = Dv;
  kp.kb_ptr = nullptr; kp.q_idx = nullptr; kp.capacity = 0;
  kp.dk = (__nv_bfloat16*)dk; kp.dv = (__nv_bfloat16*)dv; kp.status = status;
  kp.dq_acc = dq_acc; kp.turns = turns; kp.parts = tc_dense_bwd_parts(D);
  // Sixteen heads: their accumulators, Q and dO pass through the L2 once per SMs / 16 key tiles.  More where a head has so few
  // units that its tiles would come too slowly for the SMs.
  const int units = (D.S + tcb::QU - 1) / tcb::QU;
  kp.group = std::min(D.BH, std::max(16, sm_count() / units));
  return kp.parts > 1 ? tcb::launch<true, true>(D, k, v, kp, st) : tcb::launch<true, false>(D, k, v, kp, st);
}

// Registers (or clears, with null) a device buffer of 16 uint64 counters for the attention kernels'
// wait-time diagnostics.  Not part of the method; see the kernels for the counter layout.
unsigned long long* debug_wait_profile() { return tcb::g_wait_profile; }
}  // namespace vmoba

extern "C" void vmoba_debug_wait_profile(void* dev_counters16) {
  vmoba::tcb::g_wait_profile = static_cast<unsigned long long*>(dev_counters16);
}
