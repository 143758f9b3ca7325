// fp32 CUDA-core attention kernels: Step 3 of VMoBA (attention of each query over the keys
// of its selected blocks), its backward, and the dense tau = 1 limit.  These serve the fp32
// dtype (any supported head_dim) and bf16 shapes without a tensor-core kernel; all arithmetic
// is fp32.
//
// Work decomposition follows the key-block CSR: a work item is (batch, head, key block j,
// a chunk of <= 64 queries that selected j).  A query that selected several blocks gets one
// partial (o, lse) per block, merged afterwards; queries with a single block are written
// directly, queries with none are zero-filled by the merge kernel.
#pragma once

#include <algorithm>

#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include "common.cuh"

namespace vmoba {
namespace simt {

constexpr int kRows = 64;      // rows (queries, or keys in the dK/dV kernel) per CTA, and of a tile of the streamed operand
constexpr int kThreads = 256;  // 16 x 16: a thread owns a 4 x 4 piece of a 64 x 64 product, 4 rows x DH / 16 columns of a result

// item_desc[item] = {index of the (batch, head, key block) list, first list position, rows (<= rows_per_item), 0}; a warp
// per list (a thread per list took 13 us for 240 lists of 77 items, bound by the latency of its loop).
__device__ __forceinline__ void write_item_desc(const int* item_ptr, const int* __restrict__ kb_ptr, long long n_kb,
                                                long long max_items, long long capacity, int rows_per_item,
                                                int4* __restrict__ desc, long long warp, long long n_warps) {
  const int lane = threadIdx.x & 31;
  for (long long i = warp; i < n_kb; i += n_warps) {
    const long long t0 = item_ptr[i], t1 = min((long long)item_ptr[i + 1], max_items);
    const long long lo = min((long long)kb_ptr[i], capacity), hi = min((long long)kb_ptr[i + 1], capacity);
    for (long long t = t0 + lane; t < t1; t += 32) {
      const long long l = lo + (t - t0) * rows_per_item;
      desc[t] = make_int4((int)i, (int)l, (int)min((long long)rows_per_item, hi - l), 0);
    }
  }
}

// chunk-count prefix over the (batch, head, key block) lists: item_ptr[i] = number of work
// items before list i when every list is cut into chunks of `rows` queries.
static __global__ void __launch_bounds__(1024)
item_ptr_kernel(const int* __restrict__ kb_ptr, long long n_kb, int rows, long long capacity,
                int* item_ptr, int4* desc, long long max_items) {
  if (!grid_begin()) return;
  __shared__ long long total;
  block_exclusive_scan(
      [&](long long i) {
        long long lo = min((long long)kb_ptr[i], capacity), hi = min((long long)kb_ptr[i + 1], capacity);
        return (hi - lo + rows - 1) / rows;
      },
      item_ptr, n_kb, &total);
  if (desc) write_item_desc(item_ptr, kb_ptr, n_kb, max_items, capacity, rows, desc, threadIdx.x >> 5, blockDim.x >> 5);
}

static __global__ void __launch_bounds__(256)
item_desc_kernel(const int* __restrict__ item_ptr, const int* __restrict__ kb_ptr, long long n_kb, long long max_items,
                 long long capacity, int rows_per_item, int4* __restrict__ desc) {
  if (!grid_begin()) return;
  write_item_desc(item_ptr, kb_ptr, n_kb, max_items, capacity, rows_per_item, desc,
                  (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), (long long)gridDim.x * (blockDim.x >> 5));
}

// Offsets of the lists' items and the items' records.  One CTA does both where the lists are one trip of its scan and the
// items few (a launch less: forward and backward of 1.9K tokens 122.7 -> 119.6 us); else the records are spread over the chip.
static void make_items(const int* kb_ptr, long long n_kb, int rows, long long cap, long long max_items, int* item_ptr,
                       int4* desc, cudaStream_t st) {
  const bool one = n_kb <= 1024 && max_items <= 4096;
  launch_kernel(item_ptr_kernel, 1, 1024, 0, st, kb_ptr, n_kb, rows, cap, item_ptr, one ? desc : nullptr, max_items);
  if (!one)
    launch_kernel(item_desc_kernel, (int)std::min<long long>((n_kb + 7) / 8, sm_count() * 8), 256, 0, st, item_ptr, kb_ptr,
                  n_kb, max_items, cap, rows, desc);
  count_launches(one ? 1 : 2);
}

struct Item {
  int bh;          // batch * heads + head
  int key_begin;   // key range inside the head (block-major positions)
  int key_end;
  int list_lo;     // sparse: range of CSR positions handled by this item
  int list_hi;
};

// Sparse item decode: binary search of the chunk prefix.
__device__ __forceinline__ Item decode_sparse(int item, const int* __restrict__ item_ptr, int n_kb,
                                              const int* __restrict__ kb_ptr, int Nb, int sb, int rows,
                                              long long capacity) {
  int lo = 0, hi = n_kb;   // find the last i with item_ptr[i] <= item
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (item_ptr[mid] <= item) lo = mid; else hi = mid;
  }
  Item it;
  it.bh = lo / Nb;
  int j = lo - it.bh * Nb;
  it.key_begin = j * sb;
  it.key_end = it.key_begin + sb;
  int chunk = item - item_ptr[lo];
  long long end = min((long long)kb_ptr[lo + 1], capacity);
  it.list_lo = kb_ptr[lo] + chunk * rows;
  it.list_hi = (int)min((long long)it.list_lo + rows, end);
  return it;
}

// Tiles in shared memory: 64 rows of DH (or 64) floats, four more to a row, so that sixteen consecutive rows' float4 lie in
// different banks.
//
// A 64 x 64 product takes a thread 64 FMAs per eight 16-byte loads from shared memory.  With four threads to a row, each holding a
// quarter of its channels, a key cost a thread as many loads as four of its FMAs and two shuffles.  fp32 layer,
// forward and backward: 13 heads x 4,096 tokens in blocks of 512 keys 4570 -> 2256 us (head_dim 128), 2136 -> 1275 (64), 8 x 2,496 in
// blocks of 156 307 -> 197, 2 x 256 123 -> 77; dense, 4 x 2,000, head_dim 64, bf16, 1361 -> 829.  What bounds them now (13 x 4,096, blocks of 512 keys): the shared-memory pipe, 71 and 74 % busy in the forwards of head_dim 64
// and 128, and the latency that 16 warps per SM (8 in the backward of head_dim 128: registers) do not hide, 54 to 64 % of the issue
// slots taken; the FMA pipe is 40 to 45 % busy.  At the 128 registers of two CTAs per SM all kernels but the backward of
// head_dim 128 spill: 16 to 168 bytes of stack.  Dense calls of few tiles leave SMs idle (4 x 2,000: 128 tiles).
template <int DH> constexpr int kLd = DH + 4;
template <int DH> constexpr int kTileFloats = kRows * kLd<DH>;
constexpr int kLdP = kRows + 4;

// A tile's rows, in registers on their way from global to shared memory (rows beyond n_valid: zeros).
template <typename T, int DH>
struct TileRegs {
  static constexpr int V = DH / 4, N = kRows * V / kThreads;
  float4 x[N];
  template <typename RowOf>
  __device__ __forceinline__ void fetch(const T* __restrict__ head_base, int n_valid, RowOf row_of) {
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const int i = threadIdx.x + n * kThreads, r = i / V, c4 = i % V;
      x[n] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < n_valid) x[n] = load4(head_base + (long long)row_of(r) * DH + c4 * 4);
    }
  }
  __device__ __forceinline__ void store(float* dst) const {
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const int i = threadIdx.x + n * kThreads, r = i / V, c4 = i % V;
      *reinterpret_cast<float4*>(dst + r * kLd<DH> + c4 * 4) = x[n];
    }
  }
};

// acc[i][j] = A[4 ty + i] . B[tx + 16 j] for the first NJ * 16 rows of B, as (p0 + p1) + (p2 + p3) where pn sums the channels
// 16 g + 4 n to 16 g + 4 n + 3 of all g in their order.  These are the sums of the kernels with four threads to a row, and so is
// the order of every other sum here but that of dq: o, lse, dk and dv are theirs to the bit.  (Scores off by one rounding move
// single gradients by 1e-4 of their rms where the logits are large: 13 heads x 4,096 tokens with a smooth field in q and k, head_dim
// 128.  Sums of sixteen channels at a time are nearer to 64 bits by a quarter and as fast, but that far from what was.)
template <int DH, int NJ>
__device__ __forceinline__ void dot_quarter(const float* A, const float* B, int ty, int tx, int c0, float (&part)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) part[i][j] = 0.f;
#pragma unroll
  for (int c = 0; c < DH; c += 16) {
    float4 a[4], b[NJ];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = *reinterpret_cast<const float4*>(A + (4 * ty + i) * kLd<DH> + c0 + c);
#pragma unroll
    for (int j = 0; j < NJ; ++j) b[j] = *reinterpret_cast<const float4*>(B + (tx + 16 * j) * kLd<DH> + c0 + c);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        part[i][j] = fmaf(a[i].x, b[j].x, part[i][j]);
        part[i][j] = fmaf(a[i].y, b[j].y, part[i][j]);
        part[i][j] = fmaf(a[i].z, b[j].z, part[i][j]);
        part[i][j] = fmaf(a[i].w, b[j].w, part[i][j]);
      }
  }
}
template <int DH, int NJ>
__device__ __forceinline__ void dot_tiles_n(const float* A, const float* B, int ty, int tx, float (&acc)[4][4]) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    float x[4][4], y[4][4];
    dot_quarter<DH, NJ>(A, B, ty, tx, 8 * h, x);
    dot_quarter<DH, NJ>(A, B, ty, tx, 8 * h + 4, y);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[i][j] += y[i][j];
        acc[i][j] = h ? acc[i][j] + x[i][j] : x[i][j];
      }
  }
}
template <int DH>
__device__ __forceinline__ void dot_tiles(const float* A, const float* B, int ty, int tx, int n_b, float (&acc)[4][4]) {
  if (n_b > 32) dot_tiles_n<DH, 4>(A, B, ty, tx, acc);
  else dot_tiles_n<DH, 2>(A, B, ty, tx, acc);
}

__device__ __forceinline__ void fma4(float* acc, float w, const float4& x) {
  acc[0] = fmaf(w, x.x, acc[0]); acc[1] = fmaf(w, x.y, acc[1]); acc[2] = fmaf(w, x.z, acc[2]); acc[3] = fmaf(w, x.w, acc[3]);
}
// acc[i][4 g + c] += sum over the first n rows k of B: P[4 ty + i][k] * B[k][64 g + 4 tx + c]
template <int DH>
__device__ __forceinline__ void add_weighted(const float* P, const float* B, int ty, int tx, int n, float (&acc)[4][DH / 16]) {
#pragma unroll 1
  for (int k = 0; k < n; k += 4) {
    float4 w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const float4*>(P + (4 * ty + i) * kLdP + k);
#pragma unroll
    for (int g = 0; g < DH / 64; ++g) {
      float4 x[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) x[e] = *reinterpret_cast<const float4*>(B + (k + e) * kLd<DH> + 64 * g + 4 * tx);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fma4(&acc[i][4 * g], w[i].x, x[0]); fma4(&acc[i][4 * g], w[i].y, x[1]);
        fma4(&acc[i][4 * g], w[i].z, x[2]); fma4(&acc[i][4 * g], w[i].w, x[3]);
      }
    }
  }
}
// The same with P transposed: acc[i][..] += sum over k of P[k][4 ty + i] * B[k][..]
template <int DH>
__device__ __forceinline__ void add_weighted_t(const float* P, const float* B, int ty, int tx, int n, float (&acc)[4][DH / 16]) {
#pragma unroll 4
  for (int k = 0; k < n; ++k) {
    const float4 w = *reinterpret_cast<const float4*>(P + k * kLdP + 4 * ty);
#pragma unroll
    for (int g = 0; g < DH / 64; ++g) {
      const float4 x = *reinterpret_cast<const float4*>(B + k * kLd<DH> + 64 * g + 4 * tx);
      fma4(&acc[0][4 * g], w.x, x); fma4(&acc[1][4 * g], w.y, x); fma4(&acc[2][4 * g], w.z, x); fma4(&acc[3][4 * g], w.w, x);
    }
  }
}
// Thread tx of the sixteen that share rows: the largest x[tx / 4][tx % 4] of them all.
__device__ __forceinline__ float group_max(const float (&x)[4][4], int tx) {
  float r[16];
#pragma unroll
  for (int n = 0; n < 16; ++n) r[n] = x[n >> 2][n & 3];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int n = 0; n < o; ++n) {
      const float keep = (tx & o) ? r[n + o] : r[n], give = (tx & o) ? r[n] : r[n + o];
      r[n] = fmaxf(keep, __shfl_xor_sync(0xffffffffu, give, o));
    }
  return r[0];
}
template <int DH> constexpr int kFwdSmem = (2 * kTileFloats<DH> + kRows * kLdP) * 4;      // Q, K or V, weights

// ------------------------------------------------------------------------------ forward
template <typename T, int DH, bool DENSE>
__global__ void __launch_bounds__(kThreads, 2)
attn_fwd_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                const int* __restrict__ kb_ptr, const int* __restrict__ q_idx, const int* __restrict__ q_ptr,
                const int* __restrict__ item_ptr, int n_kb, int S, int Nb, int sb, int BH, float scale,
                T* __restrict__ o, T* __restrict__ o_resid, float* __restrict__ lse, float* __restrict__ part_o,
                float* __restrict__ part_lse, long long capacity) {
  if (!grid_begin()) return;
  extern __shared__ __align__(16) float simt_smem[];
  float* Qs = simt_smem;
  float* KVs = Qs + kTileFloats<DH>;
  float* Ps = KVs + kTileFloats<DH>;
  __shared__ int s_row[kRows];                 // in-head position of the query, -1 for none; bit 30: it has a single block
  __shared__ __align__(16) float s_max[kRows * 4], s_corr[kRows * 4];      // of a tile's rows, every sixteen keys
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  const int tiles_per_head = (S + kRows - 1) / kRows;
  const int n_items = DENSE ? BH * tiles_per_head : item_ptr[n_kb];
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    Item it;
    int rows;
    if (DENSE) {
      it.bh = item / tiles_per_head;
      it.list_lo = (item - it.bh * tiles_per_head) * kRows;
      it.key_begin = 0; it.key_end = S;
      rows = min(kRows, S - it.list_lo);
    } else {
      it = decode_sparse(item, item_ptr, n_kb, kb_ptr, Nb, sb, kRows, capacity);
      rows = it.list_hi - it.list_lo;
    }
    const long long head_off = (long long)it.bh * S;
    const T* kh = k + head_off * DH;
    const T* vh = v + head_off * DH;
    constexpr int kSingle = 1 << 30;
    __syncthreads();                           // (the item before is through with the shared memory)
    if (t < kRows) {
      int x = -1;
      if (t < rows) {
        x = DENSE ? it.list_lo + t : q_idx[it.list_lo + t];
        if (DENSE || q_ptr[head_off + x + 1] - q_ptr[head_off + x] == 1) x |= kSingle;
      }
      s_row[t] = x;
    }
    TileRegs<T, DH> next;
    next.fetch(kh, min(kRows, it.key_end - it.key_begin), [&](int i) { return it.key_begin + i; });
    __syncthreads();
    {
      TileRegs<T, DH> qt;
      qt.fetch(q + head_off * DH, rows, [&](int i) { return s_row[i] & (kSingle - 1); });
      qt.store(Qs);
    }
    next.store(KVs);
    float m = -INFINITY, l = 0.f;              // of row 4 ty + tx / 4
    float acc[4][DH / 16];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < DH / 16; ++c) acc[i][c] = 0.f;
    const bool live = (ty & ~1) * 4 < rows;    // (a warp has eight rows)
    __syncthreads();
    for (int t0 = it.key_begin; t0 < it.key_end; t0 += kRows) {
      const int nv = min(kRows, it.key_end - t0);
      next.fetch(vh, nv, [&](int i) { return t0 + i; });
      if (live) {
        float s[4][4];
        dot_tiles<DH>(Qs, KVs, ty, tx, nv, s);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) s[i][j] = tx + 16 * j < nv ? s[i][j] * scale : -INFINITY;
        // the largest score so far changes every sixteen keys: thread tx finds it for row tx / 4 at keys 16 (tx % 4) and on, and
        // what the sums so far are multiplied with there
        const float mx = group_max(s, tx);
        float mj = mx, up = __shfl_up_sync(0xffffffffu, mj, 1, 4);
        if ((tx & 3) >= 1) mj = fmaxf(mj, up);
        up = __shfl_up_sync(0xffffffffu, mj, 2, 4);
        if ((tx & 3) >= 2) mj = fmaxf(mj, up);
        mj = fmaxf(m, mj);
        up = __shfl_up_sync(0xffffffffu, mj, 1, 4);
        const float before = (tx & 3) ? up : m;
        s_max[ty * 16 + tx] = mj;
        s_corr[ty * 16 + tx] = before == -INFINITY ? 0.f : expf(before - mj);
        m = __shfl_sync(0xffffffffu, mj, 3, 4);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 m4 = *reinterpret_cast<const float4*>(s_max + 16 * ty + 4 * i);
          const float mm[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
          for (int j = 0; j < 4; ++j) Ps[(4 * ty + i) * kLdP + tx + 16 * j] = s[i][j] == -INFINITY ? 0.f : expf(s[i][j] - mm[j]);
        }
        __syncwarp();
        // the row's weights, key after key
        const float* row = Ps + (4 * ty + (tx >> 2)) * kLdP;
#pragma unroll 1
        for (int k = 0; k < nv; k += 16) {
          const float corr = s_corr[16 * ty + (tx & 12) + (k >> 4)];
#pragma unroll
          for (int c = 0; c < 16; c += 4) {
            const float4 w = *reinterpret_cast<const float4*>(row + k + c);
            l = c == 0 ? __fadd_rn(__fmul_rn(l, corr), w.x) : l + w.x;      // (not one fused operation: it was two)
            l += w.y; l += w.z; l += w.w;
          }
        }
      }
      __syncthreads();
      next.store(KVs);
      __syncthreads();
      const int t1 = t0 + kRows;
      if (t1 < it.key_end) next.fetch(kh, min(kRows, it.key_end - t1), [&](int i) { return t1 + i; });
      if (live) {
#pragma unroll 1
        for (int k = 0; k < nv; k += 16) {
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float corr = s_corr[16 * ty + 4 * i + (k >> 4)];
#pragma unroll
            for (int c = 0; c < DH / 16; ++c) acc[i][c] *= corr;
          }
          add_weighted<DH>(Ps + k, KVs + k * kLd<DH>, ty, tx, min(16, nv - k), acc);
        }
      }
      if (t1 < it.key_end) {
        __syncthreads();
        next.store(KVs);
        __syncthreads();
      }
    }
    if (!live) continue;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float total = __shfl_sync(0xffffffffu, l, 4 * i, 16), top = __shfl_sync(0xffffffffu, m, 4 * i, 16);
      const int x = s_row[4 * ty + i];
      if (x < 0) continue;
      const float inv = 1.0f / total, row_lse = top + logf(total);
      const long long G_ = head_off + (x & (kSingle - 1)), pos = (long long)it.list_lo + 4 * ty + i;
      const bool direct = (x & kSingle) != 0;
#pragma unroll
      for (int g = 0; g < DH / 64; ++g) {
        const int col = 64 * g + 4 * tx;
        const float4 r = make_float4(acc[i][4 * g] * inv, acc[i][4 * g + 1] * inv, acc[i][4 * g + 2] * inv, acc[i][4 * g + 3] * inv);
        if (direct) store4_resid(o + G_ * DH + col, o_resid ? o_resid + G_ * DH + col : nullptr, r);
        else store4(part_o + pos * DH + col, r);
      }
      if (tx == 0) { if (direct) lse[G_] = row_lse; else part_lse[pos] = row_lse; }
    }
  }
}

// Merge of the per-block partials of each query (one warp per query).  Queries with a single
// pair were written by the attention kernel; queries with none get o = 0, lse = -inf.
template <typename T, int DH, typename PT>
__global__ void __launch_bounds__(256)
merge_kernel(const int* __restrict__ q_ptr, const int* __restrict__ q_pairs, long long n_queries,
             const PT* __restrict__ part_o, const float* __restrict__ part_lse, long long capacity,
             T* __restrict__ o, T* __restrict__ o_resid, float* __restrict__ lse, const RowMap o_map) {
  if (!grid_begin()) return;
  constexpr int C = DH / 32;   // channels per lane
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long g = warp; g < n_queries; g += nwarps) {
    const long long lo = q_ptr[g], hi = min((long long)q_ptr[g + 1], capacity);
    const long long n = hi - lo;
    if (n == 1 && q_ptr[g + 1] - lo == 1) continue;
    float acc[C];
#pragma unroll
    for (int c = 0; c < C; ++c) acc[c] = 0.f;
    float out_lse = -INFINITY;
    if (n > 0) {
      // lane i of each group of 32 pairs fetches the position and lse of pair i once; the row
      // weights then travel by shuffle.  A truncated list (capacity exceeded) may hold unwritten
      // entries: keep every index in range.
      float mx = -INFINITY;
      for (long long i0 = lo; i0 < hi; i0 += 32) {
        const long long i = i0 + lane;
        const float l = i < hi ? part_lse[min(max(q_pairs[i], 0), (int)(capacity - 1))] : -INFINITY;
        mx = fmaxf(mx, l);
      }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
      float tot = 0.f;
      for (long long i0 = lo; i0 < hi; i0 += 32) {
        const long long i = i0 + lane;
        int my_pos = 0;
        float my_w = 0.f;
        if (i < hi) {
          my_pos = min(max(q_pairs[i], 0), (int)(capacity - 1));
          my_w = expf(part_lse[my_pos] - mx);
        }
        tot += my_w;
        const int m = (int)min((long long)32, hi - i0);
#pragma unroll 4
        for (int k = 0; k < m; ++k) {
          const long long pos = __shfl_sync(0xffffffffu, my_pos, k);
          const float wgt = __shfl_sync(0xffffffffu, my_w, k);
          if constexpr (C == 4 && sizeof(PT) == 4) {
            const float4 v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(part_o) + pos * DH + lane * 4);
            acc[0] = fmaf(wgt, v.x, acc[0]); acc[1] = fmaf(wgt, v.y, acc[1]);
            acc[2] = fmaf(wgt, v.z, acc[2]); acc[3] = fmaf(wgt, v.w, acc[3]);
          } else {
#pragma unroll
            for (int c = 0; c < C; ++c) acc[c] = fmaf(wgt, to_f32<PT>(part_o[pos * DH + lane * C + c]), acc[c]);
          }
        }
      }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, s);
      const float inv = 1.0f / tot;
#pragma unroll
      for (int c = 0; c < C; ++c) acc[c] *= inv;
      out_lse = mx + logf(tot);
    }
    // o goes to the caller's layout (block-major, or raster order through perm); the residual stays block-major
    T* o_row = o + o_map.off(g, DH);
    if constexpr (C == 4) {
      store4_resid(o_row + lane * 4, o_resid ? o_resid + g * DH + lane * 4 : nullptr,
                   make_float4(acc[0], acc[1], acc[2], acc[3]));
    } else {
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const T hi_ = from_f32<T>(acc[c]);
        o_row[lane * C + c] = hi_;
        if (o_resid) o_resid[g * DH + lane * C + c] = from_f32<T>(acc[c] - to_f32<T>(hi_));
      }
    }
    if (lane == 0) lse[g] = out_lse;
  }
}

// The same merge for the tensor-core path (head_dim 128).  A partial row is stored as fp16 values times a power of two
// (part_scale, one per row; the row's largest magnitude rounded up), which halves the bytes the forward writes and this
// pass reads; a value is then off by at most 2^-11 of its row's largest one.  The scale is folded into the row's merge
// weight.
//
// Bound by the latency of its loads: a query takes four that depend on one another (list bounds, pair positions, partial
// lse, rows).  A warp takes 32 consecutive queries at a time.  Queries of up to kInLane pairs: lane l works out the weights
// of query l on its own, then the warp walks the queries that need a row.  Longer ones: the weights are worked out by the
// half-warp that adds up the rows.  Either way two queries are walked at once, one per half-warp: sixteen lanes of 16 bytes
// fetch a row, and kBatch rows of each are in flight.  Nine pairs per query (907,200 queries, 2.3 GB) 536 us, 32 pairs
// (393,120 queries) 826, two to six pairs 62 to 207: with a warp per query at a time and eight bytes per lane 714, 962 and
// 72 to 255; 64 registers (four CTAs per SM) beat 80 by a tenth, kBatch = 4 loses a tenth.
//
// span (a power of two up to 32): queries a warp takes at a time, see merge_batched().
constexpr int kInLane = 8;
constexpr int kBatch = 8;
__device__ __forceinline__ void add_half8(float (&acc)[8], const uint4& v, float w) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&u[i]));
    acc[2 * i] = fmaf(w, f.x, acc[2 * i]);
    acc[2 * i + 1] = fmaf(w, f.y, acc[2 * i + 1]);
  }
}
static __global__ void __launch_bounds__(256, 4)
merge_batched_kernel(const int* __restrict__ q_ptr, const int* __restrict__ q_pairs, long long n_queries,
                     const __half* __restrict__ part_o, const float* __restrict__ part_lse,
                     const float* __restrict__ part_scale, long long capacity, __nv_bfloat16* __restrict__ o,
                     __nv_bfloat16* __restrict__ o_resid, float* __restrict__ lse, const RowMap o_map, int span) {
  if (!grid_begin()) return;
  constexpr int DH = 128;
  constexpr uint32_t FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, hl = lane & 15, half = lane >> 4;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  const int last = (int)(capacity - 1);
  const uint4* rows = reinterpret_cast<const uint4*>(part_o) + hl;
  for (long long g0 = warp * span; g0 < n_queries; g0 += nwarps * span) {
    const long long g = g0 + lane;
    int lo = 0, n = 1, n_raw = 1;        // lanes beyond the span or the last query behave like a directly written row
    if (lane < span && g < n_queries) {
      lo = q_ptr[g];
      const int hi_raw = q_ptr[g + 1];
      n_raw = hi_raw - lo;
      n = (int)(min((long long)hi_raw, capacity) - lo);
      if (n < 0) n = 0;
    }
    const bool direct = n == 1 && n_raw == 1;
    auto write_row = [&](int b, float (&acc)[8], float row_lse) {       // (b < 0: no query for this half-warp)
      if (b < 0) return;
      const long long gq = g0 + b;
      uint32_t h[4], r[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 x = __floats2bfloat162_rn(acc[2 * i], acc[2 * i + 1]);
        h[i] = *reinterpret_cast<const uint32_t*>(&x);
        const __nv_bfloat162 y = __floats2bfloat162_rn(acc[2 * i] - __uint_as_float(h[i] << 16), acc[2 * i + 1] - __uint_as_float(h[i] & 0xffff0000u));
        r[i] = *reinterpret_cast<const uint32_t*>(&y);
      }
      *reinterpret_cast<uint4*>(o + o_map.off(gq, DH) + hl * 8) = make_uint4(h[0], h[1], h[2], h[3]);
      if (o_resid) *reinterpret_cast<uint4*>(o_resid + gq * DH + hl * 8) = make_uint4(r[0], r[1], r[2], r[3]);
      if (hl == 0) lse[gq] = row_lse;
    };
    auto next_two = [&](uint32_t& todo) {          // this half-warp's query among the next two
      const int b1 = __ffs(todo) - 1;
      todo &= todo - 1;
      const int b2 = todo ? __ffs(todo) - 1 : -1;
      todo &= todo - 1;
      return half ? b2 : b1;
    };
    // ---- queries without a pair and queries of up to kInLane pairs
    uint32_t todo = __ballot_sync(FULL, !direct && n <= kInLane);
    if (todo) {
      int pos[kInLane];
      float w[kInLane];
      float out_lse = -INFINITY;
#pragma unroll
      for (int k = 0; k < kInLane; ++k) { pos[k] = 0; w[k] = 0.f; }
      if (!direct && n > 0 && n <= kInLane) {
        float sc[kInLane];
        float mx = -INFINITY, tot = 0.f;
#pragma unroll
        for (int k = 0; k < kInLane; ++k)
          if (k < n) pos[k] = min(max(q_pairs[lo + k], 0), last);
#pragma unroll
        for (int k = 0; k < kInLane; ++k) {
          sc[k] = 0.f;
          if (k < n) { w[k] = part_lse[pos[k]]; sc[k] = part_scale[pos[k]]; mx = fmaxf(mx, w[k]); }
        }
#pragma unroll
        for (int k = 0; k < kInLane; ++k) { w[k] = k < n ? expf(w[k] - mx) : 0.f; tot += w[k]; }
        const float inv = 1.0f / tot;
#pragma unroll
        for (int k = 0; k < kInLane; ++k) w[k] *= inv * sc[k];
        out_lse = mx + logf(tot);
      }
      while (todo) {
        const int b = next_two(todo), from = max(b, 0);
        const int nq = __shfl_sync(FULL, n, from), nb = b < 0 ? 0 : nq;
        const float row_lse = __shfl_sync(FULL, out_lse, from);
        float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        uint4 v[kInLane];
        float wk[kInLane];
#pragma unroll
        for (int k = 0; k < kInLane; ++k) {
          const int pk = __shfl_sync(FULL, pos[k], from);
          wk[k] = __shfl_sync(FULL, w[k], from);
          v[k] = make_uint4(0u, 0u, 0u, 0u);
          if (k < nb) v[k] = rows[(long long)pk * (DH / 8)];
        }
#pragma unroll
        for (int k = 0; k < kInLane; ++k) add_half8(acc, v[k], wk[k]);
        write_row(b, acc, row_lse);
      }
    }
    // ---- longer ones
    todo = __ballot_sync(FULL, n > kInLane);
    while (todo) {
      const int b = next_two(todo), from = max(b, 0);
      const int qlo = __shfl_sync(FULL, lo, from), nq = __shfl_sync(FULL, n, from);
      const int nb = b < 0 ? 0 : nq;
      const int n_max = max(__shfl_sync(FULL, nb, 0), __shfl_sync(FULL, nb, 16));
      // largest lse of the query; the first sixteen pairs' positions and lse stay in registers
      int pos0 = 0;
      float l0 = -INFINITY;
      if (hl < nb) { pos0 = min(max(q_pairs[qlo + hl], 0), last); l0 = part_lse[pos0]; }
      float mx = l0;
      for (int i = hl + 16; i < nb; i += 16) mx = fmaxf(mx, part_lse[min(max(q_pairs[qlo + i], 0), last)]);
#pragma unroll
      for (int s = 8; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(FULL, mx, s));
      float tot = 0.f;
      float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      for (int c0 = 0; c0 < n_max; c0 += 16) {
        if (c0 > 0) {
          pos0 = 0; l0 = -INFINITY;
          if (c0 + hl < nb) { pos0 = min(max(q_pairs[qlo + c0 + hl], 0), last); l0 = part_lse[pos0]; }
        }
        float w0 = 0.f;
        if (c0 + hl < nb) {
          w0 = expf(l0 - mx);
          tot += w0;
          w0 *= part_scale[pos0];
        }
#pragma unroll
        for (int k0 = 0; k0 < 16; k0 += kBatch) {
          if (c0 + k0 >= n_max) break;
          uint4 v[kBatch];
          float wk[kBatch];
#pragma unroll
          for (int k = 0; k < kBatch; ++k) {
            const int at = (lane & 16) + k0 + k;
            const int pk = __shfl_sync(FULL, pos0, at);
            wk[k] = __shfl_sync(FULL, w0, at);
            v[k] = make_uint4(0u, 0u, 0u, 0u);
            if (c0 + k0 + k < nb) v[k] = rows[(long long)pk * (DH / 8)];
          }
#pragma unroll
          for (int k = 0; k < kBatch; ++k) add_half8(acc, v[k], wk[k]);
        }
      }
#pragma unroll
      for (int s = 8; s > 0; s >>= 1) tot += __shfl_xor_sync(FULL, tot, s);
      const float inv = 1.0f / tot;
#pragma unroll
      for (int i = 0; i < 8; ++i) acc[i] *= inv;
      write_row(b, acc, mx + logf(tot));
    }
  }
}

// Fewer than 32 queries at a time where 32 would leave the SMs short of the 32 warps each holds: the walk through a warp's
// queries is a chain of loads, two queries after two (22,464 queries of 3 to 40 pairs: 23 us with 32).
static void merge_batched(const Dims& D, const int* q_ptr, const int* q_pairs, const __half* part_o, const float* part_lse,
                          const float* part_scale, long long cap, void* o, void* o_resid, float* lse, const RowMap& o_map,
                          cudaStream_t st) {
  const long long nq = (long long)D.BH * D.S;
  int span = 32;
  while (span > 2 && nq < (long long)sm_count() * 32 * span) span /= 2;
  launch_kernel(early_rows(D), merge_batched_kernel, (int)std::min<long long>((nq + 8 * span - 1) / (8 * span), sm_count() * 8),
                256, 0, st, q_ptr, q_pairs, nq, part_o, part_lse, part_scale, cap, (__nv_bfloat16*)o,
                (__nv_bfloat16*)o_resid, lse, o_map, span);
}

// ------------------------------------------------------------------------------ backward
// D = rowsum(dO * O), one warp per query; o and dO block-major or in raster order through their maps, the
// rounding residual of o always block-major.  If zero_acc is given, the fp32 dQ accumulator rows of the queries
// with at least one selected block (of every query without q_ptr) are cleared in the same pass: the only rows the
// backward kernel adds into.  zero_words: n_words counters to clear on the way.
// do_out (bf16, head_dim 128): a block-major copy of dO is left there on the way, so that dO in raster order needs no pass of its own (two
// batches of 32,760 queries x 12 heads: 166 us, 179 in two passes; 13,440 x 12: 41 and 43; 75,600 x 40: 761 and 783; small
// calls save a launch).
template <typename T, int DH>
__global__ void __launch_bounds__(256)
rowdot_kernel(const T* __restrict__ o, const T* __restrict__ o_resid, const T* __restrict__ d_o, long long n_queries,
              float* __restrict__ Dv, const RowMap do_map, const RowMap o_map,
              float* __restrict__ zero_acc, const int* __restrict__ q_ptr, T* __restrict__ do_out,
              int* __restrict__ zero_words, long long n_words) {
  if (!grid_begin()) return;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_words; i += (long long)gridDim.x * blockDim.x)
    zero_words[i] = 0;
  constexpr int C = DH / 32;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  if constexpr (C == 4 && sizeof(T) == 2) {
    // Four rows per warp and trip, in phases (row offsets, loads, sums, stores), so that the twelve 8-byte
    // loads of a lane are in flight together.
    constexpr int R = 4;
    for (long long g0 = warp * R; g0 < n_queries; g0 += nwarps * R) {
      uint2 ov[R], rv[R], dv[R];
      bool zero[R], used[R];
      // with the lists at hand, a query without a selected block is skipped: nothing reads its D
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const long long g = min(g0 + r, n_queries - 1);
        used[r] = !q_ptr || __ldg(q_ptr + g + 1) - __ldg(q_ptr + g) >= 1;
        zero[r] = zero_acc && g0 + r < n_queries && used[r];
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const long long g = min(g0 + r, n_queries - 1);
        ov[r] = dv[r] = rv[r] = make_uint2(0u, 0u);
        if (used[r]) {
          ov[r] = *reinterpret_cast<const uint2*>(o + o_map.off(g, DH) + lane * 4);
          if (o_resid) rv[r] = *reinterpret_cast<const uint2*>(o_resid + g * DH + lane * 4);
        }
        if (used[r] || do_out) dv[r] = *reinterpret_cast<const uint2*>(d_o + do_map.off(g, DH) + lane * 4);
      }
      float a[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        auto lo = [](uint32_t u) { return __uint_as_float(u << 16); };
        auto hi = [](uint32_t u) { return __uint_as_float(u & 0xffff0000u); };
        a[r] = (lo(ov[r].x) + lo(rv[r].x)) * lo(dv[r].x);
        a[r] = fmaf(hi(ov[r].x) + hi(rv[r].x), hi(dv[r].x), a[r]);
        a[r] = fmaf(lo(ov[r].y) + lo(rv[r].y), lo(dv[r].y), a[r]);
        a[r] = fmaf(hi(ov[r].y) + hi(rv[r].y), hi(dv[r].y), a[r]);
      }
#pragma unroll
      for (int s = 16; s > 0; s >>= 1)
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] += __shfl_xor_sync(0xffffffffu, a[r], s);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (g0 + r >= n_queries) break;
        if (lane == 0) Dv[g0 + r] = a[r];
        if (do_out) *reinterpret_cast<uint2*>(do_out + (g0 + r) * DH + lane * 4) = dv[r];
        if (zero[r]) reinterpret_cast<float4*>(zero_acc + (g0 + r) * DH)[lane] = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    return;
  }
  for (long long g = warp; g < n_queries; g += nwarps) {
    float a = 0.f;
    const T* do_row = d_o + do_map.off(g, DH);
    const T* o_row = o + o_map.off(g, DH);
    if (zero_acc && (!q_ptr || __ldg(q_ptr + g + 1) - __ldg(q_ptr + g) >= 1)) {
      float4* row = reinterpret_cast<float4*>(zero_acc + g * DH);
      for (int c = lane; c < DH / 4; c += 32) row[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      float ov = to_f32<T>(o_row[lane * C + c]);
      if (o_resid) ov += to_f32<T>(o_resid[g * DH + lane * C + c]);
      a = fmaf(ov, to_f32<T>(do_row[lane * C + c]), a);
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) a += __shfl_xor_sync(0xffffffffu, a, s);
    if (lane == 0) Dv[g] = a;
  }
}

// dK, dV: key-stationary.  A CTA owns 64 keys of one key block (or of the whole sequence when DENSE) and streams the queries that
// selected the block; dK and dV are written once.  dQ goes into dq_acc (fp32, cleared before), in whatever order the items come to
// it, but as ONE part per query and key block, so that a query with one or two blocks has the same dq in every call:
//   kDqTile     blocks of one tile of keys: the tile's part is the block's.
//   kDqCluster  blocks of up to eight: a cluster takes the block, a tile per CTA, and walks its list together.  Every CTA leaves its
//               tile's part where dO was, and adds up a share of the rows in the order of the tiles.
//   kDqNone     longer blocks and the dense path: attn_bwd_dq_kernel.
// fp32 backward of 13 heads x 4,096 tokens in blocks of 512 keys, head_dim 64 / 128: clusters 850 / 1483 us, the kernel of its own
// 998 / 1613; a part per tile, which leaves dq to the order of the CTAs, 704 / 1123.  8 x 2,496 in blocks of 156, head_dim 64: 101,
// 122, 89.
enum DqRoute { kDqNone, kDqTile, kDqCluster };
constexpr int kDqClusterMax = 8;               // what every device schedules as one cluster
__device__ __forceinline__ void red_add4(float* to, const float* x, float scale) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(to), "f"(x[0] * scale), "f"(x[1] * scale), "f"(x[2] * scale),
               "f"(x[3] * scale)
               : "memory");
}
template <int DH> constexpr int kBwdSmem = (4 * kTileFloats<DH> + kRows * kLdP) * 4;      // K, V, Q, dO, weights
template <typename T, int DH, bool DENSE, DqRoute DQ>
__global__ void __launch_bounds__(kThreads, DH == 64 ? 2 : 1)
attn_bwd_dkdv_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                     const T* __restrict__ d_o, const float* __restrict__ lse, const float* __restrict__ Dv,
                     const int* __restrict__ kb_ptr, const int* __restrict__ q_idx, int S, int Nb, int sb, int BH,
                     float scale, long long capacity, T* __restrict__ dk, T* __restrict__ dv, float* __restrict__ dq_acc) {
  if (!grid_begin()) return;
  extern __shared__ __align__(16) float simt_smem[];
  float* Ks = simt_smem;
  float* Vs = Ks + kTileFloats<DH>;
  float* Qs = Vs + kTileFloats<DH>;
  float* dOs = Qs + kTileFloats<DH>;
  float* Ps = dOs + kTileFloats<DH>;           // [key][query]: weights, then dS
  __shared__ float s_lse[kRows], s_D[kRows];
  __shared__ int s_row[kRows];
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  const int span = DENSE ? S : sb;
  const int tiles = (span + kRows - 1) / kRows;
  const long long n_items = (long long)BH * (DENSE ? 1 : Nb) * tiles;
  // (kDqCluster: clusters of `tiles` CTAs, and the grid is whole clusters: a CTA's tile is its rank)
  cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
  auto meet = [&]() { if constexpr (DQ == kDqCluster) cluster.sync(); else __syncthreads(); };
  for (long long item = blockIdx.x; item < n_items; item += gridDim.x) {
    const int tile = (int)(item % tiles);
    const long long kbi = item / tiles;          // DENSE: bh ; sparse: bh * Nb + j
    const int bh = DENSE ? (int)kbi : (int)(kbi / Nb);
    const int j0 = DENSE ? 0 : (int)(kbi - (long long)bh * Nb);
    const int key0 = j0 * sb + tile * kRows, keys = min(kRows, span - tile * kRows);
    const long long head_off = (long long)bh * S;
    long long list_lo = 0, list_hi = S;
    if (!DENSE) { list_lo = min((long long)kb_ptr[kbi], capacity); list_hi = min((long long)kb_ptr[kbi + 1], capacity); }
    float dk_[4][DH / 16], dv_[4][DH / 16];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < DH / 16; ++c) dk_[i][c] = dv_[i][c] = 0.f;
    const bool live = (ty & ~1) * 4 < keys;    // (a warp has eight rows)
    __syncthreads();                           // (the item before is through with the shared memory)
    {
      TileRegs<T, DH> x, y;
      x.fetch(k + head_off * DH, keys, [&](int i) { return key0 + i; });
      y.fetch(v + head_off * DH, keys, [&](int i) { return key0 + i; });
      x.store(Ks);
      y.store(Vs);
    }
    for (long long t0 = list_lo; t0 < list_hi; t0 += kRows) {
      const int nq = (int)min((long long)kRows, list_hi - t0);
      meet();                                  // (kDqCluster: the others are through with this CTA's part)
      if (t < kRows) {
        float a = INFINITY, b = 0.f;             // (lse = +inf for rows that are none: their weights are 0)
        int x = 0;
        if (t < nq) {
          x = DENSE ? (int)t0 + t : q_idx[t0 + t];
          a = lse[head_off + x]; b = Dv[head_off + x];
        }
        s_lse[t] = a; s_D[t] = b; s_row[t] = x;
      }
      __syncthreads();
      {
        TileRegs<T, DH> x, y;
        x.fetch(q + head_off * DH, nq, [&](int i) { return s_row[i]; });
        y.fetch(d_o + head_off * DH, nq, [&](int i) { return s_row[i]; });
        x.store(Qs);
        y.store(dOs);
      }
      __syncthreads();
      const int nq4 = (nq + 3) & ~3;
      float p[4][4];
      if (live) {
        dot_tiles<DH>(Ks, Qs, ty, tx, nq, p);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int qq = tx + 16 * j;
            p[i][j] = 4 * ty + i < keys && qq < nq ? expf(p[i][j] * scale - s_lse[qq]) : 0.f;
            Ps[(4 * ty + i) * kLdP + qq] = p[i][j];
          }
        __syncwarp();                          // (a warp reads its own eight rows)
        add_weighted<DH>(Ps, dOs, ty, tx, nq4, dv_);
        float s[4][4];
        dot_tiles<DH>(Vs, dOs, ty, tx, nq, s);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int qq = tx + 16 * j;
            Ps[(4 * ty + i) * kLdP + qq] = qq < nq ? p[i][j] * (s[i][j] - s_D[qq]) : 0.f;
          }
        __syncwarp();
        add_weighted<DH>(Ps, Qs, ty, tx, nq4, dk_);
      }
      if constexpr (DQ != kDqNone) {
        __syncthreads();
        if ((ty & ~1) * 4 < nq) {              // thread: queries 4 ty + i
          float dq_[4][DH / 16];
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int c = 0; c < DH / 16; ++c) dq_[i][c] = 0.f;
          add_weighted_t<DH>(Ps, Ks, ty, tx, keys, dq_);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (4 * ty + i >= nq) break;
            float* row = DQ == kDqTile ? dq_acc + (head_off + s_row[4 * ty + i]) * DH + 4 * tx : dOs + (4 * ty + i) * kLd<DH> + 4 * tx;
#pragma unroll
            for (int g = 0; g < DH / 64; ++g) {
              if (DQ == kDqTile) red_add4(row + 64 * g, &dq_[i][4 * g], scale);
              else *reinterpret_cast<float4*>(row + 64 * g) = make_float4(dq_[i][4 * g], dq_[i][4 * g + 1], dq_[i][4 * g + 2], dq_[i][4 * g + 3]);
            }
          }
        }
      }
      if constexpr (DQ == kDqCluster) {
        meet();
        constexpr int V = DH / 4;
        for (int u = (int)cluster.block_rank() * kThreads + t; u < nq * V; u += tiles * kThreads) {
          const int r = u / V, c = u % V * 4;
          float sum[4] = {0.f, 0.f, 0.f, 0.f};
          for (int n = 0; n < tiles; ++n) {
            const float4 x = *reinterpret_cast<const float4*>(cluster.map_shared_rank(dOs, n) + r * kLd<DH> + c);
            sum[0] += x.x; sum[1] += x.y; sum[2] += x.z; sum[3] += x.w;
          }
          red_add4(dq_acc + (head_off + s_row[r]) * DH + c, sum, scale);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (4 * ty + i >= keys) break;
#pragma unroll
      for (int g = 0; g < DH / 64; ++g) {
        const long long at = (head_off + key0 + 4 * ty + i) * DH + 64 * g + 4 * tx;
        store4(dk + at, make_float4(dk_[i][4 * g] * scale, dk_[i][4 * g + 1] * scale, dk_[i][4 * g + 2] * scale, dk_[i][4 * g + 3] * scale));
        store4(dv + at, make_float4(dv_[i][4 * g], dv_[i][4 * g + 1], dv_[i][4 * g + 2], dv_[i][4 * g + 3]));
      }
    }
  }
  if constexpr (DQ == kDqCluster) meet();      // (nobody reads this CTA's part any more)
}

// dQ: query-stationary, a CTA takes 64 rows of a head (dense; written directly) or of the list of a key block that is too long for
// a cluster; its part of dQ over the whole block is then added into dq_acc.  It works S and dP out again.
template <typename T, int DH, bool DENSE>
__global__ void __launch_bounds__(kThreads, DH == 64 ? 2 : 1)
attn_bwd_dq_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                   const T* __restrict__ d_o, const float* __restrict__ lse, const float* __restrict__ Dv,
                   const int* __restrict__ kb_ptr, const int* __restrict__ q_idx, const int* __restrict__ item_ptr, int n_kb, int S,
                   int Nb, int sb, int BH, float scale, long long capacity, T* __restrict__ dq, float* __restrict__ dq_acc) {
  if (!grid_begin()) return;
  extern __shared__ __align__(16) float simt_smem[];
  float* Qs = simt_smem;
  float* dOs = Qs + kTileFloats<DH>;
  float* Ks = dOs + kTileFloats<DH>;
  float* Vs = Ks + kTileFloats<DH>;
  float* Ps = Vs + kTileFloats<DH>;            // [query][key]: dS
  __shared__ int s_row[DENSE ? 1 : kRows];     // in-head positions of a list's queries
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  const int tiles_per_head = (S + kRows - 1) / kRows, n_items = DENSE ? BH * tiles_per_head : item_ptr[n_kb];
  for (int item = blockIdx.x; item < n_items; item += gridDim.x) {
    Item it;
    int rows;
    if (DENSE) {
      it.bh = item / tiles_per_head;
      it.list_lo = (item - it.bh * tiles_per_head) * kRows;
      it.key_begin = 0; it.key_end = S;
      rows = min(kRows, S - it.list_lo);
    } else {
      it = decode_sparse(item, item_ptr, n_kb, kb_ptr, Nb, sb, kRows, capacity);
      rows = it.list_hi - it.list_lo;
    }
    const long long head_off = (long long)it.bh * S;
    __syncthreads();                           // (the item before is through with the shared memory)
    if (!DENSE) {
      if (t < rows) s_row[t] = q_idx[it.list_lo + t];
      __syncthreads();
    }
    auto row_of = [&](int i) { return DENSE ? it.list_lo + i : s_row[DENSE ? 0 : i]; };
    float row_lse[4], row_D[4], acc[4][DH / 16];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool ok = 4 * ty + i < rows;
      row_lse[i] = ok ? lse[head_off + row_of(4 * ty + i)] : INFINITY;
      row_D[i] = ok ? Dv[head_off + row_of(4 * ty + i)] : 0.f;
#pragma unroll
      for (int c = 0; c < DH / 16; ++c) acc[i][c] = 0.f;
    }
    {
      TileRegs<T, DH> x, y;
      x.fetch(q + head_off * DH, rows, row_of);
      y.fetch(d_o + head_off * DH, rows, row_of);
      x.store(Qs);
      y.store(dOs);
    }
    const bool live = (ty & ~1) * 4 < rows;    // (a warp has eight rows)
    for (int t0 = it.key_begin; t0 < it.key_end; t0 += kRows) {
      const int nv = min(kRows, it.key_end - t0);
      {
        TileRegs<T, DH> x, y;
        x.fetch(k + head_off * DH, nv, [&](int i) { return t0 + i; });
        y.fetch(v + head_off * DH, nv, [&](int i) { return t0 + i; });
        __syncthreads();
        x.store(Ks);
        y.store(Vs);
      }
      __syncthreads();
      if (live) {
        float p[4][4], s[4][4];
        dot_tiles<DH>(Qs, Ks, ty, tx, nv, p);
        dot_tiles<DH>(dOs, Vs, ty, tx, nv, s);
        __syncwarp();
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int key = tx + 16 * j;
            Ps[(4 * ty + i) * kLdP + key] = key < nv ? expf(p[i][j] * scale - row_lse[i]) * (s[i][j] - row_D[i]) : 0.f;
          }
        __syncwarp();                          // (a warp reads its own eight rows)
        add_weighted<DH>(Ps, Ks, ty, tx, (nv + 3) & ~3, acc);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (4 * ty + i >= rows) break;
      const long long at = (head_off + row_of(4 * ty + i)) * DH + 4 * tx;
#pragma unroll
      for (int g = 0; g < DH / 64; ++g) {
        if (DENSE) store4(dq + at + 64 * g, make_float4(acc[i][4 * g] * scale, acc[i][4 * g + 1] * scale, acc[i][4 * g + 2] * scale, acc[i][4 * g + 3] * scale));
        else red_add4(dq_acc + at + 64 * g, &acc[i][4 * g], scale);
      }
    }
  }
}

// Rows of the tensor-core backward's fp32 dQ accumulator -> output dtype.  The accumulator keeps its 128 columns in the
// order that kernel reduces them in: position 32 w + 4 r + a holds column 32 w + r + 8 a.  Queries without a selected
// block (q_ptr given) get zeros without a read.  parts: accumulators behind one another, added up in order.
template <typename T>
__global__ void __launch_bounds__(256)
cast_rows_kernel(const float* __restrict__ src, T* __restrict__ dst, const int* __restrict__ q_ptr, long long n_queries,
                 const RowMap map, int parts) {
  if (!grid_begin()) return;
  constexpr int DH = 128;
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long nwarps = (long long)gridDim.x * (blockDim.x >> 5);
  // this lane's output columns 4 lane .. 4 lane + 3 sit at positions at, at + 4, at + 8, at + 12: one line of the row
  const int at = (lane & ~7) * 4 + 16 * (lane & 1) + ((lane & 7) >> 1);
  // Four rows per warp and trip, in phases (list bounds, row offsets, loads, stores), so that the
  // loads of the four rows are in flight together.
  constexpr int R = 4;
  for (long long g0 = warp * R; g0 < n_queries; g0 += nwarps * R) {
    bool used[R];
    long long off[R];
    float4 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const long long g = min(g0 + r, n_queries - 1);
      used[r] = !q_ptr || __ldg(q_ptr + g + 1) > __ldg(q_ptr + g);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) off[r] = map.off(min(g0 + r, n_queries - 1), DH);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (used[r]) {
        const float* row = src + min(g0 + r, n_queries - 1) * DH + at;
        v[r] = make_float4(__ldg(row), __ldg(row + 4), __ldg(row + 8), __ldg(row + 12));
      }
    }
    for (int part = 1; part < parts; ++part) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const float* row = src + (part * n_queries + min(g0 + r, n_queries - 1)) * DH + at;
        v[r].x += __ldg(row); v[r].y += __ldg(row + 4); v[r].z += __ldg(row + 8); v[r].w += __ldg(row + 12);
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (g0 + r < n_queries) store4(dst + off[r] + lane * 4, v[r]);
  }
}

// fp32 accumulator -> output dtype.
template <typename T>
__global__ void __launch_bounds__(256)
cast_kernel(const float* __restrict__ src, T* __restrict__ dst, long long n4) {
  if (!grid_begin()) return;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (long long)gridDim.x * blockDim.x)
    store4(dst + 4 * i, *reinterpret_cast<const float4*>(src + 4 * i));
}

}  // namespace simt
}  // namespace vmoba
