// Step 1 of VMoBA (Eq. 1): reorder tokens of the T x H x W latent into 1D / 2D / 3D blocks,
// and the inverse reordering.  A pure permutation of head_dim-wide rows, bound by HBM
// bandwidth: every row is read once and written once with 16-byte vector accesses.
#include "common.cuh"

namespace vmoba {

struct PermGeom {
  int H, W, bT, bH, bW, nH, nW, sb;
};

// Eq. 1: raster index of the token at block-major position p.
__device__ __forceinline__ int perm_of(const PermGeom& g, int p) {
  int j = p / g.sb, r = p - j * g.sb;
  int jw = j % g.nW, jt_h = j / g.nW;
  int jh = jt_h % g.nH, jt = jt_h / g.nH;
  int rw = r % g.bW, rt_h = r / g.bW;
  int rh = rt_h % g.bH, rt = rt_h / g.bH;
  int t = jt * g.bT + rt, h = jh * g.bH + rh, w = jw * g.bW + rw;
  return (t * g.H + h) * g.W + w;
}

constexpr int kMaxTensors = 4;
struct PartTensors {
  const uint4* src[kMaxTensors];
  uint4* dst[kMaxTensors];
  long long rs_b[kMaxTensors], rs_s[kMaxTensors], rs_h[kMaxTensors];      // raster strides in 16-byte vectors
};

// Rows are enumerated as ((b * S + p) * heads + head): consecutive rows share a token, so the
// raster side is touched in runs of heads * head_dim contiguous elements.  A warp takes ROWS rows:
// lane l derives the two offsets of row l once, then the warp streams the rows' 16-byte vectors
// with the offsets broadcast by shuffle, the loads of four passes ahead of their stores.  Bound by HBM.
// Four passes and a CTA per 8 x ROWS rows: three tensors of 75,600 x 40 heads 733 us (6340 GB/s), of 32,760 x 12 x 2 197, of
// 13,440 x 12 53.  Eight passes and at most 32 CTAs per SM, which walk on, took 808, 221 and 57, eight passes alone 820, 220 and
// 58, two passes 757, 205 and 57 (one tensor after the other, as before, 770, 220 and 69).
// blockIdx.y: tensor (one launch for up to four of them; the first one's CTAs also write the permutation tables).
template <int VEC_PER_ROW, int ROWS>   // 16-byte vectors per row: head_dim * elem_size / 16
__global__ void __launch_bounds__(256)
partition_kernel(PermGeom g, int S, int heads, int n_rows, int inverse, const __grid_constant__ PartTensors t,
                 int32_t* __restrict__ perm, int32_t* __restrict__ inv_perm) {
  if (!grid_begin()) return;
  constexpr int ROWS_PER_PASS = 32 / VEC_PER_ROW > 0 ? 32 / VEC_PER_ROW : 1;
  constexpr int PASSES = ROWS / ROWS_PER_PASS;
  // passes whose loads are in flight together (few rows per warp: all of them)
  constexpr int U = PASSES < 4 || ROWS < 32 ? PASSES : 4;
  const int lane = threadIdx.x & 31;
  const long long base = ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * ROWS;
  if (base >= n_rows) return;
  const int k = blockIdx.y;
  const uint4* __restrict__ src = t.src[k];
  uint4* __restrict__ dst = t.dst[k];
  const int sub = lane / VEC_PER_ROW, vec = lane % VEC_PER_ROW;
  const long long row = base + lane;
  long long off_r = 0, off_bm = 0;
  if (lane < ROWS && row < n_rows) {
    const unsigned bp = (unsigned)row / (unsigned)heads, head = (unsigned)row - bp * heads;
    const unsigned b = bp / (unsigned)S;
    const int p = (int)(bp - b * S);
    const int r = perm_of(g, p);
    off_r = b * t.rs_b[k] + (long long)r * t.rs_s[k] + head * t.rs_h[k];
    off_bm = (((long long)b * heads + head) * S + p) * VEC_PER_ROW;
    if (k == 0 && b == 0 && head == 0) {
      if (perm) perm[p] = r;
      if (inv_perm) inv_perm[r] = p;
    }
  }
  const long long off_src = inverse ? off_bm : off_r;
  const long long off_dst = inverse ? off_r : off_bm;
  const int left = (int)min((long long)ROWS, n_rows - base);
#pragma unroll 1
  for (int p0 = 0; p0 < PASSES; p0 += U) {
    uint4 v[U];
    long long to[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int from = (p0 + u) * ROWS_PER_PASS + sub;
      const long long so = __shfl_sync(0xffffffffu, off_src, from);
      to[u] = __shfl_sync(0xffffffffu, off_dst, from);
      if (from < left) v[u] = __ldg(src + so + vec);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if ((p0 + u) * ROWS_PER_PASS + sub < left) dst[to[u] + vec] = v[u];
  }
}

template <int V>
static int launch_partition(const Dims& D, const PermGeom& g, int inverse, int n, const PartTensors& t, int32_t* perm,
                            int32_t* inv_perm, cudaStream_t st) {
  const long long n_rows = (long long)D.BH * D.S;
  auto go = [&](auto kernel, int rows) {
    launch_kernel(kernel, dim3((unsigned)((n_rows + 8 * rows - 1) / (8 * rows)), n), 256, 0, st, g, D.S, D.heads,
                  (int)n_rows, inverse, t, perm, inv_perm);
  };
  // 32 rows per warp once that gives every SM its 64 warps; below, 8 rows, for more warps to hide a pass's latency
  // (22,464 rows, bf16, head_dim 128: one tensor 9.1 us with 32, three tensors 7.5 us with 8)
  if (n_rows * n >= (long long)sm_count() * 64 * 32) go(partition_kernel<V, 32>, 32);
  else go(partition_kernel<V, 8>, 8);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

static int partition_impl(const vmoba_shape* shape, int inverse, int n, const void* const* src, void* const* dst,
                          const int64_t (*strides)[3], int32_t* perm, int32_t* inv_perm, void* stream) {
  Dims D;
  int rc = make_dims(shape, &D);
  if (rc) return rc;
  if (n < 1 || n > kMaxTensors || !src || !dst || !strides) return VMOBA_ERR_ARG;
  if (inverse != 0 && inverse != 1) return VMOBA_ERR_ARG;
  if ((long long)D.BH * D.S > INT32_MAX) return VMOBA_ERR_SHAPE;
  const int per_vec = 16 / D.es;
  PartTensors t = {};
  for (int k = 0; k < n; ++k) {
    if (!src[k] || !dst[k] || !aligned16(src[k]) || !aligned16(dst[k])) return VMOBA_ERR_ARG;
    for (int i = 0; i < 3; ++i)
      if (strides[k][i] < 0 || strides[k][i] % per_vec) return VMOBA_ERR_ARG;
    t.src[k] = static_cast<const uint4*>(src[k]);
    t.dst[k] = static_cast<uint4*>(dst[k]);
    t.rs_b[k] = strides[k][0] / per_vec; t.rs_s[k] = strides[k][1] / per_vec; t.rs_h[k] = strides[k][2] / per_vec;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  PermGeom g{D.H, D.W, D.bT, D.bH, D.bW, D.nH, D.nW, D.sb};
  switch (D.d * D.es / 16) {
    case 8: return launch_partition<8>(D, g, inverse, n, t, perm, inv_perm, st);
    case 16: return launch_partition<16>(D, g, inverse, n, t, perm, inv_perm, st);
    case 32: return launch_partition<32>(D, g, inverse, n, t, perm, inv_perm, st);
    default: return VMOBA_ERR_NOT_IMPLEMENTED;
  }
}

}  // namespace vmoba

using namespace vmoba;

extern "C" int vmoba_partition(const vmoba_shape* shape, int inverse, const void* src, void* dst,
                               const int64_t raster_strides_bsh[3], int32_t* perm_or_null,
                               int32_t* inv_perm_or_null, void* stream) {
  if (!raster_strides_bsh) {
    Dims D;
    const int rc = make_dims(shape, &D);
    return rc ? rc : VMOBA_ERR_ARG;
  }
  const int64_t strides[1][3] = {{raster_strides_bsh[0], raster_strides_bsh[1], raster_strides_bsh[2]}};
  return partition_impl(shape, inverse, 1, &src, &dst, strides, perm_or_null, inv_perm_or_null, stream);
}

extern "C" int vmoba_partition_many(const vmoba_shape* shape, int inverse, int32_t n, const void* const* src,
                                    void* const* dst, const int64_t (*raster_strides_bsh)[3], int32_t* perm_or_null,
                                    int32_t* inv_perm_or_null, void* stream) {
  return partition_impl(shape, inverse, n, src, dst, raster_strides_bsh, perm_or_null, inv_perm_or_null, stream);
}
