// Step 1b + Step 2a of VMoBA: mean key-block centroids (Eq. 2) and the query x centroid
// similarity map S_hat = q b^T (Section 3.3), both in fp32.
//
// Both kernels are bound by HBM traffic: K is read once for the centroids, Q once for the
// scores, and the [S, N_b] fp32 score matrix is written once.  The contraction itself
// (2 * S * N_b * d flops) is small next to that and runs on the fp32 FMA pipe so that the
// scores carry fp32 accuracy (the selection cutoff is compared in fp32).
#include <algorithm>

#include "common.cuh"

namespace vmoba {

// scores_tc.cu: tensor-core scores for bf16 / head_dim 128
size_t scores_tc_ws_bytes(const Dims& D);
CentroidParts scores_tc_parts(const Dims& D, void* ws);
int scores_tc(const Dims& D, const void* q_bm, const CentroidParts& cent, float* scores, float* range, int32_t* status, cudaStream_t st);

size_t scores_ws_bytes(const Dims& D) {
  return (D.dtype == VMOBA_BF16 && D.d == 128) ? scores_tc_ws_bytes(D) : 256;
}

// Eq. 2.  A CTA sums DH / SPLIT columns of one (batch, head, block) with 1024 / DH row lanes, each over every (1024 / DH)-th
// row in order, then adds the row lanes' sums in order: the result does not depend on SPLIT.  Bound by HBM bandwidth, with
// few blocks by the latency of a thread's chain of loads, hence the many in flight.
// The blocks are taken from the last position of every head to the first: the partition of k, in token order over all heads,
// ends there, and what it wrote last is still in L2.
// For the tensor-core scores kernel it also leaves the centroids' parts (a launch of its own before), and in any case
// the score range's starting values for the kernel that follows.
template <typename T, int DH, int SPLIT>
__global__ void __launch_bounds__((1024 / DH) * (DH * (int)sizeof(T) / 16 / SPLIT))
centroid_kernel(const T* __restrict__ k_bm, float* __restrict__ cent, int sb, int BH, int Nb, CentroidParts out, float* __restrict__ range) {
  if (!grid_begin()) return;
  if (range && blockIdx.x == 0)
    for (int h = threadIdx.x; h < BH; h += blockDim.x) { range[2 * h] = INFINITY; range[2 * h + 1] = -INFINITY; }
  constexpr int W = 16 / sizeof(T);          // columns per thread
  constexpr int V = DH / W / SPLIT;          // threads per row
  constexpr int RL = 1024 / DH;              // row lanes
  constexpr int U = SPLIT > 1 ? 32 : 8;      // 16-byte loads of a thread in flight
  __shared__ float red[RL][V * W];
  const unsigned i = gridDim.x - 1 - blockIdx.x;
  const int part = i % SPLIT, j = (int)(i / SPLIT / BH), bh = (int)(i / SPLIT - (unsigned)j * BH);
  const long long blk = (long long)bh * Nb + j;
  const int col = threadIdx.x % V, rl = threadIdx.x / V;
  const uint4* base = reinterpret_cast<const uint4*>(k_bm + blk * (long long)sb * DH) + part * V + col;
  float acc[W];
#pragma unroll
  for (int c = 0; c < W; ++c) acc[c] = 0.f;
  for (int r0 = rl; r0 < sb; r0 += RL * U) {
    uint4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r0 + u * RL < sb) x[u] = __ldg(base + (long long)(r0 + u * RL) * (DH / W));
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (r0 + u * RL >= sb) break;
      const uint32_t w[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
      for (int c = 0; c < W; ++c) {
        if constexpr (W == 4) acc[c] += __uint_as_float(w[c]);
        else acc[c] += __uint_as_float(c & 1 ? w[c >> 1] & 0xffff0000u : w[c >> 1] << 16);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < W; ++c) red[rl][col * W + c] = acc[c];
  __syncthreads();
  const float inv = 1.0f / (float)sb;
  for (int c = threadIdx.x; c < V * W; c += RL * V) {
    float s = red[0][c];
    for (int r = 1; r < RL; ++r) s += red[r][c];
    const float x = s * inv;
    cent[blk * DH + part * V * W + c] = x;
    if constexpr (sizeof(T) == 2 && DH == 128) {
      const __nv_bfloat16 b1 = __float2bfloat16_rn(x);
      const float r1 = x - __bfloat162float(b1);
      const __nv_bfloat16 b2 = __float2bfloat16_rn(r1);
      const float r2 = r1 - __bfloat162float(b2);
      const long long at = ((long long)bh * out.Nb_pad + j) * DH + part * V * W + c;
      out.parts[at] = b1;
      out.parts[out.n + at] = b2;
      out.parts[2 * out.n + at] = __float2bfloat16_rn(r2);
      if (j == Nb - 1)
        for (int p = 0; p < 3; ++p)
          for (int r = 1; r < out.Nb_pad - j; ++r) out.parts[p * out.n + at + r * DH] = __float2bfloat16_rn(0.f);
    }
  }
}

template <typename T, int DH>
static void run_centroids(const Dims& D, const T* k, float* cent, const CentroidParts& parts, float* range, cudaStream_t st) {
  constexpr int THREADS = (1024 / DH) * (DH * (int)sizeof(T) / 16);
  const long long n = (long long)D.BH * D.Nb;
  // Four CTAs per block where one would not give every SM four.  12 heads: 24 blocks of 1,400 keys 41 us with one, 24 with
  // four; 16 blocks of 840 keys 20 and 8; 140 blocks of 234 keys 15 with one.
  if (n < sm_count() * 4ll)
    launch_kernel(centroid_kernel<T, DH, 4>, (unsigned)(4 * n), THREADS / 4, 0, st, k, cent, D.sb, D.BH, D.Nb, parts, range);
  else
    launch_kernel(centroid_kernel<T, DH, 1>, (unsigned)n, THREADS, 0, st, k, cent, D.sb, D.BH, D.Nb, parts, range);
}

// fp32 tile GEMM: a CTA computes 64 queries x 64 blocks with the whole head_dim in shared
// memory (operands stored transposed so that each thread reads its 4x4 micro-tile as float4).
template <typename T, int DH>
__global__ void __launch_bounds__(256)
scores_kernel(const T* __restrict__ q_bm, const float* __restrict__ cent, float* __restrict__ scores,
              int S, int Nb, float* __restrict__ range) {
  if (!grid_begin()) return;
  extern __shared__ float smem[];
  constexpr int LD = 64 + 4;
  float* qT = smem;                 // [DH][LD]
  float* bT = smem + DH * LD;       // [DH][LD]
  const int bh = blockIdx.z;
  const int q0 = blockIdx.x * 64;
  const int tid = threadIdx.x;
  const T* qh = q_bm + ((long long)bh * S + q0) * DH;
  // Load the query tile once: thread t reads float4 #(t % (DH/4)) of row (t / (DH/4)) + k * rows_per_pass.
  constexpr int V = DH / 4;
  for (int i = tid; i < 64 * V; i += 256) {
    int r = i / V, c4 = i % V;
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q0 + r < S) x = load4(qh + (long long)r * DH + c4 * 4);
    qT[(c4 * 4 + 0) * LD + r] = x.x;
    qT[(c4 * 4 + 1) * LD + r] = x.y;
    qT[(c4 * 4 + 2) * LD + r] = x.z;
    qT[(c4 * 4 + 3) * LD + r] = x.w;
  }
  const int ty = tid / 16, tx = tid % 16;
  const float* ch = cent + (long long)bh * Nb * DH;
  float* out = scores + ((long long)bh * S + q0) * Nb;
  float lo = INFINITY, hi = -INFINITY;      // of this thread's scores
  for (int j0 = 0; j0 < Nb; j0 += 64) {
    __syncthreads();
    for (int i = tid; i < 64 * V; i += 256) {
      int r = i / V, c4 = i % V;
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j0 + r < Nb) x = *reinterpret_cast<const float4*>(ch + (long long)(j0 + r) * DH + c4 * 4);
      bT[(c4 * 4 + 0) * LD + r] = x.x;
      bT[(c4 * 4 + 1) * LD + r] = x.y;
      bT[(c4 * 4 + 2) * LD + r] = x.z;
      bT[(c4 * 4 + 3) * LD + r] = x.w;
    }
    __syncthreads();
    float acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 8
    for (int c = 0; c < DH; ++c) {
      float4 a = *reinterpret_cast<const float4*>(qT + c * LD + ty * 4);
      float4 b = *reinterpret_cast<const float4*>(bT + c * LD + tx * 4);
      float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int r = ty * 4 + i;
      if (q0 + r >= S) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int col = j0 + tx * 4 + j;
        if (col < Nb) {
          out[(long long)r * Nb + col] = acc[i][j];
          lo = fminf(lo, acc[i][j]);
          hi = fmaxf(hi, acc[i][j]);
        }
      }
    }
  }
  if (range) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((tid & 31) == 0 && lo <= hi) { atomic_min_f32(range + 2 * bh, lo); atomic_max_f32(range + 2 * bh + 1, hi); }
  }
}

template <typename T, int DH>
static int run_scores(const Dims& D, const void* q, const void* k, float* cent, float* scores, float* range, void* ws,
                      int32_t* status, cudaStream_t st) {
  const bool tc = D.dtype == VMOBA_BF16 && DH == 128;
  const CentroidParts parts = tc ? scores_tc_parts(D, ws) : CentroidParts();
  run_centroids<T, DH>(D, static_cast<const T*>(k), cent, parts, range, st);
  VMOBA_LAUNCH_OK(1);
  if (tc) return scores_tc(D, q, parts, scores, range, status, st);
  size_t smem = 2 * DH * (64 + 4) * sizeof(float);
  VMOBA_CUDA_OK(allow_smem(scores_kernel<T, DH>, (int)smem));
  dim3 grid((D.S + 63) / 64, 1, D.BH);
  launch_kernel(scores_kernel<T, DH>, grid, 256, smem, st, static_cast<const T*>(q), cent, scores, D.S, D.Nb, range);
  VMOBA_LAUNCH_OK(1);
  return VMOBA_OK;
}

}  // namespace vmoba

using namespace vmoba;

static int block_scores_impl(const vmoba_shape* shape, const void* q_bm, const void* k_bm, float* centroids,
                             float* scores, float* range, int32_t* dev_status, void* ws, size_t ws_bytes, void* stream) {
  Dims D;
  int rc = make_dims(shape, &D);
  if (rc) return rc;
  if (!q_bm || !k_bm || !centroids || !scores || !dev_status || !ws) return VMOBA_ERR_ARG;
  if (!aligned16(q_bm) || !aligned16(k_bm) || !aligned16(centroids) || !aligned16(scores) || !aligned16(ws))
    return VMOBA_ERR_ARG;
  if (ws_bytes < scores_ws_bytes(D)) return VMOBA_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (D.dtype == VMOBA_BF16) {
    if (D.d == 128) return run_scores<__nv_bfloat16, 128>(D, q_bm, k_bm, centroids, scores, range, ws, dev_status, st);
    return run_scores<__nv_bfloat16, 64>(D, q_bm, k_bm, centroids, scores, range, ws, dev_status, st);
  }
  if (D.d == 128) return run_scores<float, 128>(D, q_bm, k_bm, centroids, scores, range, ws, dev_status, st);
  return run_scores<float, 64>(D, q_bm, k_bm, centroids, scores, range, ws, dev_status, st);
}

extern "C" int vmoba_block_scores(const vmoba_shape* shape, const void* q_bm, const void* k_bm,
                                  float* centroids, float* scores, int32_t* dev_status, void* ws,
                                  size_t ws_bytes, void* stream) {
  return block_scores_impl(shape, q_bm, k_bm, centroids, scores, nullptr, dev_status, ws, ws_bytes, stream);
}

extern "C" int vmoba_block_scores_range(const vmoba_shape* shape, const void* q_bm, const void* k_bm,
                                        float* centroids, float* scores, float* score_range, int32_t* dev_status,
                                        void* ws, size_t ws_bytes, void* stream) {
  if (!score_range) return VMOBA_ERR_ARG;
  return block_scores_impl(shape, q_bm, k_bm, centroids, scores, score_range, dev_status, ws, ws_bytes, stream);
}
