// Shared host/device helpers of the VMoBA library: derived dimensions, argument checks,
// dtype load/store, error plumbing.  Not part of the public ABI.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <utility>

#include "../../include/vmoba.h"

namespace vmoba {

struct Dims {
  int B, heads, d;
  int T, H, W, bT, bH, bW;
  int nT, nH, nW;
  int Nb;        // key blocks per head
  int sb;        // tokens per block
  int S;         // tokens per head
  int BH;        // B * heads
  int dtype;
  int es;        // element size in bytes
  int mask_words;  // ceil(Nb / 32)
  float scale;
};

// Where row (batch, head, block-major position p) of an output tensor lives.  perm == nullptr: block-major,
// row G = (batch * heads + head) * S + p at G * head_dim.  Otherwise raster order [B, S, heads, head_dim]
// through element strides: batch * sb + perm[p] * st + head * sh (the inverse of Eq. 1 folded into the
// kernel that writes the rows).
struct RowMap {
  const int* perm = nullptr;
  long long sb = 0, st = 0, sh = 0;
  int heads = 1, S = 1;
#ifdef __CUDACC__
  __device__ __forceinline__ long long off(long long G, int dh) const {
    if (!perm) return G * dh;
    long long b, hd;
    int p;
    if ((unsigned long long)G <= 0x7fffffffull) {   // the usual case: 32-bit quotients
      const unsigned g = (unsigned)G, bh = g / (unsigned)S, b32 = bh / (unsigned)heads;
      p = (int)(g - bh * (unsigned)S);
      b = b32;
      hd = bh - b32 * (unsigned)heads;
    } else {
      const long long bh = G / S;
      p = (int)(G - bh * S);
      b = bh / heads;
      hd = bh - b * heads;
    }
    return b * sb + (long long)__ldg(perm + p) * st + hd * sh;
  }
#endif
};

// Validates a shape and fills the derived sizes (Eq. 1 needs the grid divisible by the block).
inline int make_dims(const vmoba_shape* s, Dims* o) {
  if (!s) return VMOBA_ERR_ARG;
  if (s->dtype != VMOBA_F32 && s->dtype != VMOBA_BF16) return VMOBA_ERR_ARG;
  if (s->B <= 0 || s->heads <= 0 || s->T <= 0 || s->H <= 0 || s->W <= 0 || s->bT <= 0 ||
      s->bH <= 0 || s->bW <= 0)
    return VMOBA_ERR_SHAPE;
  if (s->head_dim != 64 && s->head_dim != 128) return VMOBA_ERR_SHAPE;
  if (s->T % s->bT || s->H % s->bH || s->W % s->bW) return VMOBA_ERR_SHAPE;
  if (!(s->softmax_scale >= 0.0f) || s->softmax_scale > 1e30f) return VMOBA_ERR_ARG;
  long long S = (long long)s->T * s->H * s->W;
  long long total = S * s->B * s->heads;
  if (S > (1ll << 24) || total > (1ll << 30)) return VMOBA_ERR_SHAPE;
  o->B = s->B; o->heads = s->heads; o->d = s->head_dim;
  o->T = s->T; o->H = s->H; o->W = s->W; o->bT = s->bT; o->bH = s->bH; o->bW = s->bW;
  o->nT = s->T / s->bT; o->nH = s->H / s->bH; o->nW = s->W / s->bW;
  o->Nb = o->nT * o->nH * o->nW;
  o->sb = s->bT * s->bH * s->bW;
  o->S = (int)S;
  o->BH = s->B * s->heads;
  o->dtype = s->dtype;
  o->es = s->dtype == VMOBA_BF16 ? 2 : 4;
  o->mask_words = (o->Nb + 31) / 32;
  o->scale = s->softmax_scale > 0.0f ? s->softmax_scale : 1.0f / sqrtf((float)s->head_dim);
  if ((long long)o->BH * o->Nb > (1ll << 24)) return VMOBA_ERR_SHAPE;
  return VMOBA_OK;
}

// Number of SMs of the current device, read once per device and thread (grids of the persistent kernels are
// one CTA per SM; the streaming kernels size theirs as a multiple of it).
inline int sm_count() {
  thread_local int cached_dev = -1, cached_n = 0;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (dev != cached_dev) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 1;
    cached_dev = dev; cached_n = n;
  }
  return cached_n;
}

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Lets a kernel have up to `bytes` of dynamic shared memory, ahead of every launch that needs more than 48 KB.  The limit is one
// setting per kernel and context for all threads, and a smaller one replaces a larger: every launch of a kernel gives the same number,
// whatever its shape, or one thread's small call would make another's large one fail.  It is not remembered either (57 ns of
// host time per call): a context that is new, after a reset or beside another, starts without it.
template <typename... P>
inline cudaError_t allow_smem(void (*kernel)(P...), int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
// The number for kernels whose need depends on the shape: what a CTA may have (227 KB) less room for static shared memory.
constexpr int kSmemMost = 222 * 1024;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// The debug build (-DVMOBA_DEBUG, lib/libvmoba_debug.so) stands in for a memory checker: every index read from a
// work list is range-checked before it is used (a violation records VMOBA_ERR_BOUNDS in the status word and the
// access goes to element 0 instead: no trap, the kernel carries on), and every slice of a workspace is followed by
// a 256-byte guard zone that is filled with a pattern before the stage's kernels run and verified after them.
#ifdef VMOBA_DEBUG
constexpr size_t kGuardBytes = 256;
#else
constexpr size_t kGuardBytes = 0;
#endif
constexpr uint32_t kGuardWord = 0xC0FFEE5Au;
struct Guards {
  char* base = nullptr;
  size_t off[16] = {};
  int n = 0;
};

// Carves 256-byte aligned slices out of a caller-provided workspace.
struct Carver {
  char* base;
  size_t off = 0;
  Guards guards;
  explicit Carver(void* p) : base(static_cast<char*>(p)) { guards.base = base; }
  template <typename T>
  T* take(size_t n) {
    off = align_up(off, 256);
    T* r = reinterpret_cast<T*>(base ? base + off : nullptr);
    off += n * sizeof(T);
    if (kGuardBytes) {
      off = align_up(off, 256);
      if (guards.n < 16) guards.off[guards.n++] = off;
      off += kGuardBytes;
    }
    return r;
  }
  size_t total() const { return align_up(off, 256); }
};

#define VMOBA_CUDA_OK(expr)                      \
  do {                                           \
    cudaError_t e__ = (expr);                    \
    if (e__ != cudaSuccess) return VMOBA_ERR_CUDA; \
  } while (0)

// Number of kernels this library has launched since it was loaded (reported by
// vmoba_kernel_launches(); benchmarks use it to show that the CUDA path did the work).
inline std::atomic<unsigned long long> g_kernel_launches{0};
inline void count_launches(int n) { g_kernel_launches.fetch_add((unsigned long long)n, std::memory_order_relaxed); }

// Checks the launches issued since the last check; n = how many kernels those were.
#define VMOBA_LAUNCH_OK(n)                                  \
  do {                                                      \
    if (cudaPeekAtLastError() != cudaSuccess) {             \
      cudaGetLastError();                                   \
      return VMOBA_ERR_CUDA;                                \
    }                                                       \
    ::vmoba::count_launches(n);                             \
  } while (0)

// Every kernel of a call begins with grid_begin() and is launched by launch_kernel(), `early` or not (the guard kernels of the
// range-checked build, where nothing is early, and the diagnostics' own kernel do neither).  An early launch does
// not wait for the end of the kernel before it in the stream: its CTAs are set up while the other still runs, stop in
// grid_begin() until that one has completed and its writes are visible, and then allow the same for the next.  A call is a
// chain of a dozen kernels or more (12 to 21 in bf16 with the backward), many of a few microseconds, and each early launch
// is worth 1.5 .. 3 us (forward of 33K tokens,
// 12 heads: 659 -> 624 us; forward and backward of 1.9K tokens: 204 -> 171 us).
//
// Not early: a long kernel that lives by many loads in flight, after one with another shape.  CTAs that move in beside the
// running kernel find the SM's shared memory / L1 split as that one has it, and keep it; and the SMs that run dry first take
// more than their share of them.  Measured, early against not (33K tokens, 3D blocks): merge pass 1391 / 838 us, row-dot pass
// 94 / 80 us, backward 494 / 433 us, first histogram 111 / 101 us.  Such kernels are early only where they are short themselves:
// early_rows().
template <typename... P, typename... A>
inline void launch_kernel(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
#ifdef VMOBA_DEBUG
  early = false;      // one after the other: what a test compares the library with
#endif
  cfg.numAttrs = early ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);      // (VMOBA_LAUNCH_OK looks at the error)
}
template <typename... P, typename... A>
inline void launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  launch_kernel(true, kernel, grid, block, smem, st, std::forward<A>(args)...);
}
// In clusters of `cluster` consecutive CTAs.
template <typename... P, typename... A>
inline void launch_cluster(bool early, int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cluster;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
#ifdef VMOBA_DEBUG
  early = false;
#endif
  cfg.numAttrs = early ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// One tensor of at most 16 MB: a pass over a few of them takes about ten microseconds, of which an early launch saves two.
inline bool early_rows(const Dims& D) { return (long long)D.BH * D.S * D.d * D.es <= (16ll << 20); }

// ---------------------------------------------------------------- device helpers
// Always true.  The value is opaque to the compiler and the kernel's body hangs on it (`if (!grid_begin()) return;`), so that no
// load, not even one through a const __restrict__ pointer, is moved ahead of the wait.
__device__ __forceinline__ bool grid_begin() {
  int go;
  asm volatile("griddepcontrol.wait;\n\tmov.b32 %0, 1;" : "=r"(go) :: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  return go != 0;
}

__device__ __forceinline__ void set_status(int32_t* st, int code) {
  if (st) atomicCAS(st, 0, code);
}

// An index read from a work list, about to address one of n elements.
__device__ __forceinline__ int checked_index(int v, int n, int32_t* st) {
#ifdef VMOBA_DEBUG
  if ((unsigned)v >= (unsigned)n) {
    set_status(st, VMOBA_ERR_BOUNDS);
    return 0;
  }
#endif
  return v;
}

#ifdef VMOBA_DEBUG
static __global__ void guard_arm_kernel(Guards g) {
  reinterpret_cast<uint32_t*>(g.base + g.off[blockIdx.x])[threadIdx.x] = kGuardWord;
}
static __global__ void guard_check_kernel(Guards g, int32_t* status) {
  if (reinterpret_cast<const uint32_t*>(g.base + g.off[blockIdx.x])[threadIdx.x] != kGuardWord)
    set_status(status, VMOBA_ERR_BOUNDS);
}
#define VMOBA_GUARDS_ARM(g, st) \
  do { if ((g).n && (g).base) guard_arm_kernel<<<(g).n, (int)(kGuardBytes / 4), 0, st>>>(g); } while (0)
#define VMOBA_GUARDS_CHECK(g, status, st) \
  do { if ((g).n && (g).base) guard_check_kernel<<<(g).n, (int)(kGuardBytes / 4), 0, st>>>(g, status); } while (0)
#else
#define VMOBA_GUARDS_ARM(g, st) do { } while (0)
#define VMOBA_GUARDS_CHECK(g, status, st) do { } while (0)
#endif

template <typename T>
__device__ __forceinline__ float to_f32(T x);
template <>
__device__ __forceinline__ float to_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 x) { return __bfloat162float(x); }

template <typename T>
__device__ __forceinline__ T from_f32(float x);
template <>
__device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <>
__device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Load 4 consecutive elements as floats (p must be 4-element aligned).
__device__ __forceinline__ float4 load4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16* p) {
  uint2 u = *reinterpret_cast<const uint2*>(p);
  float4 r;
  r.x = __uint_as_float(u.x << 16);
  r.y = __uint_as_float(u.x & 0xffff0000u);
  r.z = __uint_as_float(u.y << 16);
  r.w = __uint_as_float(u.y & 0xffff0000u);
  return r;
}
__device__ __forceinline__ void store4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void store4(__nv_bfloat16* p, float4 v) {
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
  __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
}

// Store 4 values and, for bf16 with a residual buffer, the rounding residual bf16(v - bf16(v)).
__device__ __forceinline__ void store4_resid(float* p, float* /*resid*/, float4 v) { store4(p, v); }
__device__ __forceinline__ void store4_resid(__nv_bfloat16* p, __nv_bfloat16* resid, float4 v) {
  // the rounded values are rebuilt from the packed words in registers (no read-back of the row just stored)
  __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y);
  __nv_bfloat162 b = __floats2bfloat162_rn(v.z, v.w);
  uint2 u;
  u.x = *reinterpret_cast<uint32_t*>(&a);
  u.y = *reinterpret_cast<uint32_t*>(&b);
  *reinterpret_cast<uint2*>(p) = u;
  if (resid)
    store4(resid, make_float4(v.x - __uint_as_float(u.x << 16), v.y - __uint_as_float(u.x & 0xffff0000u),
                              v.z - __uint_as_float(u.y << 16), v.w - __uint_as_float(u.y & 0xffff0000u)));
}

// Atomic minimum / maximum of fp32 values in global memory (the integer order of the bit patterns agrees with
// the float order for non-negative values and is reversed for negative ones).  The word starts at +inf / -inf.
__device__ __forceinline__ void atomic_min_f32(float* addr, float v) {
  if (!(v < 0.f)) atomicMin(reinterpret_cast<int*>(addr), __float_as_int(v));
  else atomicMax(reinterpret_cast<unsigned int*>(addr), __float_as_uint(v));
}
__device__ __forceinline__ void atomic_max_f32(float* addr, float v) {
  if (!(v < 0.f)) atomicMax(reinterpret_cast<int*>(addr), __float_as_int(v));
  else atomicMin(reinterpret_cast<unsigned int*>(addr), __float_as_uint(v));
}

// Order-preserving map from fp32 to uint32 (larger float <-> larger key).
__device__ __forceinline__ uint32_t float_key(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  uint32_t u = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
  return __uint_as_float(u);
}

// Single-CTA exclusive scan of in(0..n-1) (64-bit running total, outputs clamped to int32);
// out[n] receives the total.  Must be called by every thread of the CTA.  A thread takes E consecutive elements per trip;
// a trip is a chain of a load, two scans and four barriers.
template <int E, typename In>
__device__ __forceinline__ void block_exclusive_scan_by(In in, int* __restrict__ out, long long n, long long* total_out) {
  __shared__ long long s_warp[32];
  __shared__ long long s_carry;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  __syncthreads();
  if (t == 0) s_carry = 0;
  __syncthreads();
  for (long long base = 0; base < n; base += (long long)blockDim.x * E) {
    const long long i0 = base + (long long)t * E;
    long long x[E], v = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = i0 + e < n ? (long long)in(i0 + e) : 0;
#pragma unroll
    for (int e = 0; e < E; ++e) v += x[e];
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      long long x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      long long x = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0;
      long long xi = x;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        long long y = __shfl_up_sync(0xffffffffu, xi, o);
        if (lane >= o) xi += y;
      }
      s_warp[lane] = xi - x;
    }
    __syncthreads();
    long long excl = s_carry + s_warp[warp] + inc - v;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (i0 + e < n) out[i0 + e] = (int)min(excl, (long long)INT32_MAX);
      excl += x[e];
    }
    __syncthreads();
    if (t == (int)blockDim.x - 1) s_carry = excl;
    __syncthreads();
  }
  if (t == 0) {
    out[n] = (int)min(s_carry, (long long)INT32_MAX);
    *total_out = s_carry;
  }
  __syncthreads();
}

// Eight elements per thread where one each would take more than two trips (scans of 1,680 and 768 elements: 5.0 us with
// eight, 5.5 with one; 3,360 and 1,536: 6.7 and 8.2; a single one of 96: 3.7 and 2.3, for the longer code).
template <typename In>
__device__ __forceinline__ void block_exclusive_scan(In in, int* __restrict__ out, long long n, long long* total_out) {
  if (n <= 2 * (long long)blockDim.x) block_exclusive_scan_by<1>(in, out, n, total_out);
  else block_exclusive_scan_by<8>(in, out, n, total_out);
}

// Centroids as three bf16 numbers each, whose sum they are (scores_tc.cu): parts[part][head][Nb_pad][head_dim], pad rows zero.
struct CentroidParts {
  __nv_bfloat16* parts = nullptr;
  int Nb_pad = 0;
  long long n = 0;        // elements of one part
};

// Device counters set through vmoba_debug_wait_profile (null when diagnostics are off).
unsigned long long* debug_wait_profile();

}  // namespace vmoba
