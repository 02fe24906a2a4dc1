// Shared host/device helpers of the bsp library (status handling, bf16 access, small reductions).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "bsp.h"

namespace bsp {

// Last CUDA error seen by this host thread inside the library.
int& last_cuda_error_ref();

// (The runtime keeps the error of a failed call until it is asked for it: left there, the check behind the next plain
// launch would report it again.)
inline int cuda_fail(cudaError_t e) {
  cudaGetLastError();
  last_cuda_error_ref() = static_cast<int>(e);
  return BSP_ERR_CUDA;
}

#define BSP_CUDA_TRY(expr)                                  \
  do {                                                      \
    cudaError_t _e = (expr);                                \
    if (_e != cudaSuccess) return ::bsp::cuda_fail(_e);     \
  } while (0)

// Kernel launches report configuration errors through cudaGetLastError.
#define BSP_LAUNCH_CHECK()                                  \
  do {                                                      \
    cudaError_t _e = cudaGetLastError();                    \
    if (_e != cudaSuccess) return ::bsp::cuda_fail(_e);     \
  } while (0)

inline bool aligned_to(const void* p, size_t a) {
  return (reinterpret_cast<uintptr_t>(p) % a) == 0;
}
inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// Number of blocks / groups per block for a geometry; returns false when `block` does not divide.
inline bool geometry(int rows, int cols, int block, int orient, int* n_blocks, int* n_groups) {
  if (orient == BSP_ORIENT_C) {
    if (rows % block) return false;
    *n_blocks = rows / block;
    *n_groups = cols;
  } else {
    if (cols % block) return false;
    *n_blocks = cols / block;
    *n_groups = rows;
  }
  return true;
}

// Common argument screening for calls that take (W, rows, cols, ldw, block, orient).
inline int check_matrix_args(const void* W, int rows, int cols, int ldw, int block, int orient) {
  if (W == nullptr || rows <= 0 || cols <= 0 || block <= 0) return BSP_ERR_ARG;
  if (orient != BSP_ORIENT_C && orient != BSP_ORIENT_R) return BSP_ERR_ARG;
  if (!aligned_to(W, 2)) return BSP_ERR_ARG;
  if (ldw < cols) return BSP_ERR_SHAPE;
  int nb, ng;
  if (!geometry(rows, cols, block, orient, &nb, &ng)) return BSP_ERR_SHAPE;
  return BSP_OK;
}

// Workspace of the pack calls: [per-block counts][per-group flags][per-group float32 S], each
// region 256-byte aligned.  (The fused call keeps per-block penalty partials in the S region.)
struct WsLayout {
  size_t counts_off, keep_off, sumsq_off, total;
};
inline WsLayout ws_layout(int n_blocks, int n_groups) {
  WsLayout L;
  const size_t groups = static_cast<size_t>(n_blocks) * n_groups;
  L.counts_off = 0;
  L.keep_off = round_up(sizeof(int32_t) * (static_cast<size_t>(n_blocks) + 1), 256);
  L.sumsq_off = L.keep_off + round_up(groups, 256);
  L.total = L.sumsq_off + round_up(groups * sizeof(float), 256);
  return L;
}


// One matrix of a launch of the vectorised orientation-C kernels (bsp_fused.cu).  Null output
// pointers switch the matching work off.
struct FusedJob {
  const uint16_t* W;
  int rows, cols, ldw, n_blocks;
  float threshold;
  const float* threshold_dev;
  float* norms;
  const float* gamma_in;
  float* gamma_out;
  double* penalty;             // job total (written by stage 2 from `partial`, or by atomics in stage 1)
  double* partial;             // per-block penalty partial sums, or null: stage 1 adds into *penalty
  uint8_t* flags;              // per-group keep flags (null: stage 1 skips the keep decision)
  int32_t* counts;             // per-block kept counts
  int32_t* blk_ptr;
  int32_t* idx;
  uint16_t* vals;
  int64_t* kept_weights;
  uint16_t* plan;
};
constexpr int kFusedMaxJobs = 96;     // per launch; the job table travels as a kernel parameter (about 15 KB)
constexpr int kFusedMaxCols = 4096;     // stage 2 keeps 12 bytes of shared memory per column
constexpr int kFusedMaxBlocks = 1024;   // stage 2 sums the counts before its block directly
// Stage 1: sums of squares -> norms / gamma / penalty and/or keep flags + counts, one pass over W.
int fused_stage1(const FusedJob* jobs, int n_jobs, int block, float eps, int squared, cudaStream_t s);
// Stage 2: blk_ptr, index lists, packed tiles, penalty totals, optional execution layout.
int fused_stage2(const FusedJob* jobs, int n_jobs, int block, cudaStream_t s);
// Streaming one-pass kernel for batches of any size (bsp_fused_stream.cu); *used = false means nothing was launched.
int fused_stream(const FusedJob* jobs, int n_jobs, int block, float eps, int squared, int32_t* const* part_counts,
                 double* const* part_partial, cudaStream_t s, bool* used);
// Whether a matrix can go through the vectorised kernels.
inline bool fused_shape_ok(const void* W, int rows, int cols, int ldw, int block) {
  return cols % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16) && cols <= kFusedMaxCols && rows / block <= kFusedMaxBlocks;
}

// Rows of one trip to memory (see sumsq8) for a launch of `ctas` CTAs that sum row-blocks of `block` rows, of which `per_sm16`
// and `per_sm32` fit an SM with 16 and 32 rows in flight.  The longest trip while all CTAs run at once, with an eighth to
// spare for those of the launch before; shorter ones where that leaves CTAs waiting for a seat, or where there are no rows
// for it.  Norms, trips of 16 or 32 for all blocks / by this rule: 8192 x 3072 in single rows 77.7 / 42.2 us, in 8-row blocks
// 17.6 / 14.2, in 32-row blocks 13.8 / 11.1; 768 x 3072 in 2-row blocks 5.2 / 3.6; percentile of 12 matrices of 512 x 512 in
// 8-row blocks 11.2 / 9.8, of 40 of 512 x 64 in 32-row blocks 10.6 / 8.4.
inline int rows_per_trip(int block, long long ctas, int per_sm16, int per_sm32, int sms) {
  if (block < 8) return 4;
  if (block >= 32 && ctas <= static_cast<long long>(sms) * per_sm32 * 7 / 8) return 32;
  return ctas <= static_cast<long long>(sms) * per_sm16 * 7 / 8 ? 16 : 8;
}

// Widest vector load (in elements: 8, 4 or 1) that reads whole orientation-R groups: rows of `block`
// contiguous elements starting at multiples of `block` in a row of leading dimension ldw.
inline int contig_vec(const void* W, int ldw, int block) {
  if (block % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16)) return 8;
  if (block % 4 == 0 && ldw % 4 == 0 && aligned_to(W, 8)) return 4;
  return 1;
}

// Set-up that a kernel needs once on every device before its first launch.  First calls may come from several host
// threads at once (the binding runs them without the interpreter lock); doing it twice does no harm.
struct OncePerDevice {
  std::atomic<bool> done[64];
};
template <class K>
inline int allow_dynamic_smem(OncePerDevice& once, K* kernel, int bytes) {
  int device = 0;
  BSP_CUDA_TRY(cudaGetDevice(&device));
  if (device < 0 || device >= 64) return BSP_ERR_CUDA;
  if (!once.done[device].load(std::memory_order_acquire)) {
    BSP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    once.done[device].store(true, std::memory_order_release);
  }
  return BSP_OK;
}
inline int sm_count(int* sms) {
  int dev = 0;
  BSP_CUDA_TRY(cudaGetDevice(&dev));
  BSP_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return BSP_OK;
}
#define BSP_TRY(expr)                \
  do {                               \
    const int _st = (expr);          \
    if (_st != BSP_OK) return _st;   \
  } while (0)

#ifdef __CUDACC__
// Launch with programmatic stream serialization: the grid may take its seats while the previous kernel of
// the stream drains; it saves about 1 us between two of this library's short kernels.
// The rule that keeps the order of the stream: a thread signals (pdl_launch_dependents) only after its own
// pdl_wait.  A grid starts once every CTA of its direct predecessor has signalled or ended, so a grid that has
// started knows that everything BEFORE that predecessor is complete, though not the predecessor itself; and once
// its own pdl_wait returns, that too.  Hence global memory is touched after pdl_wait, except for
//   - data older than the direct predecessor, where the library itself launched that predecessor: W and the sums
//     behind the percentile's clearing kernel (bsp_select.cu), W in the second packing stage (bsp_fused.cu);
//   - the weights of a plan that the caller vouches for (BSP_LINEAR_PLAN_STABLE): the weight warp of
//     linear_tc_kernel, gemm_pair_kernel and gemm_split_kernel, which does not wait and therefore does not signal either.
// A kernel that allocates tensor memory signals behind its allocation: a dependent CTA that took the memory first would wait for
// this grid, and this grid for the memory.
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Only after the same thread's pdl_wait (see launch_pdl).
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Fetches into L2 of what a CTA will read once pdl_wait returns.  They change nothing but what L2 holds, which is
// coherent, so they may go out before the wait, while the previous kernel of the stream is still running: short
// kernels (a 768 x 768 matrix re-packed in 3 us) leave HBM idle meanwhile, and the next kernel's first wave of CTAs
// then finds its operands in L2.  Retraining 12 BERT-base layers (48 x Adam step, re-pack): 621 -> 608 us; an iteration
// of reweighted training on a 1024-wide layer: 113 -> 107 us.
__device__ __forceinline__ void prefetch_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
// `bytes` a multiple of 16, p 16-byte aligned.
__device__ __forceinline__ void prefetch_bytes(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// A load of what an earlier launch may have written, for kernels that are resident while that launch still runs (every
// kernel that calls pdl_wait): an ordinary coherent load, which the wait's memory clobber keeps behind it.  Such data
// does change while the kernel lives, so the read-only path (__ldg, or const __restrict__ parameters, which a compiler
// may send there and may read ahead of the wait) is not defined for it.  Without __restrict__ a load does not move
// ahead of a store either: loops that copy ask for several elements before they store the first.
template <class T>
__device__ __forceinline__ T ld_global(const T* p) {
  return *p;
}

// The type that moves N 16-bit elements at once.
template <int N>
struct VectorOf {
  using type = uint16_t;
};
template <>
struct VectorOf<4> {
  using type = uint2;
};
template <>
struct VectorOf<8> {
  using type = uint4;
};
template <int N>
using vector_of = typename VectorOf<N>::type;

__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) {
  return __uint_as_float(static_cast<uint32_t>(b) << 16);
}

// Sum of squares of one group in float32, elements taken in increasing index order starting
// from +0.  The square of a bf16 value is exact in float32, so the fused multiply-add rounds
// exactly once per element, the same as a separate multiply and add would.
__device__ __forceinline__ float group_sumsq_strided(const uint16_t* p, int n, size_t stride) {
  float acc = 0.0f;
  for (int e = 0; e < n; ++e) {
    const float w = bf16_bits_to_float(ld_global(p + static_cast<size_t>(e) * stride));
    acc = __fmaf_rn(w, w, acc);
  }
  return acc;
}
// The same with eight loads in flight, for kernels that do little else.
__device__ __forceinline__ float group_sumsq_strided8(const uint16_t* p, int n, size_t stride) {
  float acc = 0.0f;
  int e = 0;
  for (; e + 8 <= n; e += 8, p += 8 * stride) {
    uint16_t v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = ld_global(p + u * stride);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float w = bf16_bits_to_float(v[u]);
      acc = __fmaf_rn(w, w, acc);
    }
  }
  if (e + 4 <= n) {
    uint16_t v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = ld_global(p + u * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float w = bf16_bits_to_float(v[u]);
      acc = __fmaf_rn(w, w, acc);
    }
    e += 4;
    p += 4 * stride;
  }
  for (; e < n; ++e, p += stride) {
    const float w = bf16_bits_to_float(ld_global(p));
    acc = __fmaf_rn(w, w, acc);
  }
  return acc;
}

// The same for a group of contiguous elements (orientation R), by vectors of `vec` elements (contig_vec).
__device__ __forceinline__ float group_sumsq_contig(const uint16_t* p, int n, int vec) {
  float acc = 0.0f;
  if (vec == 8) {
#pragma unroll 4
    for (int e = 0; e < n; e += 8) {
      const uint4 v = ld_global(reinterpret_cast<const uint4*>(p + e));
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xffff0000u);
        acc = __fmaf_rn(hi, hi, __fmaf_rn(lo, lo, acc));
      }
    }
  } else if (vec == 4) {
#pragma unroll 4
    for (int e = 0; e < n; e += 4) {
      const uint2 v = ld_global(reinterpret_cast<const uint2*>(p + e));
      const uint32_t w[2] = {v.x, v.y};
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float lo = __uint_as_float(w[i] << 16), hi = __uint_as_float(w[i] & 0xffff0000u);
        acc = __fmaf_rn(hi, hi, __fmaf_rn(lo, lo, acc));
      }
    }
  } else {
    acc = group_sumsq_strided(p, n, 1);
  }
  return acc;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Float32 sums of squares of 8 adjacent columns over the d rows of a row-block: eight independent
// sequential chains, each the defined decision quantity of its group.  Two neighbouring chains share a packed float32 FMA
// (fma.rn.f32x2: two independent correctly rounded FMAs, the same bits as two of them in half the instructions).
struct SumSq8 {
  unsigned long long pair[4] = {0ull, 0ull, 0ull, 0ull};
  __device__ __forceinline__ void add(const uint4& v) {
    const uint32_t w32[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned long long x;
      asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(w32[i] << 16), "r"(w32[i] & 0xffff0000u));
      asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(pair[i]) : "l"(x));
    }
  }
  __device__ __forceinline__ void get(float (&acc)[8]) const {
#pragma unroll
    for (int i = 0; i < 4; ++i) asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[2 * i]), "=f"(acc[2 * i + 1]) : "l"(pair[i]));
  }
};
// The same without register pairs, for kernels whose threads have 32 to 40 registers (the keep-count select would spill).
struct SumSq8Few {
  float acc8[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  __device__ __forceinline__ void add(const uint4& v) {
    const uint32_t w32[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float lo = __uint_as_float(w32[i] << 16), hi = __uint_as_float(w32[i] & 0xffff0000u);
      acc8[2 * i] = __fmaf_rn(lo, lo, acc8[2 * i]);
      acc8[2 * i + 1] = __fmaf_rn(hi, hi, acc8[2 * i + 1]);
    }
  }
  __device__ __forceinline__ void get(float (&acc)[8]) const {
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] = acc8[i];
  }
};
template <bool kTogether>
struct SumSq8Of {
  using type = SumSq8;
};
template <>
struct SumSq8Of<false> {
  using type = SumSq8Few;
};
// kTogether: every load is issued before the first is used.  Left to itself the compiler interleaves loads and arithmetic to
// save registers (54 instead of 90 here), which makes several trips to memory of one; a barrier of the warp keeps the loads
// ahead of it (each thread names the threads that it is converged with, and they all come to it).  Norms of the matrices of a
// 1024-wide layer, in an iteration of reweighted training: 24.5 -> 20.8 us, the iteration 106.2 -> 102.5.
// kPast: the rows are not kept in L1.
template <int ROWS, bool kTogether, bool kPast>
__device__ __forceinline__ void sumsq8_rows(const uint16_t* p, int ldw, typename SumSq8Of<kTogether>::type& acc) {
  uint4 v[ROWS];
#pragma unroll
  for (int u = 0; u < ROWS; ++u) {
    const uint4* src = reinterpret_cast<const uint4*>(p + static_cast<size_t>(u) * ldw);
    if (kPast) asm volatile("ld.global.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v[u].x), "=r"(v[u].y), "=r"(v[u].z), "=r"(v[u].w) : "l"(src) : "memory");
    else v[u] = ld_global(src);
  }
  if (kTogether && ROWS > 1) __syncwarp(__activemask());
#pragma unroll
  for (int u = 0; u < ROWS; ++u) acc.add(v[u]);     // rows in increasing order: the chains stay sequential
}
// kTrip: rows of one trip to memory, all of them in flight.  A row takes four registers, so a longer trip leaves fewer CTAs on
// an SM: 4 rows 56 registers in the norms' kernel, 8 rows 64, 16 rows 90, 32 rows 156 (see rows_per_trip).  0: as the compiler
// likes, for kernels of few registers.
template <int kTrip, bool kPast = false>
__device__ __forceinline__ void sumsq8(const uint16_t* p, int d, int ldw, float (&acc)[8]) {
  constexpr bool kTogether = kTrip > 0;
  constexpr int kMost = kTogether ? kTrip : 16;
  typename SumSq8Of<kTogether>::type sums;
  int r = 0;
  if (kMost >= 32)
    for (; r + 32 <= d; r += 32) sumsq8_rows<32, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums);   // 512 bytes in flight
  if (kMost >= 16)
    for (; r + 16 <= d; r += 16) sumsq8_rows<16, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums);   // 256 bytes in flight
  // (12 rows in one trip, not 8 and 4: pruning 768 x 768 in 12-row blocks 20.5 -> 20.1 us; 9 to 15 as far as they exist took 30
  // registers more and 0.4 us of a layer's milestone)
  if (kTogether && kMost == 16 && r + 12 <= d) { sumsq8_rows<12, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums); r += 12; }
  if (kMost == 16 && r + 8 <= d) { sumsq8_rows<8, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums); r += 8; }
  if (kMost == 8)
    for (; r + 8 <= d; r += 8) sumsq8_rows<8, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums);
  for (; r + 4 <= d; r += 4) sumsq8_rows<4, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums);
  for (; r < d; ++r) sumsq8_rows<1, kTogether, kPast>(p + static_cast<size_t>(r) * ldw, ldw, sums);
  sums.get(acc);
}

// Block-wide exclusive prefix sum of one int per thread (blockDim.x a multiple of 32, <= 1024).
__device__ __forceinline__ int block_exclusive_scan(int v, int* s_warp, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    int w = lane < n_warps ? s_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += up;
    }
    s_warp[lane] = w;  // inclusive totals of warps
  }
  __syncthreads();
  const int before = warp ? s_warp[warp - 1] : 0;
  *total = s_warp[n_warps - 1];
  __syncthreads();  // s_warp may be reused by the caller's next round
  return before + incl - v;
}

// Norm and reciprocal of the reported (not the deciding) quantities: the hardware's approximate square
// root and reciprocal, each within about one unit in the last place of float32, far inside the 1e-5
// these outputs are held to, at a sixth of the instructions of the correctly rounded forms.  Every
// kernel that writes norms or gamma goes through these two, so all of them give the same bits.
__device__ __forceinline__ float norm_from_sumsq(float S) {
  float n;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(n) : "f"(S));
  return n;
}
__device__ __forceinline__ float reciprocal(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

struct NormOut {
  float* norms;
  const float* gamma_in;
  float* gamma_out;
  double* penalty;
  float eps;
  int squared;  // 0: gamma = 1/(n+eps), term gamma*n ; 1: alpha = 1/(S+eps), term alpha*S
};

// Finishes one group from its float32 sum of squares; returns the group's penalty term.
__device__ __forceinline__ double finish_group(const NormOut& o, size_t g, float S) {
  const float n = norm_from_sumsq(S);
  const float base = o.squared ? S : n;
  const float fresh = reciprocal(base + o.eps);
  if (o.norms) o.norms[g] = n;
  if (o.gamma_out) o.gamma_out[g] = fresh;
  const float weight = o.gamma_in ? o.gamma_in[g] : fresh;
  return static_cast<double>(weight) * static_cast<double>(base);
}

#endif  // __CUDACC__

}  // namespace bsp
