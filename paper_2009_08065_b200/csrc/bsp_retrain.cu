// Algorithm 2's retraining loop on the device: "update W ... using Adam", then "W = W * Mask", in
// one pass (bsp_masked_adam_step), and the refresh of the packed values of Section 3.1's storage
// under the fixed kept sets (bsp_repack_values); and the mask loop itself (bsp_dense_mask).
//
// Adam is taken as published (Kingma & Ba 2015, with bias correction); the paper gives no
// hyper-parameters beyond the learning rate, so they are the caller's.  The weights that the
// optimiser owns are float32 (a bf16 weight of size 0.02 cannot absorb a step of 3e-5); the bf16
// copy that the linear layer reads, already multiplied by the mask, is written in the same pass:
// it IS the zero-expanded execution layout of bsp_linear_planned.
// HBM-bound, one thread per 4 adjacent weights: 16 bytes of gradient, weight and both moments in,
// weight and moments out plus the bf16 copy: 16 + 12 + 2 = 30 bytes per weight.
#include <math.h>

#include "bsp_common.cuh"

namespace bsp {
namespace {

struct AdamArgs {
  float* W;
  const float* G;
  float* M;
  float* V;
  int rows, cols, ldw, ldg;
  const uint8_t* keep;       // per-group flags, or null (no mask)
  int block, orient;
  int keep_vec;              // keep is 4-byte aligned
  float lr, beta1, beta2, eps, decay;
  float inv_c1, inv_c2;      // 1 / (1 - beta^step)
  uint16_t* Wb;              // bf16 copy, or null
  int ldb;
  unsigned first_wave;       // CTAs that are resident at once
};

// One 4-weight item; `keep` decides per weight.
__device__ __forceinline__ void adam_item(const AdamArgs& A, int r, int c) {
  const size_t iw = static_cast<size_t>(r) * A.ldw + c, ig = static_cast<size_t>(r) * A.ldg + c;
  const float4 w4 = *reinterpret_cast<const float4*>(A.W + iw);
  const float4 g4 = ld_global(reinterpret_cast<const float4*>(A.G + ig));
  const float4 m4 = *reinterpret_cast<const float4*>(A.M + iw);
  const float4 v4 = *reinterpret_cast<const float4*>(A.V + iw);
  float w[4] = {w4.x, w4.y, w4.z, w4.w};
  const float g[4] = {g4.x, g4.y, g4.z, g4.w};
  float m[4] = {m4.x, m4.y, m4.z, m4.w};
  float v[4] = {v4.x, v4.y, v4.z, v4.w};
  uint32_t keep[4] = {1u, 1u, 1u, 1u};
  if (A.keep != nullptr) {
    if (A.orient == BSP_ORIENT_C) {
      const uint8_t* f = A.keep + static_cast<size_t>(r / A.block) * A.cols + c;
      if (A.keep_vec) {
        const uint32_t f4 = ld_global(reinterpret_cast<const uint32_t*>(f));
#pragma unroll
        for (int i = 0; i < 4; ++i) keep[i] = (f4 >> (8 * i)) & 0xffu;
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) keep[i] = f[i];
      }
    } else {
      const uint8_t* f = A.keep + static_cast<size_t>(r) * (A.cols / A.block);
#pragma unroll
      for (int i = 0; i < 4; ++i) keep[i] = f[(c + i) / A.block];
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = __fmaf_rn(A.beta1, m[i], (1.0f - A.beta1) * g[i]);
    v[i] = __fmaf_rn(A.beta2, v[i], (1.0f - A.beta2) * g[i] * g[i]);
    const float mhat = m[i] * A.inv_c1, vhat = v[i] * A.inv_c2;
    const float upd = __fdiv_rn(mhat, __fsqrt_rn(vhat) + A.eps) + A.decay * w[i];
    w[i] = keep[i] ? __fmaf_rn(-A.lr, upd, w[i]) : 0.0f;
  }
  *reinterpret_cast<float4*>(A.W + iw) = make_float4(w[0], w[1], w[2], w[3]);
  *reinterpret_cast<float4*>(A.M + iw) = make_float4(m[0], m[1], m[2], m[3]);
  *reinterpret_cast<float4*>(A.V + iw) = make_float4(v[0], v[1], v[2], v[3]);
  if (A.Wb != nullptr) {
    uint32_t lo, hi;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(w[1]), "f"(w[0]));
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(w[3]), "f"(w[2]));
    *reinterpret_cast<uint2*>(A.Wb + static_cast<size_t>(r) * A.ldb + c) = make_uint2(lo, hi);
  }
}

// One item per thread.  (A single wave of CTAs that loop over the items was 8 % slower; 32-bit item numbers where
// they suffice: the 64-bit division to row and column is a third of the kernel's instructions.)
template <typename Index>
__global__ void __launch_bounds__(256)
masked_adam_kernel(AdamArgs A) {
  const Index quads = static_cast<Index>(A.cols >> 2);
  const Index item = static_cast<Index>(blockIdx.x) * 256u + threadIdx.x;
  // the CTAs that can be waiting for the previous kernel: their own lines (eight items each) and those of the CTAs
  // that will take their places
  if (blockIdx.x < A.first_wave && (threadIdx.x & 7) == 0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const Index it = item + static_cast<Index>(u) * A.first_wave * 256u;
      if (it < static_cast<Index>(A.rows) * quads) {
        const Index r = it / quads;
        const size_t c = static_cast<size_t>(it - r * quads) << 2;
        const size_t iw = static_cast<size_t>(r) * A.ldw + c;
        prefetch_line(A.W + iw);
        prefetch_line(A.G + static_cast<size_t>(r) * A.ldg + c);
        prefetch_line(A.M + iw);
        prefetch_line(A.V + iw);
      }
    }
  }
  pdl_wait();
  pdl_launch_dependents();
  if (item >= static_cast<Index>(A.rows) * quads) return;
  const Index r = item / quads;
  adam_item(A, static_cast<int>(r), static_cast<int>(item - r * quads) << 2);
}

// Rows of one row-block: tile[r][p] = W[b*d + r][idx[lo + p]].  The vectorised form stages kRepackRows rows and
// the block's index list (2 bytes per entry) in shared memory, 16 bytes per load with all of a thread's loads
// in flight (at the usual rates every 32-byte sector of a row holds a kept column, so whole rows are read
// anyway), and gathers from there, two positions per 4-byte store.  HBM-bound in total, latency-bound per
// matrix: four rows per CTA, two of wide matrices of few row-blocks, and the list travels beside the rows.  12 layers of four
// matrices, on average: 5.3 us gathering from global memory, 2.9 us.
constexpr int kRepackRows = 4, kRepackThreads = 256, kRepackLoads = 6, kRepackMaxCols = 3072;
__global__ void __launch_bounds__(kRepackThreads)
repack_vec_kernel(const uint16_t* W, int cols, int ldw, int block, int rows_per, const int32_t* blk_ptr,
                  const int32_t* idx, uint16_t* vals) {
  extern __shared__ __align__(16) uint16_t s_rows[];             // [rows_per][cols], then the list [cols]
  const int b = blockIdx.x, r_lo = blockIdx.y * rows_per, n_rows = min(rows_per, block - r_lo);
  const int chunks = cols >> 3;
  uint16_t* s_list = s_rows + rows_per * cols;
  if (threadIdx.x == 0) prefetch_line(blk_ptr + b);
  if (static_cast<int>(threadIdx.x) < n_rows)
    prefetch_bytes(W + (static_cast<size_t>(b) * block + r_lo + threadIdx.x) * ldw, static_cast<uint32_t>(cols) * 2u);
  pdl_wait();
  pdl_launch_dependents();
  const int lo = ld_global(blk_ptr + b), kc = ld_global(blk_ptr + b + 1) - lo;
  int col[4];                                                    // the first of the list, in flight beside the rows
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int p = static_cast<int>(threadIdx.x) + u * kRepackThreads;
    if (p < kc) col[u] = ld_global(idx + lo + p);
  }
  const uint16_t* src = W + (static_cast<size_t>(b) * block + r_lo) * ldw;
  const int total = n_rows * chunks;
  for (int e0 = threadIdx.x; e0 < total; e0 += kRepackLoads * kRepackThreads) {
    uint4 v[kRepackLoads];
#pragma unroll
    for (int u = 0; u < kRepackLoads; ++u) {
      const int e = e0 + u * kRepackThreads, r = e / chunks;
      if (e < total) v[u] = ld_global(reinterpret_cast<const uint4*>(src + static_cast<size_t>(r) * ldw + ((e - r * chunks) << 3)));
    }
#pragma unroll
    for (int u = 0; u < kRepackLoads; ++u) {
      const int e = e0 + u * kRepackThreads;
      if (e < total) reinterpret_cast<uint4*>(s_rows)[e] = v[u];   // rows are packed: chunk e of the pass
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int p = static_cast<int>(threadIdx.x) + u * kRepackThreads;
    if (p < kc) s_list[p] = static_cast<uint16_t>(col[u]);
  }
  for (int p = threadIdx.x + 4 * kRepackThreads; p < kc; p += kRepackThreads) s_list[p] = static_cast<uint16_t>(ld_global(idx + lo + p));
  __syncthreads();
  uint16_t* tile = vals + static_cast<size_t>(block) * lo + static_cast<size_t>(r_lo) * kc;
  if ((reinterpret_cast<uintptr_t>(tile) & 3) == 0 && (kc & 1) == 0) {
    uint32_t* out = reinterpret_cast<uint32_t*>(tile);
    const int pairs = kc >> 1;
    for (int p = threadIdx.x; p < pairs; p += kRepackThreads) {
      const uint32_t cc = reinterpret_cast<const uint32_t*>(s_list)[p];
      const uint16_t *a = s_rows + (cc & 0xffffu), *c = s_rows + (cc >> 16);
#pragma unroll
      for (int r = 0; r < kRepackRows; ++r)
        if (r < n_rows) out[static_cast<size_t>(r) * pairs + p] = static_cast<uint32_t>(a[r * cols]) | (static_cast<uint32_t>(c[r * cols]) << 16);
    }
  } else {
    for (int p = threadIdx.x; p < kc; p += kRepackThreads) {
      const uint16_t* a = s_rows + s_list[p];
#pragma unroll
      for (int r = 0; r < kRepackRows; ++r)
        if (r < n_rows) tile[static_cast<size_t>(r) * kc + p] = a[r * cols];
    }
  }
}

// Any alignment or width, four positions of a row in flight per thread.
__global__ void __launch_bounds__(256)
repack_kernel(const uint16_t* W, int ldw, int block, const int32_t* blk_ptr,
              const int32_t* idx, uint16_t* vals) {
  const int b = blockIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  const int lo = blk_ptr[b], kc = blk_ptr[b + 1] - lo;
  const uint16_t* wblk = W + static_cast<size_t>(b) * block * ldw;
  uint16_t* tile = vals + static_cast<size_t>(block) * lo;
  const int r_lo = blockIdx.y * kRepackRows, r_hi = min(block, r_lo + kRepackRows);
  for (int p0 = threadIdx.x; p0 < kc; p0 += 4 * 256) {
    int col[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) col[u] = ld_global(idx + lo + min(p0 + u * 256, kc - 1));
    for (int r = r_lo; r < r_hi; ++r) {
      uint16_t v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ld_global(wblk + static_cast<size_t>(r) * ldw + col[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (p0 + u * 256 < kc) tile[static_cast<size_t>(r) * kc + p0 + u * 256] = v[u];
    }
  }
}

// Algorithm 2's mask loop: Mask_ij = 0 if W_ij == 0 else 1 (either sign of zero is zero).
__global__ void __launch_bounds__(256)
dense_mask_kernel(const uint16_t* __restrict__ W, int rows, int cols, int ldw, uint8_t* __restrict__ mask, int ldm) {
  const long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= static_cast<long long>(rows) * cols) return;
  const int r = static_cast<int>(e / cols), c = static_cast<int>(e - static_cast<long long>(r) * cols);
  mask[static_cast<size_t>(r) * ldm + c] = (W[static_cast<size_t>(r) * ldw + c] & 0x7fffu) != 0 ? 1 : 0;
}

}  // namespace
}  // namespace bsp

extern "C" int bsp_dense_mask(const void* W, int rows, int cols, int ldw, uint8_t* mask, int ldm, void* stream) {
  using namespace bsp;
  if (W == nullptr || mask == nullptr || rows <= 0 || cols <= 0) return BSP_ERR_ARG;
  if (ldw < cols || ldm < cols) return BSP_ERR_SHAPE;
  const long long elems = static_cast<long long>(rows) * cols;
  const long long blocks = (elems + 255) / 256;
  if (blocks > 0x7fffffffLL) return BSP_ERR_UNSUPPORTED;
  dense_mask_kernel<<<static_cast<unsigned>(blocks), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint16_t*>(W), rows, cols, ldw, mask, ldm);
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

extern "C" int bsp_masked_adam_step(float* W, const float* grad, float* m, float* v, int rows, int cols, int ldw,
                                    int ldg, const uint8_t* keep, int block, int orient, float lr, float beta1,
                                    float beta2, float eps, float weight_decay, int step, void* W_bf16, int ldb,
                                    void* stream) {
  using namespace bsp;
  if (W == nullptr || grad == nullptr || m == nullptr || v == nullptr) return BSP_ERR_ARG;
  if (rows <= 0 || cols <= 0 || step < 1) return BSP_ERR_ARG;
  if (!(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) || !(eps >= 0.0f) || !(lr == lr) ||
      !(weight_decay == weight_decay))
    return BSP_ERR_ARG;
  if (ldw < cols || ldg < cols || (W_bf16 != nullptr && ldb < cols)) return BSP_ERR_SHAPE;
  if (keep != nullptr) {
    if (block <= 0 || (orient != BSP_ORIENT_C && orient != BSP_ORIENT_R)) return BSP_ERR_ARG;
    int nb, ng;
    if (!geometry(rows, cols, block, orient, &nb, &ng)) return BSP_ERR_SHAPE;
  }
  if (cols % 4 || ldw % 4 || ldg % 4 || !aligned_to(W, 16) || !aligned_to(grad, 16) || !aligned_to(m, 16) ||
      !aligned_to(v, 16) || (W_bf16 != nullptr && (ldb % 4 || !aligned_to(W_bf16, 8))))
    return BSP_ERR_UNSUPPORTED;
  AdamArgs A;
  A.W = W; A.G = grad; A.M = m; A.V = v;
  A.rows = rows; A.cols = cols; A.ldw = ldw; A.ldg = ldg;
  A.keep_vec = aligned_to(keep, 4) ? 1 : 0;
  A.keep = keep; A.block = block; A.orient = orient;
  A.lr = lr; A.beta1 = beta1; A.beta2 = beta2; A.eps = eps; A.decay = weight_decay;
  // bias corrections in double on the host, rounded once
  A.inv_c1 = static_cast<float>(1.0 / (1.0 - pow(static_cast<double>(beta1), step)));
  A.inv_c2 = static_cast<float>(1.0 / (1.0 - pow(static_cast<double>(beta2), step)));
  A.Wb = static_cast<uint16_t*>(W_bf16);
  A.ldb = ldb;
  const long long items = static_cast<long long>(rows) * (cols >> 2);
  const long long blocks = (items + 255) / 256;
  if (blocks > 0x7fffffffLL) return BSP_ERR_UNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const dim3 grid(static_cast<unsigned>(blocks));
  int sms = 0;
  BSP_TRY(sm_count(&sms));
  A.first_wave = 5u * static_cast<unsigned>(sms);        // 48 registers x 256 threads: five CTAs per SM
  if (blocks * 256 < (1LL << 32)) BSP_CUDA_TRY(launch_pdl(masked_adam_kernel<unsigned>, grid, dim3(256), 0, s, A));
  else BSP_CUDA_TRY(launch_pdl(masked_adam_kernel<unsigned long long>, grid, dim3(256), 0, s, A));
  return BSP_OK;
}

extern "C" int bsp_repack_values(const void* W, int rows, int cols, int ldw, int block, const int32_t* blk_ptr,
                                 const int32_t* idx, void* vals, void* stream) {
  using namespace bsp;
  if (blk_ptr == nullptr || idx == nullptr || vals == nullptr) return BSP_ERR_ARG;
  int st = check_matrix_args(W, rows, cols, ldw, block, BSP_ORIENT_C);
  if (st != BSP_OK) return st;
  const int nb = rows / block;
  const dim3 grid(nb, (block + kRepackRows - 1) / kRepackRows);
  if (grid.y > 65535) return BSP_ERR_UNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint16_t* w = static_cast<const uint16_t*>(W);
  // Staged rows, where several CTAs fit an SM and have all of their rows.  Behind the Adam step, staged / gathered from
  // global memory: 4096 x 1024 in 16-row blocks 4.0 / 5.7 us, 768 x 3072 5.5 / 5.2, 8192 x 4096 49 / 26, 5344 x 920 in single
  // rows 11.2 / 10.2; 6042 x 2128 in pairs, by itself, 10.7 / 7.5.
  if (cols % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16) && cols <= kRepackMaxCols && block >= kRepackRows) {
    // Two rows where four of them give fewer than two CTAs per SM and two are 1536 elements (a chunk of eight for most of the
    // threads): between the Adam steps of a stack (768 x 768 and 768 x 3072 have 192 CTAs of four rows) a call is then bound by
    // a shorter chain of loads and stores.  Four rows / two, behind the Adam step: 768 x 768 in 16-row blocks 6.65 / 6.31 us,
    // 1024 x 1024 10.9 / 10.5, 992 x 2528 19.0 / 17.9; calls by themselves, one behind the other: the matrices of 12 layers of
    // 512 features 2.84 / 2.60 on average, of 768 3.03 / 2.98, but one shape again and again out of L2 768 x 768 2.1 / 2.4, 1024 x
    // 1024 2.5 / 3.0.  Single rows are no better behind Adam and cost by themselves (480 x 1920 in four, two and one 9.64 / 9.38 /
    // 9.52 and 2.38 / 2.23 / 2.75), and so do two rows of narrow matrices (12 layers of 256 features 216 -> 227);
    // 704 x 704, just below the line, would gain what 768 x 768 does (6.65 / 6.26).
    int sms = 0;
    BSP_TRY(sm_count(&sms));
    const bool two = 2 * cols >= 1536 && static_cast<long long>(nb) * ((block + kRepackRows - 1) / kRepackRows) < 2LL * sms;
    const int rows_per = two ? kRepackRows / 2 : kRepackRows;
    const dim3 pieces(nb, (block + rows_per - 1) / rows_per);
    BSP_CUDA_TRY(launch_pdl(repack_vec_kernel, pieces, dim3(kRepackThreads), static_cast<size_t>(cols) * (rows_per + 1) * 2, s, w, cols, ldw,
                            block, rows_per, blk_ptr, idx, static_cast<uint16_t*>(vals)));
  } else {
    BSP_CUDA_TRY(launch_pdl(repack_kernel, grid, dim3(256), 0, s, w, ldw, block, blk_ptr, idx, static_cast<uint16_t*>(vals)));
  }
  return BSP_OK;
}
