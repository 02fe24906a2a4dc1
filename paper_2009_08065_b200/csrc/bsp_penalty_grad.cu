// bsp_penalty_grad: gradient of the reweighted group-Lasso term with respect to W, the penalty
// weights held fixed (Algorithm 2 keeps gamma between milestones while the optimiser minimises
// mixed_loss = l1loss + f(W, b)):
//   Eq. 2 / Eq. 3 form:   d/dW_e [ gamma_g ||W_g||_2 ] = gamma_g W_e / ||W_g||_2   (0 for an all-zero group)
//   squared-norm variant: d/dW_e [ alpha_g ||W_g||^2 ] = 2 alpha_g W_e
// HBM-bound: W is read (the second read of a group hits L1/L2), one float is written per weight.
#include "bsp_common.cuh"

namespace bsp {
namespace {

struct GradArgs {
  const uint16_t* W;
  int rows, cols, ldw, block, orient, squared, accumulate;
  const float* gamma;
  float scale;
  float* grad;
  int ldg;
  unsigned first_wave;       // CTAs of the tiled kernel that are resident at once
};

// Orientation C, 8-element alignment, blocks of 8 to 32 rows: a CTA takes 256 columns of a row-block.  Its
// loads (8 columns of a row per item: 16 bytes of W and, when adding to a gradient, 32 bytes of it) are all
// issued before anything is computed, W goes through shared memory, each thread sums the squares of one
// column in row order and the factors come back through shared memory.  HBM-bound: 2 bytes in and 4 (8 when
// accumulating) per weight.  One thread per 8 columns walking down the rows, as the kernel below does, has
// 1/16 of the loads in flight: 14 us instead of 6 for a 4096 x 1024 matrix of 16-row blocks, accumulating.
constexpr int kGradCols = 256, kGradMinRows = 8, kGradMaxRows = 32;
template <int ITEMS>
__global__ void __launch_bounds__(256)
grad_c_tile_kernel(GradArgs A) {
  __shared__ __align__(16) uint16_t s_w[8 * ITEMS][kGradCols];
  __shared__ __align__(16) float s_f[kGradCols];
  const int b = blockIdx.x, c0 = blockIdx.y * kGradCols;
  const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;     // a warp per row, 8 columns per lane
  const int c = c0 + (lane << 3);
  const bool on = c < A.cols;
  const size_t r0 = static_cast<size_t>(b) * A.block;
  // (only the CTAs that can be waiting: behind them it would cost issue slots for nothing)
  const bool early = blockIdx.y * gridDim.x + blockIdx.x < A.first_wave;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int r = row + 8 * i;
    if (early && on && r < A.block) {
      if ((lane & 7) == 0) prefetch_line(A.W + (r0 + r) * A.ldw + c);
      if (A.accumulate && (lane & 3) == 0) prefetch_line(A.grad + (r0 + r) * A.ldg + c);
    }
  }
  if (early && on && row == 0 && (lane & 3) == 0) prefetch_line(A.gamma + static_cast<size_t>(b) * A.cols + c);
  pdl_wait();
  pdl_launch_dependents();
  uint4 w[ITEMS];
  float4 g[ITEMS][2];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int r = row + 8 * i;
    if (on && r < A.block) w[i] = ld_global(reinterpret_cast<const uint4*>(A.W + (r0 + r) * A.ldw + c));
  }
  const float gamma = c0 + static_cast<int>(threadIdx.x) < A.cols ? ld_global(A.gamma + static_cast<size_t>(b) * A.cols + c0 + threadIdx.x) : 0.0f;
  if (A.accumulate) {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const int r = row + 8 * i;
      if (on && r < A.block) {
        const float4* src = reinterpret_cast<const float4*>(A.grad + (r0 + r) * A.ldg + c);
        g[i][0] = src[0];
        g[i][1] = src[1];
      }
    }
  }
  if (!A.squared) {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
      if (on && row + 8 * i < A.block) *reinterpret_cast<uint4*>(&s_w[row + 8 * i][lane << 3]) = w[i];
    __syncthreads();
    float acc = 0.0f;
    for (int r = 0; r < A.block; ++r) {
      const float v = bf16_bits_to_float(s_w[r][threadIdx.x]);
      acc = __fmaf_rn(v, v, acc);
    }
    const float n = __fsqrt_rn(acc);
    s_f[threadIdx.x] = c0 + static_cast<int>(threadIdx.x) < A.cols && n > 0.0f ? __fdiv_rn(A.scale * gamma, n) : 0.0f;
  } else {
    s_f[threadIdx.x] = 2.0f * A.scale * gamma;
  }
  __syncthreads();
  const float4 f0 = *reinterpret_cast<const float4*>(&s_f[lane << 3]), f1 = *reinterpret_cast<const float4*>(&s_f[(lane << 3) + 4]);
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int r = row + 8 * i;
    if (!on || r >= A.block) continue;
    float4 o0 = make_float4(f0.x * __uint_as_float(w[i].x << 16), f0.y * __uint_as_float(w[i].x & 0xffff0000u),
                            f0.z * __uint_as_float(w[i].y << 16), f0.w * __uint_as_float(w[i].y & 0xffff0000u));
    float4 o1 = make_float4(f1.x * __uint_as_float(w[i].z << 16), f1.y * __uint_as_float(w[i].z & 0xffff0000u),
                            f1.z * __uint_as_float(w[i].w << 16), f1.w * __uint_as_float(w[i].w & 0xffff0000u));
    if (A.accumulate) {
      o0.x += g[i][0].x; o0.y += g[i][0].y; o0.z += g[i][0].z; o0.w += g[i][0].w;
      o1.x += g[i][1].x; o1.y += g[i][1].y; o1.z += g[i][1].z; o1.w += g[i][1].w;
    }
    float4* dst = reinterpret_cast<float4*>(A.grad + (r0 + r) * A.ldg + c);
    dst[0] = o0;
    dst[1] = o1;
  }
}

// The same for other blocks: one thread per 8 adjacent columns of a row-block.
__global__ void __launch_bounds__(256)
grad_c_vec8_kernel(GradArgs A) {
  pdl_wait();
  pdl_launch_dependents();
  const int chunks = A.cols >> 3;
  const long long item = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (item >= static_cast<long long>(A.rows / A.block) * chunks) return;
  const int b = static_cast<int>(item / chunks), q = static_cast<int>(item - static_cast<long long>(b) * chunks);
  const uint16_t* p = A.W + static_cast<size_t>(b) * A.block * A.ldw + (q << 3);
  float factor[8];
  const float4 g0 = ld_global(reinterpret_cast<const float4*>(A.gamma + static_cast<size_t>(b) * A.cols + (q << 3)));
  const float4 g1 = ld_global(reinterpret_cast<const float4*>(A.gamma + static_cast<size_t>(b) * A.cols + (q << 3) + 4));
  const float gam[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
  if (A.squared) {
#pragma unroll
    for (int i = 0; i < 8; ++i) factor[i] = 2.0f * A.scale * gam[i];
  } else {
    float acc[8];
    sumsq8<16>(p, A.block, A.ldw, acc);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float n = __fsqrt_rn(acc[i]);
      factor[i] = n > 0.0f ? __fdiv_rn(A.scale * gam[i], n) : 0.0f;
    }
  }
  // (the address passes through an empty statement behind the wait, and so do these loads; unlike ordinary ones they may
  // pass the stores of the rows before)
  asm volatile("" : "+l"(p));
#pragma unroll 4
  for (int r = 0; r < A.block; ++r) {
    uint4 v;
    asm("ld.global.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p + static_cast<size_t>(r) * A.ldw));
    const uint32_t w32[4] = {v.x, v.y, v.z, v.w};
    float o[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[2 * i] = factor[2 * i] * __uint_as_float(w32[i] << 16);
      o[2 * i + 1] = factor[2 * i + 1] * __uint_as_float(w32[i] & 0xffff0000u);
    }
    float4* dst = reinterpret_cast<float4*>(A.grad + (static_cast<size_t>(b) * A.block + r) * A.ldg + (q << 3));
    if (A.accumulate) {
      const float4 a = dst[0], c = dst[1];
      o[0] += a.x; o[1] += a.y; o[2] += a.z; o[3] += a.w;
      o[4] += c.x; o[5] += c.y; o[6] += c.z; o[7] += c.w;
    }
    dst[0] = make_float4(o[0], o[1], o[2], o[3]);
    dst[1] = make_float4(o[4], o[5], o[6], o[7]);
  }
}

// Any geometry: one thread per group.  It overlaps the kernel before it only where it has a CTA per SM or fewer: CTAs
// placed while that kernel still holds seats spread unevenly over the SMs, and 2848 x 2080 in strips of 32 took 78 us
// against 53.
template <bool kOverlap>
__global__ void __launch_bounds__(256)
grad_generic_kernel(GradArgs A) {
  if (kOverlap) {
    pdl_wait();
    pdl_launch_dependents();
  }
  const bool c_orient = A.orient == BSP_ORIENT_C;
  const long long n_groups = c_orient ? static_cast<long long>(A.rows / A.block) * A.cols
                                      : static_cast<long long>(A.rows) * (A.cols / A.block);
  const long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (g >= n_groups) return;
  size_t first, stride;
  if (c_orient) {
    const long long b = g / A.cols;
    first = static_cast<size_t>(b) * A.block * A.ldw + static_cast<size_t>(g - b * A.cols);
    stride = A.ldw;
  } else {
    const int per_row = A.cols / A.block;
    const long long i = g / per_row;
    first = static_cast<size_t>(i) * A.ldw + static_cast<size_t>(g - i * per_row) * A.block;
    stride = 1;
  }
  float factor;
  if (A.squared) {
    factor = 2.0f * A.scale * A.gamma[g];
  } else {
    const float n = __fsqrt_rn(group_sumsq_strided(A.W + first, A.block, stride));
    factor = n > 0.0f ? __fdiv_rn(A.scale * A.gamma[g], n) : 0.0f;
  }
  // the same element position in grad: row = first / ldw, col = first % ldw
  const size_t row0 = first / A.ldw, col0 = first - row0 * A.ldw;
  for (int e = 0; e < A.block; ++e) {
    const size_t row = c_orient ? row0 + e : row0, col = c_orient ? col0 : col0 + e;
    const float v = factor * bf16_bits_to_float(A.W[first + e * stride]);
    float* dst = A.grad + row * A.ldg + col;
    *dst = A.accumulate ? *dst + v : v;
  }
}

}  // namespace
}  // namespace bsp

extern "C" int bsp_penalty_grad(const void* W, int rows, int cols, int ldw, int block, int orient, int pen,
                                const float* gamma, float scale, float* grad, int ldg, int accumulate,
                                void* stream) {
  using namespace bsp;
  int st = check_matrix_args(W, rows, cols, ldw, block, orient);
  if (st != BSP_OK) return st;
  if (pen != BSP_PEN_L2 && pen != BSP_PEN_L2SQ) return BSP_ERR_ARG;
  if (gamma == nullptr || grad == nullptr || !aligned_to(grad, 4) || !aligned_to(gamma, 4)) return BSP_ERR_ARG;
  if (scale != scale) return BSP_ERR_ARG;
  if (ldg < cols) return BSP_ERR_SHAPE;
  GradArgs A{static_cast<const uint16_t*>(W), rows, cols, ldw, block, orient, pen == BSP_PEN_L2SQ ? 1 : 0,
             accumulate ? 1 : 0, gamma, scale, grad, ldg, 0u};
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const bool vec = orient == BSP_ORIENT_C && cols % 8 == 0 && ldw % 8 == 0 && ldg % 4 == 0 && aligned_to(W, 16) &&
                   aligned_to(grad, 16) && aligned_to(gamma, 16);
  int sms = 0;
  BSP_TRY(sm_count(&sms));
  const dim3 tiles(rows / block, (cols + kGradCols - 1) / kGradCols);
  // A warp per row: blocks of fewer than 8 rows leave warps without work, which counts once the CTAs are more than run at
  // once (5343 x 920 in single rows 27 us, 12 by the other kernel, 7048 x 2160 in fours 28 and 21; but 117 x 544 in threes
  // 2.1 and 4.0).
  const bool tiled = tiles.y <= 65535 && block <= kGradMaxRows &&
                     (block >= kGradMinRows || static_cast<long long>(tiles.x) * tiles.y <= 8LL * sms);
  if (vec && tiled) {
    A.first_wave = 4u * static_cast<unsigned>(sms);
    BSP_CUDA_TRY(launch_pdl(block <= 8 ? grad_c_tile_kernel<1> : block <= 16 ? grad_c_tile_kernel<2> : grad_c_tile_kernel<4>, tiles,
                            dim3(256), 0, s, A));
  } else if (vec) {
    const long long items = static_cast<long long>(rows / block) * (cols / 8);
    BSP_CUDA_TRY(launch_pdl(grad_c_vec8_kernel, dim3(static_cast<unsigned>((items + 255) / 256)), dim3(256), 0, s, A));
  } else {
    int nb, ng;
    geometry(rows, cols, block, orient, &nb, &ng);
    const long long groups = static_cast<long long>(nb) * ng;
    const dim3 grid(static_cast<unsigned>((groups + 255) / 256));
    if (grid.x <= static_cast<unsigned>(sms)) BSP_CUDA_TRY(launch_pdl(grad_generic_kernel<true>, grid, dim3(256), 0, s, A));
    else grad_generic_kernel<false><<<grid, 256, 0, s>>>(A);
    BSP_LAUNCH_CHECK();
  }
  return BSP_OK;
}
