// Vectorised orientation-C kernels shared by bsp_group_norms, bsp_prune_pack and
// bsp_prepare_batched.  Two stages over a batch of matrices:
//   stage 1  one CTA per row-block, one thread per 8 adjacent columns: 16-byte loads down the
//            block's rows (8 rows in flight), eight independent sequential float32 sums of
//            squares (the defined decision quantity), then any of: norms / gamma (two 16-byte
//            stores each), penalty partial, keep flags (one 8-byte store) and the block's count.
//   stage 2  grid (row-blocks, row ranges of about 16K weights): blk_ptr from the counts before
//            the block, the ascending index list from the flags, and the rows, staged in shared
//            memory by asynchronous copies; from there (a) the zero-expanded execution layout,
//            (b) the packed tile, two values per 4-byte store.
#include <new>

#include "bsp_common.cuh"

namespace bsp {
namespace {

constexpr int kRowsPerPass = 4;   // rows staged in shared memory at a time

// The job table travels as a kernel parameter; a single-matrix call gets a table of one job (0.2 KB instead
// of the 15 KB of a full batch, which every launch has to copy).
template <int N>
struct BatchT {
  int n_jobs, block, squared;
  float eps;
  int parts;                // stage 1 without flags: CTAs per row-block, each with part_chunks of its 8-column pieces
  int part_chunks;
  int early;                // stage 1: CTAs that can be waiting for the previous kernel
  int first_block[N + 1];   // CTA index of each job's first row-block
  FusedJob job[N];
};

// Job that owns CTA `cta`: the last j with first_block[j] <= cta (binary search).
template <int N>
__device__ __forceinline__ int find_job(const BatchT<N>& B, int cta) {
  int lo = 0, hi = B.n_jobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.first_block[mid] <= cta) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// (kParts as a template parameter: with the ranges as run-time values whole row-blocks took up to 2 us longer)
// Short blocks: 56 registers, which 288 threads of four CTAs leave, and not the 58 that the compiler would take: ten CTAs of 96
// threads per SM instead of twelve made a second wave of 1536 (6144 x 768 in 4-row blocks 3.2 -> 3.7 us).
template <int N, bool kParts, int kTrip>
__global__ void __launch_bounds__(kTrip == 4 && !kParts ? 288 : 256, kTrip == 4 && !kParts ? 4 : 0)
fused_stage1_kernel(const __grid_constant__ BatchT<N> B) {
  __shared__ int s_cnt[8];
  __shared__ double s_pen[8];
  const int cta = kParts ? static_cast<int>(blockIdx.x) / B.parts : static_cast<int>(blockIdx.x);
  const int q0 = kParts ? (static_cast<int>(blockIdx.x) - cta * B.parts) * B.part_chunks : 0;
  const int j = find_job(B, cta);
  const FusedJob& J = B.job[j];
  const int b = cta - B.first_block[j];
  const int q_end = kParts ? min(J.cols >> 3, q0 + B.part_chunks) : J.cols >> 3;
  // (the rows of the CTAs that wait for the previous kernel, often a clearing one, come to L2 meanwhile: see prefetch_bytes)
  if (static_cast<int>(blockIdx.x) < B.early)
    for (int r = threadIdx.x; r < B.block; r += blockDim.x)
      prefetch_bytes(J.W + (static_cast<size_t>(b) * B.block + r) * J.ldw + (q0 << 3), static_cast<uint32_t>(q_end - q0) * 16u);
  pdl_wait();
  pdl_launch_dependents();
  const bool want_flags = J.flags != nullptr;
  const bool want_pen = J.penalty != nullptr;
  const bool want_norms = J.norms != nullptr || J.gamma_out != nullptr || want_pen;
  float t2 = 0.0f;
  bool keep_all = false;
  if (want_flags) {
    const float t = J.threshold_dev ? *J.threshold_dev : J.threshold;
    keep_all = t < 0.0f;
    t2 = __fmul_rn(t, t);
  }
  int count = 0;
  float pen = 0.0f;
  for (int q = q0 + threadIdx.x; q < q_end; q += blockDim.x) {
    float acc[8];
    sumsq8<kTrip>(J.W + static_cast<size_t>(b) * B.block * J.ldw + (q << 3), B.block, J.ldw, acc);
    const size_t g0 = static_cast<size_t>(b) * J.cols + (q << 3);
    if (want_flags) {
      uint32_t lo = 0, hi = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t k0 = (keep_all || acc[i] > t2) ? 1u : 0u;
        const uint32_t k1 = (keep_all || acc[4 + i] > t2) ? 1u : 0u;
        lo |= k0 << (8 * i);
        hi |= k1 << (8 * i);
        count += static_cast<int>(k0 + k1);
      }
      *reinterpret_cast<uint2*>(J.flags + g0) = make_uint2(lo, hi);
    }
    if (want_norms) {
      float n[8], base[8], fresh[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        n[i] = norm_from_sumsq(acc[i]);
        base[i] = B.squared ? acc[i] : n[i];
        fresh[i] = reciprocal(base[i] + B.eps);
      }
      if (J.norms) {
        *reinterpret_cast<float4*>(J.norms + g0) = make_float4(n[0], n[1], n[2], n[3]);
        *reinterpret_cast<float4*>(J.norms + g0 + 4) = make_float4(n[4], n[5], n[6], n[7]);
      }
      if (J.gamma_out) {
        *reinterpret_cast<float4*>(J.gamma_out + g0) = make_float4(fresh[0], fresh[1], fresh[2], fresh[3]);
        *reinterpret_cast<float4*>(J.gamma_out + g0 + 4) = make_float4(fresh[4], fresh[5], fresh[6], fresh[7]);
      }
      if (want_pen) {
        if (J.gamma_in) {
          const float4 a = ld_global(reinterpret_cast<const float4*>(J.gamma_in + g0));
          const float4 c = ld_global(reinterpret_cast<const float4*>(J.gamma_in + g0 + 4));
          const float w[8] = {a.x, a.y, a.z, a.w, c.x, c.y, c.z, c.w};
#pragma unroll
          for (int i = 0; i < 8; ++i) pen = fmaf(w[i], base[i], pen);
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) pen = fmaf(fresh[i], base[i], pen);
        }
      }
    }
  }
  // block totals: count (int) and penalty (float per thread, float64 from here on, fixed order)
  count = warp_sum(count);
  double pd = warp_sum(static_cast<double>(pen));
  const int warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) { s_cnt[warp] = count; s_pen[warp] = pd; }
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
    double p = 0.0;
    for (int w = 0; w < n_warps; ++w) { c += s_cnt[w]; p += s_pen[w]; }
    if (want_flags) J.counts[b] = c;
    if (want_pen) {
      if (J.partial) J.partial[b] = p;
      else if (p != 0.0) atomicAdd(J.penalty, p);
    }
  }
}

// Rows staged in shared memory at a time: about 24 KB (the whole block for narrow matrices).
// With the 4-byte index list per column the dynamic shared memory stays under 48 KB for
// every width up to kFusedMaxCols.
__host__ __device__ inline int rows_per_pass(int cols) {
  int r = 12288 / cols;
  r = r < 3 ? 3 : r;
  return r > 16 ? 16 : r;
}
static_assert(kFusedMaxCols * (3 * 2 + 4) + 1024 <= 48 * 1024, "stage-2 shared memory must fit the default limit");

// Rows of a row-block that one stage-2 CTA handles: about 16K weights per CTA, a multiple of the
// 4-row staging pass, so that narrow matrices build their index list once per block and wide ones
// still spread over several CTAs.
__host__ __device__ inline int rows_per_cta(int cols, int d) {
  int r = (16384 / cols) / kRowsPerPass * kRowsPerPass;
  if (r < kRowsPerPass) r = kRowsPerPass;
  return r > d ? d : r;
}

template <int N>
__global__ void __launch_bounds__(256)
fused_stage2_kernel(const __grid_constant__ BatchT<N> B) {
  extern __shared__ __align__(16) uint8_t s_raw[];
  __shared__ int s_warp[32];
  __shared__ int s_part[8];
  __shared__ double s_red[8];
  const int j = find_job(B, blockIdx.x);
  const FusedJob& J = B.job[j];
  const int b = blockIdx.x - B.first_block[j];
  const int d = B.block;
  const int per_cta = rows_per_cta(J.cols, d);
  const int r_begin = blockIdx.y * per_cta;
  if (r_begin >= d) return;
  const int r_end = min(d, r_begin + per_cta);
  const int pass_rows = rows_per_pass(J.cols);
  uint16_t* s_w = reinterpret_cast<uint16_t*>(s_raw);                                                   // [pass_rows][cols]
  uint16_t* s_idx = reinterpret_cast<uint16_t*>(s_raw + static_cast<size_t>(pass_rows) * J.cols * 2);  // [cols]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
  const uint16_t* wblk = J.W + static_cast<size_t>(b) * d * J.ldw;
  const uint8_t* flags = J.flags + static_cast<size_t>(b) * J.cols;
  const int chunks = J.cols >> 3;

  // Rows of a pass into shared memory, one warp per row, by asynchronous copies: the first pass's rows, the counts
  // before the block and the flags are all on their way at once, so the CTA pays one trip to memory before it
  // writes (it used to be four in a row, 8 us for a 3072 x 768 matrix of 16-row blocks).
  auto fetch_rows = [&](int r_lo) {
    const int n_rows = min(pass_rows, r_end - r_lo);
    for (int rr = warp; rr < n_rows; rr += n_warps) {
      const uint16_t* src = wblk + static_cast<size_t>(r_lo + rr) * J.ldw;
      const uint32_t dst = static_cast<uint32_t>(__cvta_generic_to_shared(s_w + rr * J.cols));
      for (int q = lane; q < chunks; q += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + static_cast<uint32_t>(q) * 16u), "l"(src + (q << 3)) : "memory");
    }
  };
  // (The flags and counts come from the launch right before.  W does not, and this grid has started only because all
  // that came before that launch is complete, so the rows travel while the flags are made: 9.0 -> 8.2 us for the two
  // launches at 3072 x 768.  The same for the norms behind the clearing of their penalty gave nothing.)
  fetch_rows(r_begin);
  pdl_wait();
  pdl_launch_dependents();
  const int q_first = static_cast<int>(threadIdx.x);
  uint2 f = q_first < chunks ? *reinterpret_cast<const uint2*>(flags + (q_first << 3)) : make_uint2(0u, 0u);
  const int kc = J.counts[b];
  int part = 0;                                              // blk_ptr[b] = sum of counts[0..b)
  for (int i = threadIdx.x; i < b; i += blockDim.x) part += J.counts[i];

  // penalty total of the job: its first CTA adds the per-block partials in a fixed order
  if (b == 0 && blockIdx.y == 0 && J.penalty != nullptr && J.partial != nullptr) {
    double p = 0.0;
    for (int i = threadIdx.x; i < J.n_blocks; i += blockDim.x) p += J.partial[i];
    p = warp_sum(p);
    if (lane == 0) s_red[warp] = p;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int w = 0; w < n_warps; ++w) tot += s_red[w];
      *J.penalty = tot;
    }
  }

  // the sum of the counts and the first round of the list (each thread inspects 8 flags) share one barrier
  part = warp_sum(part);
  int incl = __popc(f.x) + __popc(f.y);
  const int mine = incl;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  if (lane == 31) s_warp[warp] = incl;
  if (lane == 0) s_part[warp] = part;
  __syncthreads();
  int base = 0, running = 0, p0 = incl - mine;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    base += s_part[w];
    if (w < warp) p0 += s_warp[w];
    running += s_warp[w];
  }
  if (blockIdx.y == 0 && threadIdx.x == 0) {
    J.blk_ptr[b] = base;
    if (b == J.n_blocks - 1) {
      J.blk_ptr[J.n_blocks] = base + kc;
      if (J.kept_weights) *J.kept_weights = static_cast<int64_t>(base + kc) * d;
    }
  }
  auto list8 = [&](uint2 fl, int q, int p) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t bit = ((i < 4 ? fl.x : fl.y) >> (8 * (i & 3))) & 1u;
      if (bit) {
        s_idx[p] = static_cast<uint16_t>((q << 3) + i);
        if (blockIdx.y == 0) J.idx[base + p] = (q << 3) + i;
        ++p;
      }
    }
  };
  list8(f, q_first, p0);
  for (int q0 = blockDim.x; q0 < chunks; q0 += blockDim.x) {
    const int q = q0 + threadIdx.x;
    f = q < chunks ? *reinterpret_cast<const uint2*>(flags + (q << 3)) : make_uint2(0u, 0u);
    int total;
    __syncthreads();                                         // s_warp of the round before has been read
    const int p = running + block_exclusive_scan(__popc(f.x) + __popc(f.y), s_warp, &total);
    running += total;
    list8(f, q, p);
  }
  // (no return before this point: other threads' copies are in flight)

  const long long tile0 = static_cast<long long>(d) * base;  // element offset of the block's tile in vals
  const bool pair_ok = (reinterpret_cast<uintptr_t>(J.vals) & 3) == 0;
  for (int r_lo = r_begin; r_lo < r_end; r_lo += pass_rows) {
    const int n_rows = min(pass_rows, r_end - r_lo);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();   // s_w (and, on the first pass, s_idx) complete
    // execution layout: the rows with the pruned columns zeroed
    // (a plan that IS W: in-place mode, only pieces that change are written)
    if (J.plan != nullptr) {
      const bool in_place = J.plan == J.W;
      for (int rr = warp; rr < n_rows; rr += n_warps) {
        uint16_t* pdst = J.plan + (static_cast<size_t>(b) * d + r_lo + rr) * (in_place ? J.ldw : J.cols);
        for (int q = lane; q < chunks; q += 32) {
          const uint4 w = *reinterpret_cast<const uint4*>(s_w + rr * J.cols + (q << 3));
          const uint2 fl = *reinterpret_cast<const uint2*>(flags + (q << 3));
          uint4 m;   // a flag byte is 0 or 1: flag * 0xffff masks the matching 16-bit element
          m.x = w.x & (((fl.x & 0xffu) * 0xffffu) | (((fl.x >> 8) & 0xffu) * 0xffff0000u));
          m.y = w.y & ((((fl.x >> 16) & 0xffu) * 0xffffu) | (((fl.x >> 24) & 0xffu) * 0xffff0000u));
          m.z = w.z & (((fl.y & 0xffu) * 0xffffu) | (((fl.y >> 8) & 0xffu) * 0xffff0000u));
          m.w = w.w & ((((fl.y >> 16) & 0xffu) * 0xffffu) | (((fl.y >> 24) & 0xffu) * 0xffff0000u));
          if (!in_place || ((m.x ^ w.x) | (m.y ^ w.y) | (m.z ^ w.z) | (m.w ^ w.w)) != 0u)
            *reinterpret_cast<uint4*>(pdst + (q << 3)) = m;
        }
      }
    }
    // packed tile rows of this pass, one warp per row: row r occupies vals[tile0 + r*kc, tile0 + (r+1)*kc).  A lane
    // takes two neighbouring positions (two values a few columns apart: different banks from lane to lane) and
    // stores them as one word; a row that starts at an odd element has its first one stored alone.
    for (int rr = warp; rr < n_rows; rr += n_warps) {
      const uint16_t* srow = s_w + rr * J.cols;
      const long long e0 = tile0 + static_cast<long long>(r_lo + rr) * kc;
      uint16_t* out_row = J.vals + e0;                               // element p of the row goes to out_row[p]
      if (pair_ok) {
        const int head = static_cast<int>(e0 & 1);
        const int n_pairs = kc > head ? (kc - head) >> 1 : 0;
        uint32_t* out32 = reinterpret_cast<uint32_t*>(out_row + head);
#pragma unroll 4
        for (int p = lane; p < n_pairs; p += 32) {
          const int at = head + 2 * p;
          out32[p] = static_cast<uint32_t>(srow[s_idx[at]]) | (static_cast<uint32_t>(srow[s_idx[at + 1]]) << 16);
        }
        if (lane == 0 && head && kc > 0) out_row[0] = srow[s_idx[0]];
        if (lane == 1 && head + 2 * n_pairs < kc) out_row[kc - 1] = srow[s_idx[kc - 1]];
      } else {
        for (int p = lane; p < kc; p += 32) out_row[p] = srow[s_idx[p]];
      }
    }
    if (r_lo + pass_rows < r_end) {
      __syncthreads();   // s_w is overwritten by the next pass
      fetch_rows(r_lo + pass_rows);
    }
  }
}

template <int N>
void fill_batch(BatchT<N>& B, const FusedJob* jobs, int n_jobs, int block, int* total, int* max_cols) {
  B.n_jobs = n_jobs;
  B.block = block;
  *total = 0;
  *max_cols = 0;
  for (int i = 0; i < n_jobs; ++i) {
    B.job[i] = jobs[i];
    B.first_block[i] = *total;
    *total += jobs[i].n_blocks;
    if (jobs[i].cols > *max_cols) *max_cols = jobs[i].cols;
  }
  B.first_block[n_jobs] = *total;
}

template <int N, bool kParts>
auto* stage1_kernel(int trip) {
  return trip == 4 ? fused_stage1_kernel<N, kParts, 4> : trip == 8 ? fused_stage1_kernel<N, kParts, 8>
         : trip == 16 ? fused_stage1_kernel<N, kParts, 16> : fused_stage1_kernel<N, kParts, N == 1 ? 32 : 16>;
}

template <int N>
int launch_stage1(const FusedJob* jobs, int n_jobs, int block, float eps, int squared, cudaStream_t s) {
  BatchT<N> B;
  int total, max_cols;
  fill_batch(B, jobs, n_jobs, block, &total, &max_cols);
  B.eps = eps;
  B.squared = squared;
  const int chunks = max_cols >> 3;
  int threads = (chunks + 31) / 32 * 32;
  threads = threads > 256 ? 256 : threads;
  B.parts = 1;
  B.part_chunks = chunks;
  int sms = 0;
  BSP_TRY(sm_count(&sms));
  if (N == 1 && jobs[0].flags == nullptr && jobs[0].partial == nullptr && total < sms && chunks > 128) {
    // A matrix of few wide row-blocks leaves SMs idle: they are cut into column ranges of a piece per thread (11 blocks of
    // 96 x 3072: 13.7 -> 8.9 us; ranges of 64 or 32 pieces cost 0.7 us more than whole blocks of 1024 columns).  Not where
    // a row-block is counted as a whole.
    threads = 128;
    B.parts = (chunks + 127) / 128;
    B.part_chunks = 128;
  }
  B.early = 2 * sms;
  // (warps per SM: 21 with 16 rows in flight, 12 with 32)
  const int warps = threads / 32;
  const int trip = rows_per_trip(block, static_cast<long long>(total) * B.parts, 21 / warps, N == 1 ? 12 / warps : 0, sms);
  auto* kernel = B.parts > 1 ? stage1_kernel<N, N == 1>(trip) : stage1_kernel<N, false>(trip);
  BSP_CUDA_TRY(launch_pdl(kernel, dim3(total * B.parts), dim3(threads), 0, s, B));
  return BSP_OK;
}

template <int N>
int launch_stage2(const FusedJob* jobs, int n_jobs, int block, cudaStream_t s) {
  BatchT<N> B;
  int total, max_cols;
  fill_batch(B, jobs, n_jobs, block, &total, &max_cols);
  B.eps = 0.0f;
  B.squared = 0;
  B.parts = 1;
  B.part_chunks = 0;
  B.early = 0;
  int splits = 1;
  size_t smem = 0;
  for (int i = 0; i < n_jobs; ++i) {
    const int per = rows_per_cta(B.job[i].cols, block);
    const int need = (block + per - 1) / per;
    if (need > splits) splits = need;
    const size_t bytes = static_cast<size_t>(B.job[i].cols) * (rows_per_pass(B.job[i].cols) * 2 + 4);
    if (bytes > smem) smem = bytes;
  }
  BSP_CUDA_TRY(launch_pdl(fused_stage2_kernel<N>, dim3(total, splits), dim3(256), smem, s, B));
  return BSP_OK;
}

}  // namespace

int fused_stage1(const FusedJob* jobs, int n_jobs, int block, float eps, int squared, cudaStream_t s) {
  if (n_jobs == 1) return launch_stage1<1>(jobs, 1, block, eps, squared, s);
  for (int j0 = 0; j0 < n_jobs; j0 += kFusedMaxJobs) {
    const int n = n_jobs - j0 < kFusedMaxJobs ? n_jobs - j0 : kFusedMaxJobs;
    const int st = launch_stage1<kFusedMaxJobs>(jobs + j0, n, block, eps, squared, s);
    if (st != BSP_OK) return st;
  }
  return BSP_OK;
}

int fused_stage2(const FusedJob* jobs, int n_jobs, int block, cudaStream_t s) {
  if (n_jobs == 1) return launch_stage2<1>(jobs, 1, block, s);
  for (int j0 = 0; j0 < n_jobs; j0 += kFusedMaxJobs) {
    const int n = n_jobs - j0 < kFusedMaxJobs ? n_jobs - j0 : kFusedMaxJobs;
    const int st = launch_stage2<kFusedMaxJobs>(jobs + j0, n, block, s);
    if (st != BSP_OK) return st;
  }
  return BSP_OK;
}

}  // namespace bsp

extern "C" int bsp_prepare_batched(const bsp_layer_job* jobs, int n_jobs, int block, float eps, int pen,
                                   void* stream) {
  using namespace bsp;
  if (jobs == nullptr || n_jobs <= 0 || block <= 0) return BSP_ERR_ARG;
  if (pen != BSP_PEN_L2 && pen != BSP_PEN_L2SQ) return BSP_ERR_ARG;
  if (!(eps >= 0.0f)) return BSP_ERR_ARG;
  if (n_jobs > 4096) return BSP_ERR_UNSUPPORTED;
  // validate everything before the first launch
  for (int i = 0; i < n_jobs; ++i) {
    const bsp_layer_job& u = jobs[i];
    int st = check_matrix_args(u.W, u.rows, u.cols, u.ldw, block, BSP_ORIENT_C);
    if (st != BSP_OK) return st;
    if (u.blk_ptr == nullptr || u.idx == nullptr || u.vals == nullptr || u.ws == nullptr) return BSP_ERR_ARG;
    if (!aligned_to(u.ws, 256) || !aligned_to(u.blk_ptr, 4) || !aligned_to(u.idx, 4) || !aligned_to(u.vals, 2)) return BSP_ERR_ARG;
    if (u.threshold != u.threshold) return BSP_ERR_ARG;
    if (u.ws_bytes < ws_layout(u.rows / block, u.cols).total) return BSP_ERR_WORKSPACE;
    if (u.plan != nullptr && u.plan != u.W) {          // plan == W: in-place mode, W itself becomes the layout
      if (!aligned_to(u.plan, 256)) return BSP_ERR_ARG;
      if (u.plan_bytes < static_cast<size_t>(u.rows) * u.cols * 2) return BSP_ERR_WORKSPACE;
    }
    const bool ok = fused_shape_ok(u.W, u.rows, u.cols, u.ldw, block) && (u.keep == nullptr || aligned_to(u.keep, 8)) &&
                    (u.norms == nullptr || aligned_to(u.norms, 16)) && (u.gamma_out == nullptr || aligned_to(u.gamma_out, 16)) &&
                    (u.gamma_in == nullptr || aligned_to(u.gamma_in, 16));
    if (!ok) return BSP_ERR_UNSUPPORTED;
  }
  FusedJob* fj = new (std::nothrow) FusedJob[n_jobs];
  if (fj == nullptr) return BSP_ERR_ARG;
  for (int i = 0; i < n_jobs; ++i) {
    const bsp_layer_job& u = jobs[i];
    const int nb = u.rows / block;
    const WsLayout L = ws_layout(nb, u.cols);
    char* wsb = static_cast<char*>(u.ws);
    fj[i] = FusedJob{static_cast<const uint16_t*>(u.W), u.rows, u.cols, u.ldw, nb, u.threshold, u.threshold_dev,
                     u.norms, u.gamma_in, u.gamma_out, u.penalty, reinterpret_cast<double*>(wsb + L.sumsq_off),
                     u.keep ? u.keep : reinterpret_cast<uint8_t*>(wsb + L.keep_off),
                     reinterpret_cast<int32_t*>(wsb + L.counts_off), u.blk_ptr, u.idx, static_cast<uint16_t*>(u.vals),
                     u.kept_weights, static_cast<uint16_t*>(u.plan)};
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // The streaming one-pass kernel (W read once) takes the batch when every matrix fits its limits.  Its
  // per-item counts and penalty partials live in the workspace's S region, which this call does not use otherwise.
  int st = BSP_OK;
  bool done = false;
  {
    int32_t** pcounts = new (std::nothrow) int32_t*[n_jobs];
    double** ppartial = new (std::nothrow) double*[n_jobs];
    bool fits = pcounts != nullptr && ppartial != nullptr;
    for (int i = 0; i < n_jobs && fits; ++i) {
      const bsp_layer_job& u = jobs[i];
      const int nb = u.rows / block;
      const WsLayout L = ws_layout(nb, u.cols);
      char* region = static_cast<char*>(u.ws) + L.sumsq_off;          // 4 bytes per group
      const size_t slots = static_cast<size_t>(nb) * 32;              // at most 31 parts per block, plus two counters
      pcounts[i] = reinterpret_cast<int32_t*>(region);
      ppartial[i] = reinterpret_cast<double*>(region + round_up(slots * sizeof(int32_t), 256));
      if (round_up(slots * 4, 256) + slots * 8 > static_cast<size_t>(nb) * u.cols * 4) fits = false;
    }
    const int squared = pen == BSP_PEN_L2SQ ? 1 : 0;
    if (fits) st = fused_stream(fj, n_jobs, block, eps, squared, pcounts, ppartial, s, &done);
    delete[] pcounts;
    delete[] ppartial;
  }
  if (st == BSP_OK && !done) {
    st = fused_stage1(fj, n_jobs, block, eps, pen == BSP_PEN_L2SQ ? 1 : 0, s);
    if (st == BSP_OK) st = fused_stage2(fj, n_jobs, block, s);
  }
  delete[] fj;
  return st;
}
