// bsp_percentile_threshold and its batched form: the threshold that a target compression rate implies
// (Section 3.1's percentile), a radix select on the bit patterns of the groups' float32 sums of squares
// (monotone, they are not negative).  Three launches for any number of matrices:
//   clear    the matrix's histogram and counters (in the part of the workspace that holds flags elsewhere);
//   sums     the sum of every group, W read once (HBM-bound: 2 bytes per weight in, 4 per group out, 16-byte
//            loads wherever the geometry allows), and a histogram of their upper 12 bits: in shared memory
//            per CTA, then one global addition per bin that was hit (a hundred or so);
//   select   every CTA looks the answer's bin up in the histogram, lists its keys of that bin (a few per
//            cent) in the workspace, and the last CTA of a matrix to do so finds the answer among them in two
//            more digits (10 and 9 bits).
// Matrices whose flag region is too small for histogram and list are selected by one CTA straight from the
// sums, and so is what overflows the list (a matrix of equal groups).  Latency bounds all of this: 3 us for
// the sums of a 3072 x 768 matrix and 5 us for the select, against 197 us for one CTA with four 8-bit digits
// over all keys and 12 us for a cluster of eight that merged its histograms through distributed shared memory.
#include "bsp_common.cuh"

namespace bsp {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kBits1 = 12, kBits2 = 10, kBits3 = 9;          // 31 bits: the sign of a sum of squares is 0
constexpr int kBins1 = 1 << kBits1, kBins2 = 1 << kBits2, kBins3 = 1 << kBits3;
constexpr int kHeadWords = kBins1 + 64;                      // histogram, then list length and finished CTAs
constexpr int kSelectBatch = 96;                             // matrices per launch; the table is a kernel parameter
constexpr int kSumThreads = 128;

struct SelectJob {
  const uint16_t* W;
  int cols, ldw, n_blocks, vec;
  float* S;
  float* out;
  long long n, r;
  uint32_t* head;            // histogram and counters, or null: one CTA selects straight from the sums
  uint32_t list_cap;         // keys that fit behind them
  int chunks;                // CTAs of the select
};
template <int N>
struct SelectBatchT {
  int n_jobs, block;
  int loads;                 // 16-byte loads per thread and CTA of the select
  int first_block[N];        // apart from the wide records: a search stays within a few lines of the constant cache
  int first_chunk[N];
  SelectJob job[N];
};
template <int N>
__device__ __forceinline__ int owner(const int (&first)[N], int n, int at) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first[mid] <= at) lo = mid; else hi = mid - 1;
  }
  return lo;
}

template <int N>
__global__ void __launch_bounds__(kSelThreads)
select_clear_kernel(const __grid_constant__ SelectBatchT<N> B) {
  pdl_wait();
  pdl_launch_dependents();
  uint32_t* head = B.job[blockIdx.x].head;
  if (head == nullptr) return;
  for (int i = threadIdx.x; i < kHeadWords; i += kSelThreads) head[i] = 0u;
}

// ------------------------------------------------------------------------------------------ sums
__device__ __forceinline__ void clear_bins(uint32_t* hist) {
  for (int i = threadIdx.x; i < kBins1 / 4; i += blockDim.x) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
}
__device__ __forceinline__ void count_key(uint32_t* hist, float S) { atomicAdd(&hist[__float_as_uint(S) >> (kBits2 + kBits3)], 1u); }
__device__ __forceinline__ void add_bins(const uint32_t* hist, uint32_t* head) {
  for (int i = threadIdx.x; i < kBins1 / 4; i += blockDim.x) {
    const uint4 c = reinterpret_cast<const uint4*>(hist)[i];
    if ((c.x | c.y | c.z | c.w) == 0u) continue;
    if (c.x) atomicAdd(head + 4 * i, c.x);
    if (c.y) atomicAdd(head + 4 * i + 1, c.y);
    if (c.z) atomicAdd(head + 4 * i + 2, c.z);
    if (c.w) atomicAdd(head + 4 * i + 3, c.w);
  }
}

// Orientation C, one CTA per row-block of every matrix.
template <int N>
__global__ void __launch_bounds__(kSumThreads)
sums_c_kernel(const __grid_constant__ SelectBatchT<N> B) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  const int jn = owner(B.first_block, B.n_jobs, static_cast<int>(blockIdx.x));
  const SelectJob& J = B.job[jn];
  const int b = static_cast<int>(blockIdx.x) - B.first_block[jn];
  const uint16_t* wblk = J.W + static_cast<size_t>(b) * B.block * J.ldw;
  float* out = J.S + static_cast<size_t>(b) * J.cols;
  const bool count = J.head != nullptr;
  if (count) clear_bins(hist);
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  if (J.vec) {
    for (int q = threadIdx.x; q < (J.cols >> 3); q += kSumThreads) {
      float acc[8];
      sumsq8(wblk + (q << 3), B.block, J.ldw, acc);
      float4* dst = reinterpret_cast<float4*>(out + (q << 3));
      dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
      if (count) {
#pragma unroll
        for (int i = 0; i < 8; ++i) count_key(hist, acc[i]);
      }
    }
  } else {
    for (int g = threadIdx.x; g < J.cols; g += kSumThreads) {
      const float S = group_sumsq_strided(wblk + g, B.block, J.ldw);
      out[g] = S;
      if (count) count_key(hist, S);
    }
  }
  if (!count) return;
  __syncthreads();
  add_bins(hist, J.head);
}

// Orientation R: one thread per group, neighbouring threads on neighbouring groups of a row.
__global__ void __launch_bounds__(256)
sums_r_kernel(const uint16_t* __restrict__ W, int rows, int per_row, int ldw, int block, int vec, float* __restrict__ S,
              uint32_t* head) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  if (head != nullptr) clear_bins(hist);
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  const long long g = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (g < static_cast<long long>(rows) * per_row) {
    const long long i = g / per_row;
    const int a = static_cast<int>(g - i * per_row);
    const float v = group_sumsq_contig(W + static_cast<size_t>(i) * ldw + static_cast<size_t>(a) * block, block, vec);
    S[g] = v;
    if (head != nullptr) count_key(hist, v);
  }
  if (head == nullptr) return;
  __syncthreads();
  add_bins(hist, head);
}

// ---------------------------------------------------------------------------------------- select
// The bin of a histogram that holds the want-th smallest key (1-based) and the rank inside that bin; the whole
// CTA takes part and gets the answer.  A warp adds up a 32nd of the bins, every warp scans the 32 sums, and the
// one that holds the answer scans its bins.
struct Pick {
  uint32_t bin, want;
};
template <int BINS>
__device__ __forceinline__ Pick pick_bin(const uint32_t* hist, uint32_t want, uint32_t* s_sum, uint32_t* s_pick) {
  constexpr int kPerWarp = BINS / 32, kRounds = (kPerWarp + 31) / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t c[kRounds], sums[kRounds], sum = 0u;
#pragma unroll
  for (int i = 0; i < kRounds; ++i) c[i] = i * 32 + lane < kPerWarp ? hist[warp * kPerWarp + i * 32 + lane] : 0u;
#pragma unroll
  for (int i = 0; i < kRounds; ++i) {
    sums[i] = __reduce_add_sync(0xffffffffu, c[i]);
    sum += sums[i];
  }
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  const uint32_t w = s_sum[lane];
  uint32_t incl = w;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  uint32_t before = __shfl_sync(0xffffffffu, incl - w, warp);
  if (before < want && want <= before + sum) {               // all lanes of a warp agree; exactly one warp goes on
    uint32_t mine = c[0];
    int round = 0;
#pragma unroll
    for (int i = 0; i + 1 < kRounds; ++i)
      if (round == i && want > before + sums[i]) { before += sums[i]; round = i + 1; mine = c[i + 1]; }
    uint32_t in = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, in, o);
      if (lane >= o) in += up;
    }
    if (before + in - mine < want && want <= before + in) {
      s_pick[0] = static_cast<uint32_t>(warp * kPerWarp + round * 32 + lane);
      s_pick[1] = want - (before + in - mine);
    }
  }
  __syncthreads();
  return Pick{s_pick[0], s_pick[1]};
}

// Calls f(key) for every key whose upper bits (from bit `above` on) are `prefix`: one CTA, all of the keys
// (read from L2: a list was written by other CTAs of the same launch).
template <class F>
__device__ __forceinline__ void for_matching(const uint32_t* __restrict__ keys, long long n, int above, uint32_t prefix, F f) {
  const uint4* v4 = reinterpret_cast<const uint4*>(keys);
  const long long n4 = n >> 2;
  for (long long i = threadIdx.x; i < n4; i += 4 * kSelThreads) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i + u * kSelThreads < n4) v[u] = __ldcg(v4 + i + u * kSelThreads);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (i + u * kSelThreads >= n4) break;
      const uint32_t k[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if ((k[e] >> above) == prefix) f(k[e]);
    }
  }
  if (threadIdx.x < static_cast<unsigned>(n & 3)) {
    const uint32_t k = __ldcg(keys + (n4 << 2) + threadIdx.x);
    if ((k >> above) == prefix) f(k);
  }
}

template <int N>
__global__ void __launch_bounds__(kSelThreads)
select_kernel(const __grid_constant__ SelectBatchT<N> B) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  __shared__ uint32_t s_sum[32];
  __shared__ uint32_t s_pick[2];
  __shared__ uint32_t s_n, s_base;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int jn = owner(B.first_chunk, B.n_jobs, static_cast<int>(blockIdx.x));
  const SelectJob& J = B.job[jn];
  const int chunk = static_cast<int>(blockIdx.x) - B.first_chunk[jn];
  const uint32_t* keys = reinterpret_cast<const uint32_t*>(J.S);
  const long long n = J.n;
  if (threadIdx.x == 0) s_n = 0u;
  pdl_wait();
  pdl_launch_dependents();
  if (J.r <= 0) {
    if (chunk == 0 && threadIdx.x == 0) *J.out = -1.0f;
    return;
  }
  Pick p{0u, static_cast<uint32_t>(J.r)};
  uint32_t prefix;
  uint32_t found = 0xffffffffu;                              // keys on the list; too many to use it where there is none
  if (J.head != nullptr) {
    // this CTA's keys are on their way while the histogram is looked at
    uint32_t k[16], valid = 0u;
    const uint4* v4 = reinterpret_cast<const uint4*>(keys);
    const long long n4 = n >> 2, i0 = static_cast<long long>(chunk) * B.loads * kSelThreads + threadIdx.x;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (u < B.loads && i0 + u * kSelThreads < n4) {
        const uint4 v = __ldcg(v4 + i0 + u * kSelThreads);
        k[4 * u] = v.x; k[4 * u + 1] = v.y; k[4 * u + 2] = v.z; k[4 * u + 3] = v.w;
        valid |= 0xfu << (4 * u);
      }
    }
    reinterpret_cast<uint4*>(hist)[threadIdx.x] = __ldcg(reinterpret_cast<const uint4*>(J.head) + threadIdx.x);
    static_assert(kBins1 == 4 * kSelThreads, "a 16-byte piece of the histogram per thread");
    __syncthreads();
    p = pick_bin<kBins1>(hist, p.want, s_sum, s_pick);
    uint32_t hit = 0u;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if ((valid >> i & 1u) && (k[i] >> (kBits2 + kBits3)) == p.bin) hit |= 1u << i;
    uint32_t tail = 0u;                                      // the last n mod 4 keys: the last CTA's
    const bool has_tail = chunk == J.chunks - 1 && threadIdx.x < static_cast<unsigned>(n & 3);
    if (has_tail) tail = __ldcg(keys + (n4 << 2) + threadIdx.x);
    const bool hit_tail = has_tail && (tail >> (kBits2 + kBits3)) == p.bin;
    const uint32_t mine = __popc(hit) + (hit_tail ? 1u : 0u);
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
      const uint32_t w = s_sum[lane];
      uint32_t in = w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t up = __shfl_up_sync(0xffffffffu, in, o);
        if (lane >= o) in += up;
      }
      s_sum[lane] = in - w;
      if (lane == 31) s_base = in ? atomicAdd(J.head + kBins1, in) : 0u;
    }
    __syncthreads();
    uint32_t at = s_base + s_sum[warp] + incl - mine;
    uint32_t* list = J.head + kHeadWords;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (hit >> i & 1u) {
        if (at < J.list_cap) list[at] = k[i];
        ++at;
      }
    if (hit_tail && at < J.list_cap) list[at] = tail;
    // the last CTA of the matrix goes on (every CTA's part of the list is visible to it)
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
      s_n = atomicAdd(J.head + kBins1 + 1, 1u);
      __threadfence();
    }
    __syncthreads();
    if (s_n + 1u != static_cast<uint32_t>(J.chunks)) return;
    found = __ldcg(J.head + kBins1);
    prefix = p.bin;
  } else {
    clear_bins(hist);
    __syncthreads();
    for_matching(keys, n, 31, 0u, [&](uint32_t k) { atomicAdd(&hist[k >> (kBits2 + kBits3)], 1u); });
    __syncthreads();
    p = pick_bin<kBins1>(hist, p.want, s_sum, s_pick);
    prefix = p.bin;
  }
  const bool listed = J.head != nullptr && found <= J.list_cap;
  if (listed) keys = J.head + kHeadWords;
  const long long left = listed ? static_cast<long long>(found) : n;
  hist[threadIdx.x] = 0u;                                    // two digits more, each with bins of its own
  if (threadIdx.x < kBins3) hist[kBins2 + threadIdx.x] = 0u;
  __syncthreads();
  for_matching(keys, left, kBits2 + kBits3, prefix, [&](uint32_t k) { atomicAdd(&hist[(k >> kBits3) & (kBins2 - 1)], 1u); });
  __syncthreads();
  p = pick_bin<kBins2>(hist, p.want, s_sum, s_pick);
  prefix = (prefix << kBits2) | p.bin;
  __syncthreads();
  for_matching(keys, left, kBits3, prefix, [&](uint32_t k) { atomicAdd(&hist[kBins2 + (k & (kBins3 - 1))], 1u); });
  __syncthreads();
  p = pick_bin<kBins3>(hist + kBins2, p.want, s_sum, s_pick);
  if (threadIdx.x == 0) {
    const float s_r = __uint_as_float((prefix << kBits3) | p.bin);
    float t = __fsqrt_rn(s_r);
    while (__fmul_rn(t, t) < s_r) t = __uint_as_float(__float_as_uint(t) + 1u);  // next float up (t >= 0)
    *J.out = t;
  }
}

// r = floor(G * (1 - 1/c)) in float64, as the definition states it
long long groups_to_remove(long long groups, double rate) {
  return static_cast<long long>(static_cast<double>(groups) * (1.0 - 1.0 / rate));
}

// A matrix's entry of the table; n_blocks x n_groups is its geometry in either orientation.
SelectJob select_job(const void* W, int cols, int ldw, int n_blocks, int n_groups, double rate, void* ws, float* out) {
  const long long groups = static_cast<long long>(n_blocks) * n_groups;
  const WsLayout L = ws_layout(n_blocks, n_groups);
  char* base = static_cast<char*>(ws);
  SelectJob J{};
  J.W = static_cast<const uint16_t*>(W);
  J.cols = cols;
  J.ldw = ldw;
  J.n_blocks = n_blocks;
  J.vec = cols % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16) ? 1 : 0;
  J.S = reinterpret_cast<float*>(base + L.sumsq_off);
  J.out = out;
  J.n = groups;
  J.r = groups_to_remove(groups, rate);
  // the region of the flags: one byte per group.  Below 1024 list entries (20 thousand groups) one CTA reads
  // all keys three times instead.
  const size_t words = (L.sumsq_off - L.keep_off) / 4;
  if (words >= kHeadWords + 1024) {
    J.head = reinterpret_cast<uint32_t*>(base + L.keep_off);
    J.list_cap = static_cast<uint32_t>(words - kHeadWords);
  }
  return J;
}

// The select counts in 32 bits.
bool too_many_groups(long long groups) { return groups >= (1LL << 32); }

template <int N>
int launch_select(SelectBatchT<N>& B, int sms, cudaStream_t s) {
  // 4096 keys per CTA and 16-byte load of a thread: as few loads as keep the grid to two CTAs per SM, at most four
  long long keys = 0;
  for (int i = 0; i < B.n_jobs; ++i) keys += B.job[i].n;
  B.loads = 1;
  while (B.loads < 4 && keys > 2LL * sms * B.loads * 4 * kSelThreads) B.loads *= 2;
  const long long per_cta = 4LL * kSelThreads * B.loads;
  int chunks = 0;
  for (int i = 0; i < B.n_jobs; ++i) {
    SelectJob& J = B.job[i];
    J.chunks = J.head == nullptr ? 1 : static_cast<int>((J.n + per_cta - 1) / per_cta);
    B.first_chunk[i] = chunks;
    chunks += J.chunks;
  }
  BSP_CUDA_TRY(launch_pdl(select_kernel<N>, dim3(chunks), dim3(kSelThreads), 0, s, B));
  return BSP_OK;
}

int sm_count(int* sms) {
  int dev = 0;
  BSP_CUDA_TRY(cudaGetDevice(&dev));
  BSP_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return BSP_OK;
}

}  // namespace
}  // namespace bsp

extern "C" int bsp_percentile_threshold(const void* W, int rows, int cols, int ldw, int block,
                                        int orient, double rate, float* threshold_out, void* ws,
                                        size_t ws_bytes, void* stream) {
  using namespace bsp;
  int st = check_matrix_args(W, rows, cols, ldw, block, orient);
  if (st != BSP_OK) return st;
  if (threshold_out == nullptr || ws == nullptr || !aligned_to(ws, 256)) return BSP_ERR_ARG;
  if (!(rate >= 1.0)) return BSP_ERR_ARG;
  int nb, ng;
  geometry(rows, cols, block, orient, &nb, &ng);
  const WsLayout L = ws_layout(nb, ng);
  if (ws_bytes < L.total) return BSP_ERR_WORKSPACE;
  const long long groups = static_cast<long long>(nb) * ng;
  if (too_many_groups(groups)) return BSP_ERR_UNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms;
  st = sm_count(&sms);
  if (st != BSP_OK) return st;
  SelectBatchT<1> B;
  B.n_jobs = 1;
  B.block = block;
  B.first_block[0] = 0;
  B.job[0] = select_job(W, cols, ldw, nb, ng, rate, ws, threshold_out);
  if (B.job[0].head != nullptr) BSP_CUDA_TRY(launch_pdl(select_clear_kernel<1>, dim3(1), dim3(kSelThreads), 0, s, B));
  if (orient == BSP_ORIENT_C) {
    BSP_CUDA_TRY(launch_pdl(sums_c_kernel<1>, dim3(nb), dim3(kSumThreads), 0, s, B));
  } else {
    BSP_CUDA_TRY(launch_pdl(sums_r_kernel, dim3(static_cast<unsigned>((groups + 255) / 256)), dim3(256), 0, s, B.job[0].W, rows, nb,
                            ldw, block, contig_vec(W, ldw, block), B.job[0].S, B.job[0].head));
  }
  return launch_select(B, sms, s);
}

extern "C" int bsp_percentile_threshold_batched(const bsp_layer_job* jobs, int n_jobs, int block, const double* rates,
                                                void* stream) {
  using namespace bsp;
  if (jobs == nullptr || rates == nullptr || n_jobs <= 0 || block <= 0) return BSP_ERR_ARG;
  if (n_jobs > 4096) return BSP_ERR_UNSUPPORTED;
  for (int i = 0; i < n_jobs; ++i) {                       // everything is checked before the first launch
    const bsp_layer_job& u = jobs[i];
    int st = check_matrix_args(u.W, u.rows, u.cols, u.ldw, block, BSP_ORIENT_C);
    if (st != BSP_OK) return st;
    if (u.threshold_dev == nullptr || u.ws == nullptr || !aligned_to(u.ws, 256)) return BSP_ERR_ARG;
    if (!(rates[i] >= 1.0)) return BSP_ERR_ARG;
    if (u.ws_bytes < ws_layout(u.rows / block, u.cols).total) return BSP_ERR_WORKSPACE;
    if (too_many_groups(static_cast<long long>(u.rows / block) * u.cols)) return BSP_ERR_UNSUPPORTED;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms;
  int st = sm_count(&sms);
  if (st != BSP_OK) return st;
  SelectBatchT<kSelectBatch> B;
  for (int j0 = 0; j0 < n_jobs; j0 += kSelectBatch) {
    B.n_jobs = n_jobs - j0 < kSelectBatch ? n_jobs - j0 : kSelectBatch;
    B.block = block;
    int blocks = 0;
    for (int i = 0; i < B.n_jobs; ++i) {
      const bsp_layer_job& u = jobs[j0 + i];
      B.job[i] = select_job(u.W, u.cols, u.ldw, u.rows / block, u.cols, rates[j0 + i], u.ws, const_cast<float*>(u.threshold_dev));
      B.first_block[i] = blocks;
      blocks += B.job[i].n_blocks;
    }
    BSP_CUDA_TRY(launch_pdl(select_clear_kernel<kSelectBatch>, dim3(B.n_jobs), dim3(kSelThreads), 0, s, B));
    BSP_CUDA_TRY(launch_pdl(sums_c_kernel<kSelectBatch>, dim3(blocks), dim3(kSumThreads), 0, s, B));
    st = launch_select(B, sms, s);
    if (st != BSP_OK) return st;
  }
  return BSP_OK;
}
