// bsp_percentile_threshold and its batched form: the threshold that a target compression rate implies
// (Section 3.1's percentile), a radix select on the bit patterns of the groups' float32 sums of squares
// (monotone, they are not negative).  Three launches for any number of matrices:
//   clear    the matrix's histogram (in the part of the workspace that holds flags elsewhere);
//   sums     the sum of every group, W read once (HBM-bound: 2 bytes per weight in, 4 per group out, 16-byte
//            loads wherever the geometry allows), and a histogram of their upper 12 bits: in shared memory
//            per CTA, then one global addition per bin that was hit (a hundred or so);
//   select   one thread-block cluster per matrix: every CTA looks the answer's bin up in the histogram and
//            lists its keys of that bin (a few per cent) in shared memory; CTA 0 gathers the lists through
//            distributed shared memory and finds the answer among them: a digit of 10 bits more, then a warp ranks
//            the few keys that are left (or a last digit of 9 bits, where many are alike).
// Matrices whose flag region is too small for the histogram are selected by one CTA straight from the sums, and
// so is what overflows a list (a matrix of equal groups).  Latency bounds all of this.  Measured on 147456
// groups: one CTA with four 8-bit digits over all keys 197 us; a cluster that also made the histogram 12 us;
// many CTAs with their lists in global memory, the last one finishing, 9 us (fences and atomics through L2
// instead of cluster barriers); one launch for everything, a cluster of 16 CTAs that sums its matrix itself, 16 us (W
// through 16 SMs, histograms through distributed shared memory).  The three launches: 15.0 -> 11.6 us for 3072 x 768 in
// 16-row blocks, 54.6 -> 48.3 for 72 matrices of a BERT-base stack, when the sums no longer waited for the clearing, the
// list was stored with predicated stores, all keys of a thread were asked for in one round, the gather kept four remote
// loads in flight and the last digit became a ranking.
#include "bsp_tc.cuh"

namespace bsp {
namespace {

constexpr int kSelThreads = 1024;
constexpr int kBits1 = 12, kBits2 = 10, kBits3 = 9;          // 31 bits: the sign of a sum of squares is 0
constexpr int kBins1 = 1 << kBits1, kBins2 = 1 << kBits2, kBins3 = 1 << kBits3;
constexpr int kList = 4096, kCandidates = 12288;              // keys on a CTA's list, and that CTA 0 gathers
constexpr int kSelSmem = (kList + kCandidates) * 4;
constexpr int kSelMaxCluster = 8;
constexpr int kSelLoads = 6;                                 // 16-byte loads of a thread in flight: a round of the list
// Copies of a histogram: a CTA of the sums adds to one of them (its number modulo the copies).  A sum of squares
// falls into a hundred bins or so, and 192 CTAs adding to the same words kept the next launch waiting for 1 us.
constexpr int kReplicas = 4;
constexpr int kSelectBatch = 96;                             // matrices per launch; the table is a kernel parameter
constexpr int kSumThreads = 128;
constexpr int kSumRowBytes = 24 * 1024;                      // rows of one item of the streaming sums kernel
constexpr int kSumPerSm = 3;                                 // its CTAs per SM: two row buffers and a histogram each

struct SelectJob {
  const uint16_t* W;
  int cols, ldw, n_blocks, vec;
  int parts, part_cols;      // sums in orientation C: column ranges of a row-block
  float* S;
  float* out;
  long long n, r;
  uint32_t* head;            // histograms, or null: one CTA selects straight from the sums
  int replicas;              // histograms: as many as fit, up to kReplicas
};
template <int N>
struct SelectBatchT {
  int n_jobs, block;
  int cleared;                      // the kernel before the sums is the clearing one
  int max_part_cols, total_items;   // sums_stream_kernel (its items), sums_flat_kernel (its pieces)
  int* status;
  int first_block[N];        // (row-blocks x parts before the job's own) apart from the wide records: a search stays within a few lines of the constant cache
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
  const SelectJob& J = B.job[blockIdx.x];
  if (J.head == nullptr) return;
  for (int i = threadIdx.x; i < J.replicas * (kBins1 / 4); i += kSelThreads) reinterpret_cast<uint4*>(J.head)[i] = make_uint4(0u, 0u, 0u, 0u);
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

// Behind the clearing kernel the sums have started only because everything before that one is complete (it signals
// after its wait, see launch_pdl): W may be read and the sums written at once, and only the additions to the histogram
// wait for the zeros.  A warp of its own waits early and lets the select take its seats.
// Orientation C, one CTA per row-block of every matrix, or per column range of one.
// (kParts as a template parameter: with the ranges as run-time values whole row-blocks took up to 2 us longer)
template <int N, bool kParts, int kTrip>
__global__ void __launch_bounds__(kSumThreads + 32)
sums_c_kernel(const __grid_constant__ SelectBatchT<N> B) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  const int jn = owner(B.first_block, B.n_jobs, static_cast<int>(blockIdx.x));
  const SelectJob& J = B.job[jn];
  const int at = static_cast<int>(blockIdx.x) - B.first_block[jn];
  const int b = kParts ? at / J.parts : at;
  const int c0 = kParts ? (at - b * J.parts) * J.part_cols : 0, c_end = kParts ? min(J.cols, c0 + J.part_cols) : J.cols;
  const uint16_t* wblk = J.W + static_cast<size_t>(b) * B.block * J.ldw;
  float* out = J.S + static_cast<size_t>(b) * J.cols;
  const bool count = J.head != nullptr;
  if (count) clear_bins(hist);
  if (!B.cleared) pdl_wait();
  __syncthreads();
  if (threadIdx.x >= kSumThreads) {
    pdl_wait();
    pdl_launch_dependents();
  } else if (J.vec) {
    for (int q = (c0 >> 3) + threadIdx.x; q < (c_end >> 3); q += kSumThreads) {
      float acc[8];
      sumsq8<kTrip>(wblk + (q << 3), B.block, J.ldw, acc);
      float4* dst = reinterpret_cast<float4*>(out + (q << 3));
      dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
      if (count) {
#pragma unroll
        for (int i = 0; i < 8; ++i) count_key(hist, acc[i]);
      }
    }
  } else {
    for (int g = c0 + threadIdx.x; g < c_end; g += kSumThreads) {
      const float S = group_sumsq_strided(wblk + g, B.block, J.ldw);
      out[g] = S;
      if (count) count_key(hist, S);
    }
  }
  if (!count) return;
  __syncthreads();
  pdl_wait();
  add_bins(hist, J.head + (blockIdx.x % J.replicas) * kBins1);
}

// The same for batches of many row-blocks: a CTA works through a run of items (a row-block, or a column range of
// it whose rows fit 24 KB) with the next item's rows on their way into a second buffer (bulk copies, one per row)
// while the current item is summed, and adds its histogram once per matrix.  One CTA per row-block, as above, loads,
// sums and leaves, and with 10 CTAs per SM coming and going a third of the time nothing was in flight: 72 matrices
// of a BERT-base stack (170 MB) 46 us, 3.7 TB/s.
template <int N>
__global__ void __launch_bounds__(kSumThreads)
sums_stream_kernel(const __grid_constant__ SelectBatchT<N> B) {
  extern __shared__ __align__(128) uint8_t s_raw[];          // [2][block rows][max_part_cols], then the histogram
  __shared__ __align__(8) uint64_t s_bar[2];
  const int d = B.block;
  const uint32_t buf_bytes = static_cast<uint32_t>((d * B.max_part_cols * 2 + 127) / 128 * 128);
  uint32_t* hist = reinterpret_cast<uint32_t*>(s_raw + 2 * buf_bytes);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    tc::mbar_init(tc::smem_u32(&s_bar[0]), 1);
    tc::mbar_init(tc::smem_u32(&s_bar[1]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  clear_bins(hist);
  const long long total = B.total_items;
  const int i0 = static_cast<int>(total * blockIdx.x / gridDim.x), i1 = static_cast<int>(total * (blockIdx.x + 1) / gridDim.x);
  // an item: matrix, row-block, first column and columns (first_block counts items here)
  auto locate = [&](int item, int& jn, int& b, int& c0, int& pc) {
    while (jn + 1 < B.n_jobs && B.first_block[jn + 1] <= item) ++jn;
    const SelectJob& J = B.job[jn];
    const int at = item - B.first_block[jn];
    b = at / J.parts;
    c0 = (at - b * J.parts) * J.part_cols;
    pc = min(J.part_cols, J.cols - c0);
  };
  auto fetch = [&](int jn, int b, int c0, int pc, int slot) {   // by warp 0
    const SelectJob& J = B.job[jn];
    const uint32_t bar = tc::smem_u32(&s_bar[slot]), dst = tc::smem_u32(s_raw) + static_cast<uint32_t>(slot) * buf_bytes;
    const uint32_t row_bytes = static_cast<uint32_t>(pc) * 2u;
    if (lane == 0) tc::mbar_arrive_expect_tx(bar, row_bytes * static_cast<uint32_t>(d));
    __syncwarp();
    const uint16_t* src = J.W + static_cast<size_t>(b) * d * J.ldw + c0;
    for (int r = lane; r < d; r += 32)
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                   ::"r"(dst + static_cast<uint32_t>(r) * row_bytes),
                     "l"(reinterpret_cast<uint64_t>(src + static_cast<size_t>(r) * J.ldw)), "r"(row_bytes), "r"(bar)
                   : "memory");
  };
  int jn = owner(B.first_block, B.n_jobs, i0), b, c0, pc;
  if (!B.cleared) pdl_wait();
  __syncthreads();
  locate(i0, jn, b, c0, pc);
  if (warp == 0 && i0 < i1) fetch(jn, b, c0, pc, 0);
  pdl_wait();
  pdl_launch_dependents();
  uint32_t parity[2] = {0u, 0u};
  for (int item = i0; item < i1; ++item) {
    const int slot = (item - i0) & 1;
    int jn2 = jn, b2 = 0, c2 = 0, pc2 = 0;
    if (item + 1 < i1) {
      locate(item + 1, jn2, b2, c2, pc2);
      if (warp == 0) fetch(jn2, b2, c2, pc2, slot ^ 1);       // (its readers are behind the barrier below)
    }
    if (!__syncthreads_and(tc::mbar_wait_suspended(tc::smem_u32(&s_bar[slot]), parity[slot], B.status) ? 1 : 0)) {
      // the rows never arrived: record it, hold the buffers a millisecond for copies still on their way, leave
      if (threadIdx.x == 0) atomicExch(B.status, BSP_ERR_TIMEOUT);
      const unsigned long long start = tc::global_timer_ns();
      while (tc::global_timer_ns() - start < tc::kQuietNs) __nanosleep(2000);
      return;
    }
    parity[slot] ^= 1u;
    const SelectJob& J = B.job[jn];
    const uint16_t* s_w = reinterpret_cast<const uint16_t*>(s_raw + static_cast<size_t>(slot) * buf_bytes);
    const bool count = J.head != nullptr;
    for (int k = threadIdx.x; k < (pc >> 3); k += kSumThreads) {
      SumSq8 sums;
#pragma unroll 8
      for (int r = 0; r < d; ++r) sums.add(*reinterpret_cast<const uint4*>(s_w + r * pc + (k << 3)));   // rows in increasing order: the defined decision quantity
      float acc[8];
      sums.get(acc);
      float4* dst = reinterpret_cast<float4*>(J.S + static_cast<size_t>(b) * J.cols + c0 + (k << 3));
      dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
      dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
      if (count) {
#pragma unroll
        for (int i = 0; i < 8; ++i) count_key(hist, acc[i]);
      }
    }
    __syncthreads();                                          // the buffer and, before a flush, the bins are complete
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (count && (item + 1 == i1 || jn2 != jn)) {
      add_bins(hist, J.head + (blockIdx.x % J.replicas) * kBins1);
      if (item + 1 < i1) {
        __syncthreads();
        clear_bins(hist);
        __syncthreads();
      }
    }
    jn = jn2; b = b2; c0 = c2; pc = pc2;
  }
}

// The same for batches of small row-blocks (short ones, or narrow matrices): a CTA works through a run of pieces (32 adjacent
// 8-column chunks of a matrix, its row-blocks one after the other), a warp a piece, and adds its histogram once per matrix.
// The warps meet nowhere else: a lane asks for 16 rows at once, and the 16 warps of an SM keep 128 KB on their way, where the
// streaming kernel's buffers would be half empty.  The percentiles of 72 matrices, streamed / this way: 12 layers of 256
// features in 8-row blocks 21.2 / 14.5 us, of 640 56.7 / 44.8, four of 768 32.9 / 26.9; 12 of 256 in 16-row blocks 18.0 /
// 13.6.  With larger row-blocks it is as fast by itself (12 of 768 in 16-row blocks 48.5 / 47.0), but between other work, with
// L2 full of what that has written, slower: the reads of 72 such matrices took 52 us there instead of 40.
constexpr int kFlatThreads = 256, kFlatPerSm = 2;
template <int N, bool kPast>
__global__ void __launch_bounds__(kFlatThreads, kFlatPerSm)
sums_flat_kernel(const __grid_constant__ SelectBatchT<N> B) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  clear_bins(hist);
  const long long total = B.total_items;
  const int i1 = static_cast<int>(total * (blockIdx.x + 1) / gridDim.x);
  int at = static_cast<int>(total * blockIdx.x / gridDim.x);
  int jn = owner(B.first_block, B.n_jobs, at);                // (first_block counts pieces here)
  if (!B.cleared) pdl_wait();
  __syncthreads();
  bool waited = false;
  for (; at < i1; ++jn) {
    const SelectJob& J = B.job[jn];
    const int first = B.first_block[jn], end = jn + 1 < B.n_jobs ? min(i1, B.first_block[jn + 1]) : i1;
    const int chunks = J.cols >> 3, all = J.n_blocks * chunks;
    const bool count = J.head != nullptr;
    for (int i = at + warp; i < end; i += kFlatThreads / 32) {
      const int c = (i - first) * 32 + lane;
      if (c < all) {
        const int b = c / chunks, k = c - b * chunks;
        float acc[8];
        sumsq8<16, kPast>(J.W + static_cast<size_t>(b) * B.block * J.ldw + (k << 3), B.block, J.ldw, acc);
        float4* dst = reinterpret_cast<float4*>(J.S + static_cast<size_t>(c) * 8);
        dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
        dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
        if (count) {
#pragma unroll
          for (int u = 0; u < 8; ++u) count_key(hist, acc[u]);
        }
      }
      if (!waited) {
        pdl_wait();
        pdl_launch_dependents();
        waited = true;
      }
    }
    at = end;
    if (!waited) {
      pdl_wait();
      pdl_launch_dependents();
      waited = true;
    }
    if (!count) continue;
    __syncthreads();
    add_bins(hist, J.head + (blockIdx.x % J.replicas) * kBins1);
    if (at < i1) {
      __syncthreads();
      clear_bins(hist);
      __syncthreads();
    }
  }
}

// Orientation R: one thread per group, neighbouring threads on neighbouring groups of a row.
constexpr int kSumRThreads = 256;
__global__ void __launch_bounds__(kSumRThreads + 32)
sums_r_kernel(const uint16_t* W, int rows, int per_row, int ldw, int block, int vec, float* S,
              uint32_t* head, int replicas) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  if (head != nullptr) clear_bins(hist);
  else pdl_wait();                                           // (no clearing kernel)
  __syncthreads();
  if (threadIdx.x >= kSumRThreads) {
    pdl_wait();
    pdl_launch_dependents();
  } else {
    const long long n = static_cast<long long>(rows) * per_row, step = static_cast<long long>(gridDim.x) * kSumRThreads;
    for (long long g = static_cast<long long>(blockIdx.x) * kSumRThreads + threadIdx.x; g < n; g += step) {
      const long long i = g / per_row;
      const int a = static_cast<int>(g - i * per_row);
      const float v = group_sumsq_contig(W + static_cast<size_t>(i) * ldw + static_cast<size_t>(a) * block, block, vec);
      S[g] = v;
      if (head != nullptr) count_key(hist, v);
    }
  }
  if (head == nullptr) return;
  __syncthreads();
  pdl_wait();
  add_bins(hist, head + (blockIdx.x % replicas) * kBins1);
}

// ---------------------------------------------------------------------------------------- select
// The bin of a histogram that holds the want-th smallest key (1-based) and the rank inside that bin; the whole
// CTA takes part and gets the answer.  A warp adds up a 32nd of the bins, every warp adds up the sums before its own,
// and the one that holds the answer scans its bins.
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
  uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? s_sum[lane] : 0u);
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
__device__ __forceinline__ void for_matching(const uint32_t* keys, long long n, int above, uint32_t prefix, F f) {
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

__device__ __forceinline__ uint32_t ld_cluster(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
// The least float whose square, rounded, reaches the sum of squares with these bits.
__device__ __forceinline__ float threshold_of(uint32_t bits) {
  const float s_r = __uint_as_float(bits);
  float t = __fsqrt_rn(s_r);
  while (__fmul_rn(t, t) < s_r) t = __uint_as_float(__float_as_uint(t) + 1u);  // next float up (t >= 0)
  return t;
}

template <int N>
__global__ void __launch_bounds__(kSelThreads)
select_kernel(const __grid_constant__ SelectBatchT<N> B) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  __shared__ uint32_t s_sum[32];
  __shared__ uint32_t s_pick[2];
  __shared__ uint32_t s_n, s_last_n, s_last[32], s_len[kSelMaxCluster];
  extern __shared__ uint32_t s_list[];                       // [kList], then in CTA 0 [kCandidates]
  uint32_t* s_cand = s_list + kList;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = tc::cluster_rank(), n_cta = tc::cluster_size();
  const SelectJob& J = B.job[blockIdx.x / n_cta];
  const uint32_t* keys = reinterpret_cast<const uint32_t*>(J.S);
  const long long n = J.n;
  if (threadIdx.x == 0) s_n = s_last_n = 0u;
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  pdl_wait();
  pdl_launch_dependents();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");   // every CTA of the cluster has started
  if (J.r <= 0) {                                            // the same for the whole cluster
    if (rank == 0 && threadIdx.x == 0) *J.out = -1.0f;
    return;
  }
  Pick p{0u, static_cast<uint32_t>(J.r)};
  uint32_t prefix = 0u;
  uint32_t found = 0xffffffffu;                              // keys on the lists; all ones: read them all
  if (J.head != nullptr) {
    // this CTA's first keys are on their way while the histogram is looked at
    const uint4* v4 = reinterpret_cast<const uint4*>(keys);
    const long long n4 = n >> 2, step = static_cast<long long>(n_cta) * kSelThreads;
    long long i0 = static_cast<long long>(rank) * kSelThreads;
    uint32_t k[4 * kSelLoads];
    auto load = [&]() {
#pragma unroll
      for (int u = 0; u < kSelLoads; ++u) {
        uint4 v = make_uint4(~0u, ~0u, ~0u, ~0u);             // (no key: the sign bit is set)
        if (i0 + u * step + threadIdx.x < n4) v = __ldcg(v4 + i0 + u * step + threadIdx.x);
        k[4 * u] = v.x; k[4 * u + 1] = v.y; k[4 * u + 2] = v.z; k[4 * u + 3] = v.w;
      }
    };
    load();
    uint4 h[kReplicas];
#pragma unroll
    for (int r = 0; r < kReplicas; ++r)
      h[r] = r < J.replicas ? __ldcg(reinterpret_cast<const uint4*>(J.head + r * kBins1) + threadIdx.x) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int r = 1; r < kReplicas; ++r) { h[0].x += h[r].x; h[0].y += h[r].y; h[0].z += h[r].z; h[0].w += h[r].w; }
    reinterpret_cast<uint4*>(hist)[threadIdx.x] = h[0];
    static_assert(kBins1 == 4 * kSelThreads, "a 16-byte piece of the histogram per thread");
    __syncthreads();
    p = pick_bin<kBins1>(hist, p.want, s_sum, s_pick);
    prefix = p.bin;
    if (rank == 0) {                                         // the bins of the digits to come
      hist[threadIdx.x] = 0u;
      if (threadIdx.x < kBins3) hist[kBins2 + threadIdx.x] = 0u;
    }
    const uint32_t in_bin = prefix << (kBits2 + kBits3);
    for (;;) {
      // (32 warps share the issue slots, so instructions count: a warp's places on the list come from one addition)
      uint32_t hit = 0u;
#pragma unroll
      for (int u = 0; u < kSelLoads; ++u) {
        if (u > 0 && i0 + u * step + (threadIdx.x & ~31u) >= n4) break;   // none of the warp's lanes has a key here
#pragma unroll
        for (int i = 4 * u; i < 4 * u + 4; ++i)
          if ((k[i] ^ in_bin) < (1u << (kBits2 + kBits3))) hit |= 1u << i;
      }
      if (__any_sync(0xffffffffu, hit != 0u)) {
        const uint32_t mine = __popc(hit);
        uint32_t incl = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t up = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += up;
        }
        uint32_t at = 0u;
        if (lane == 31) at = atomicAdd(&s_n, incl);
        const uint32_t end = __shfl_sync(0xffffffffu, at + incl, 31);
        at = __shfl_sync(0xffffffffu, at, 31) + incl - mine;
        if (end <= kList) {                                  // (a list that overflows is not used)
          // predicated by hand: as branches, the 24 stores of a warp that keeps ten keys took 0.8 us
          uint32_t to = tc::smem_u32(s_list + at);
#pragma unroll
          for (int i = 0; i < 4 * kSelLoads; ++i)
            asm volatile("{\n.reg .pred p;\n.reg .b32 t;\nand.b32 t, %2, %3;\nsetp.ne.u32 p, t, 0;\n@p st.shared.u32 [%0], %1;\n@p add.u32 %0, %0, 4;\n}"
                         : "+r"(to) : "r"(k[i]), "r"(hit), "r"(1u << i) : "memory");
        }
      }
      i0 += kSelLoads * step;
      if (i0 >= n4) break;
      load();
    }
    if (rank == 0 && threadIdx.x < static_cast<unsigned>(n & 3)) {   // the last n mod 4 keys
      const uint32_t tail = __ldcg(keys + (n4 << 2) + threadIdx.x);
      if ((tail >> (kBits2 + kBits3)) == prefix) {
        const uint32_t at = atomicAdd(&s_n, 1u);
        if (at < kList) s_list[at] = tail;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) st_cluster(tc::map_to_cta(tc::smem_u32(&s_len[rank]), 0u), s_n);
    tc::cluster_sync();                                          // the lists and their lengths are complete
    if (rank == 0) {
      const uint32_t length = lane < static_cast<int>(n_cta) ? s_len[lane] : 0u;
      found = __reduce_add_sync(0xffffffffu, length);
      if (__any_sync(0xffffffffu, length > kList) || found > kCandidates) {
        found = 0xffffffffu;
      } else {
        // eight warps a list, four lists at a time; a list's keys go behind those of the lists before it
        for (uint32_t q = warp & 3u; q < n_cta; q += 4u) {
          const uint32_t len = __shfl_sync(0xffffffffu, length, static_cast<int>(q));
          const uint32_t at = __reduce_add_sync(0xffffffffu, lane < static_cast<int>(q) ? length : 0u);
          const uint32_t src = tc::map_to_cta(tc::smem_u32(s_list), q);
          for (uint32_t i0 = static_cast<uint32_t>((warp >> 2) * 32 + lane); i0 < len; i0 += 4 * (kSelThreads / 4)) {
            uint32_t c[4];
#pragma unroll
            for (uint32_t u = 0; u < 4u; ++u) c[u] = i0 + u * (kSelThreads / 4) < len ? ld_cluster(src + 4u * (i0 + u * (kSelThreads / 4))) : 0u;
#pragma unroll
            for (uint32_t u = 0; u < 4u; ++u)
              if (i0 + u * (kSelThreads / 4) < len) s_cand[at + i0 + u * (kSelThreads / 4)] = c[u];
          }
        }
      }
    }
  } else {
    if (rank == 0) {
      clear_bins(hist);
      __syncthreads();
      for_matching(keys, n, 31, 0u, [&](uint32_t k) { atomicAdd(&hist[k >> (kBits2 + kBits3)], 1u); });
      __syncthreads();
      p = pick_bin<kBins1>(hist, p.want, s_sum, s_pick);
      prefix = p.bin;
      hist[threadIdx.x] = 0u;
      if (threadIdx.x < kBins3) hist[kBins2 + threadIdx.x] = 0u;
    }
    tc::cluster_sync();
  }
  if (rank != 0) {
    tc::cluster_arrive_relaxed();
    tc::cluster_wait();                                          // CTA 0 has read this CTA's list
    return;
  }
  // the next digit over the listed keys or all of them; then a warp ranks the few keys that are left, or the last
  // digit has bins of its own
  __syncthreads();
  tc::cluster_arrive_relaxed();                                  // (the lists have been read: the other CTAs may leave)
  auto over_keys = [&](int above, uint32_t upper, auto f) {
    if (found != 0xffffffffu) {
      for (uint32_t i = threadIdx.x; i < found; i += kSelThreads)
        if ((s_cand[i] >> above) == upper) f(s_cand[i]);
    } else {
      for_matching(keys, n, above, upper, f);
    }
  };
  over_keys(kBits2 + kBits3, prefix, [&](uint32_t k) { atomicAdd(&hist[(k >> kBits3) & (kBins2 - 1)], 1u); });
  __syncthreads();
  p = pick_bin<kBins2>(hist, p.want, s_sum, s_pick);
  prefix = (prefix << kBits2) | p.bin;
  over_keys(kBits3, prefix, [&](uint32_t k) {
    const uint32_t at = atomicAdd(&s_last_n, 1u);
    if (at < 32u) s_last[at] = k;
  });
  __syncthreads();
  const uint32_t left = s_last_n;
  if (left <= 32u) {
    if (warp == 0) {
      const uint32_t k = lane < static_cast<int>(left) ? s_last[lane] : ~0u;
      uint32_t less = 0u, upto = 0u;
      for (uint32_t j = 0; j < left; ++j) {
        const uint32_t o = __shfl_sync(0xffffffffu, k, static_cast<int>(j));
        less += o < k ? 1u : 0u;
        upto += o <= k ? 1u : 0u;
      }
      if (lane < static_cast<int>(left) && less < p.want && p.want <= upto) *J.out = threshold_of(k);   // (equal keys agree)
    }
  } else {
    over_keys(kBits3, prefix, [&](uint32_t k) { atomicAdd(&hist[kBins2 + (k & (kBins3 - 1))], 1u); });
    __syncthreads();
    p = pick_bin<kBins3>(hist + kBins2, p.want, s_sum, s_pick);
    if (threadIdx.x == 0) *J.out = threshold_of((prefix << kBits3) | p.bin);
  }
  tc::cluster_wait();
}

// ------------------------------------------------------------ select where counts do not fit 32 bits (select_large)
// A launch counts one digit over all keys (in shared memory per CTA, whose keys do fit 32 bits), a launch of one CTA
// picks the digit that holds the answer.  Bound by the passes over the sums.
struct LargeState {                                          // in the part of the workspace that holds flags elsewhere
  unsigned long long want, hist[kBins1];
  uint32_t prefix;
};
__global__ void __launch_bounds__(kSelThreads)
large_start_kernel(LargeState* state, long long r) {
  pdl_wait();
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < kBins1; i += kSelThreads) state->hist[i] = 0ull;
  if (threadIdx.x == 0) {
    state->want = static_cast<unsigned long long>(r);
    state->prefix = 0u;
  }
}
__global__ void __launch_bounds__(256)
large_count_kernel(const uint32_t* keys, long long n, int above, int bits, LargeState* state) {
  __shared__ __align__(16) uint32_t hist[kBins1];
  clear_bins(hist);
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  const uint32_t prefix = state->prefix, mask = (1u << bits) - 1u;
  const int shift = above - bits;
  const long long n4 = n >> 2, step = static_cast<long long>(gridDim.x) * 256;
  auto count = [&](uint32_t k) {
    if ((k >> above) == prefix) atomicAdd(&hist[(k >> shift) & mask], 1u);
  };
  for (long long i = static_cast<long long>(blockIdx.x) * 256 + threadIdx.x; i < n4; i += step) {
    const uint4 v = ld_global(reinterpret_cast<const uint4*>(keys) + i);
    count(v.x); count(v.y); count(v.z); count(v.w);
  }
  if (blockIdx.x == 0 && threadIdx.x < static_cast<unsigned>(n & 3)) count(ld_global(keys + (n4 << 2) + threadIdx.x));
  __syncthreads();
  for (int i = threadIdx.x; i < kBins1; i += 256)
    if (hist[i] != 0u) atomicAdd(&state->hist[i], static_cast<unsigned long long>(hist[i]));
}
__global__ void __launch_bounds__(kSelThreads)
large_pick_kernel(LargeState* state, int bits, long long r, float* out) {
  __shared__ unsigned long long hist[kBins1];
  pdl_wait();
  pdl_launch_dependents();
  for (int i = threadIdx.x; i < kBins1; i += kSelThreads) {
    hist[i] = state->hist[i];
    state->hist[i] = 0ull;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  unsigned long long want = state->want;
  uint32_t bin = 0u;
  if (r > 0)
    for (; want > hist[bin]; ++bin) want -= hist[bin];
  state->want = want;
  state->prefix = (state->prefix << bits) | bin;
  if (out != nullptr) *out = r > 0 ? threshold_of(state->prefix) : -1.0f;
}
int launch_select_large(const SelectJob& J, void* state_bytes, int sms, cudaStream_t s) {
  LargeState* state = static_cast<LargeState*>(state_bytes);
  BSP_CUDA_TRY(launch_pdl(large_start_kernel, dim3(1), dim3(kSelThreads), 0, s, state, J.r));
  int above = kBits1 + kBits2 + kBits3;
  for (const int bits : {kBits1, kBits2, kBits3}) {
    BSP_CUDA_TRY(launch_pdl(large_count_kernel, dim3(4 * sms), dim3(256), 0, s, reinterpret_cast<const uint32_t*>(J.S), J.n, above, bits, state));
    above -= bits;
    BSP_CUDA_TRY(launch_pdl(large_pick_kernel, dim3(1), dim3(kSelThreads), 0, s, state, bits, J.r, above == 0 ? J.out : nullptr));
  }
  return BSP_OK;
}

// r = floor(G * (1 - 1/c)) in float64, as the definition states it
long long groups_to_remove(long long groups, double rate) {
  return static_cast<long long>(static_cast<double>(groups) * (1.0 - 1.0 / rate));
}

// The histograms and lists of the select count in 32 bits.
bool select_large(long long groups) { return groups >= (1LL << 32); }

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
  // the region of the flags: one byte per group
  const size_t fit = (L.sumsq_off - L.keep_off) / (kBins1 * sizeof(uint32_t));
  J.replicas = fit < kReplicas ? static_cast<int>(fit) : kReplicas;
  if (fit > 0 && !select_large(groups)) J.head = reinterpret_cast<uint32_t*>(base + L.keep_off);
  return J;
}

// CTAs per matrix: as many as fit the GPU at once (one per SM: 1024 threads of 48 registers), up to the portable
// cluster size, but not so many that a CTA has fewer than 2048 keys.
int select_cluster(int n_jobs, long long largest, int sms) {
  int c = kSelMaxCluster;
  while (c > 1 && (static_cast<long long>(n_jobs) * c > sms || largest < 2048LL * c)) c >>= 1;
  return c;
}
template <int N>
int launch_select(const SelectBatchT<N>& B, int sms, cudaStream_t s) {
  long long largest = 0;
  for (int i = 0; i < B.n_jobs; ++i)
    if (B.job[i].n > largest) largest = B.job[i].n;
  const int c = select_cluster(B.n_jobs, largest, sms);
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, select_kernel<N>, kSelSmem));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(B.n_jobs * c));
  cfg.blockDim = dim3(kSelThreads);
  cfg.dynamicSmemBytes = kSelSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = c;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  BSP_CUDA_TRY(cudaLaunchKernelEx(&cfg, select_kernel<N>, B));
  return BSP_OK;
}

template <int N, bool kParts>
auto* sums_kernel(int trip) {
  return trip == 4 ? sums_c_kernel<N, kParts, 4> : trip == 8 ? sums_c_kernel<N, kParts, 8> : trip == 16 ? sums_c_kernel<N, kParts, 16>
                                                                                                      : sums_c_kernel<N, kParts, 32>;
}

// Sums of a batch in orientation C, where every matrix can be read in 16-byte pieces: warps on their own from 54 KB per SM on
// where an item of the streaming kernel would be 16 KB or less on average, streaming where there are several items for every
// CTA; one CTA per row-block otherwise (its single trip to memory is what a small batch needs: one layer of 256 features 9.9
// us, 10.4 by warps).  From 324 KB per SM on the rows pass L1 by.  Percentiles of 8-row blocks, with the preparation behind them,
// streamed / by warps through L1 / past it: 4 layers of 512 features (166 KB per SM) 45.7 / 43.3 / 43.6 us, 12 of 400 (304 KB)
// 80.6 / 72.3 / 73.3, 4 of 768 (374) 71.9 / 72.3 / 73.3, 6 of 640 (389) 83.4 / 83.3 / 82.8, 12 of 576 (630) 129.3 / 115.6 /
// 114.5, 12 of 640 (778) 143.0 / 141.4 / 134.6, 12 of 768 (1121) 184.5 / 185.5 / 176.2; in 16-row blocks 12 of 256 (125) 37.1 /
// 34.0 / 34.3.
template <int N>
int launch_sums_c(SelectBatchT<N>& B, int sms, cudaStream_t s) {
  const int max_cols = kSumRowBytes / (2 * B.block) / 8 * 8;
  bool stream = max_cols >= 8;
  int blocks = 0, items = 0;
  bool narrow = true;                                       // a matrix's chunks are numbered in 32 bits
  long long bytes = 0, pieces = 0;
  B.max_part_cols = 0;
  for (int i = 0; i < B.n_jobs; ++i) {
    SelectJob& J = B.job[i];
    stream = stream && J.vec;
    blocks += J.n_blocks;
    if (!stream) continue;
    J.parts = (J.cols + max_cols - 1) / max_cols;
    J.part_cols = ((J.cols + J.parts - 1) / J.parts + 7) / 8 * 8;
    J.parts = (J.cols + J.part_cols - 1) / J.part_cols;
    items += J.n_blocks * J.parts;
    bytes += 2 * J.n * B.block;
    pieces += (J.n / 8 + 31) / 32;
    narrow = narrow && J.n < (1LL << 33);
    if (J.part_cols > B.max_part_cols) B.max_part_cols = J.part_cols;
  }
  if (stream && narrow && bytes >= 54LL * 1024 * sms && bytes <= 16LL * 1024 * items && pieces < (1LL << 31)) {
    int at = 0;
    for (int i = 0; i < B.n_jobs; ++i) { B.first_block[i] = at; at += static_cast<int>((B.job[i].n / 8 + 31) / 32); }
    B.total_items = at;
    BSP_CUDA_TRY(launch_pdl(bytes >= 324LL * 1024 * sms ? sums_flat_kernel<N, true> : sums_flat_kernel<N, false>, dim3(kFlatPerSm * sms),
                            dim3(kFlatThreads), 0, s, B));
    return BSP_OK;
  }
  if (stream && items >= 2 * kSumPerSm * sms) {
    TcDevice* dev = tc_device();
    if (dev == nullptr) return BSP_ERR_CUDA;
    B.status = dev->status;
    B.total_items = items;
    int at = 0;
    for (int i = 0; i < B.n_jobs; ++i) { B.first_block[i] = at; at += B.job[i].n_blocks * B.job[i].parts; }
    const size_t smem = 2 * round_up(static_cast<size_t>(B.block) * B.max_part_cols * 2, 128) + kBins1 * 4;
    static OncePerDevice once;
    BSP_TRY(allow_dynamic_smem(once, sums_stream_kernel<N>, 2 * kSumRowBytes + 256 + kBins1 * 4));
    BSP_CUDA_TRY(launch_pdl(sums_stream_kernel<N>, dim3(kSumPerSm * sms), dim3(kSumThreads), smem, s, B));
    return BSP_OK;
  }
  // few row-blocks: cut into ranges of a piece per thread (narrower ones cost more in histograms than they gain: 9.6 ->
  // 11.6 us for 768 x 768)
  int at = 0;
  bool parts = false;
  for (int i = 0; i < B.n_jobs; ++i) {
    SelectJob& J = B.job[i];
    const int width = kSumThreads * (J.vec ? 8 : 1);
    J.part_cols = blocks < sms && width < J.cols ? width : J.cols;
    J.parts = (J.cols + J.part_cols - 1) / J.part_cols;
    parts = parts || J.parts > 1;
    B.first_block[i] = at;
    at += J.n_blocks * J.parts;
  }
  const int trip = rows_per_trip(B.block, at, 4, 2, sms);     // (CTAs of five warps with 88 and 152 registers)
  auto* kernel = parts ? sums_kernel<N, true>(trip) : sums_kernel<N, false>(trip);
  BSP_CUDA_TRY(launch_pdl(kernel, dim3(at), dim3(kSumThreads + 32), 0, s, B));
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
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms;
  st = sm_count(&sms);
  if (st != BSP_OK) return st;
  SelectBatchT<1> B;
  B.n_jobs = 1;
  B.block = block;
  B.job[0] = select_job(W, cols, ldw, nb, ng, rate, ws, threshold_out);
  B.cleared = B.job[0].head != nullptr ? 1 : 0;
  if (B.cleared) BSP_CUDA_TRY(launch_pdl(select_clear_kernel<1>, dim3(1), dim3(kSelThreads), 0, s, B));
  if (orient == BSP_ORIENT_C) {
    st = launch_sums_c(B, sms, s);
    if (st != BSP_OK) return st;
  } else {
    // (at most four CTAs per SM, since every one adds a histogram of its own in the end)
    const long long ctas = (groups + kSumRThreads - 1) / kSumRThreads;
    BSP_CUDA_TRY(launch_pdl(sums_r_kernel, dim3(static_cast<unsigned>(ctas < 4 * sms ? ctas : 4 * sms)), dim3(kSumRThreads + 32), 0, s, B.job[0].W, rows, nb,
                            ldw, block, contig_vec(W, ldw, block), B.job[0].S, B.job[0].head,
                            B.job[0].replicas));
  }
  if (select_large(groups)) return launch_select_large(B.job[0], static_cast<char*>(ws) + L.keep_off, sms, s);
  return launch_select(B, sms, s);
}

extern "C" int bsp_percentile_threshold_batched(const bsp_layer_job* jobs, int n_jobs, int block, const double* rates,
                                                void* stream) {
  using namespace bsp;
  if (jobs == nullptr || rates == nullptr || n_jobs <= 0 || block <= 0) return BSP_ERR_ARG;
  if (n_jobs > 4096) return BSP_ERR_UNSUPPORTED;
  bool large = false;
  for (int i = 0; i < n_jobs; ++i) {                       // everything is checked before the first launch
    const bsp_layer_job& u = jobs[i];
    int st = check_matrix_args(u.W, u.rows, u.cols, u.ldw, block, BSP_ORIENT_C);
    if (st != BSP_OK) return st;
    if (u.threshold_dev == nullptr || u.ws == nullptr || !aligned_to(u.ws, 256)) return BSP_ERR_ARG;
    if (!(rates[i] >= 1.0)) return BSP_ERR_ARG;
    if (u.ws_bytes < ws_layout(u.rows / block, u.cols).total) return BSP_ERR_WORKSPACE;
    large = large || select_large(static_cast<long long>(u.rows / block) * u.cols);
  }
  if (large) {                                             // (a workspace of 20 GB each: one after the other)
    for (int i = 0; i < n_jobs; ++i) {
      const bsp_layer_job& u = jobs[i];
      BSP_TRY(bsp_percentile_threshold(u.W, u.rows, u.cols, u.ldw, block, BSP_ORIENT_C, rates[i], const_cast<float*>(u.threshold_dev),
                                       u.ws, u.ws_bytes, stream));
    }
    return BSP_OK;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int sms;
  int st = sm_count(&sms);
  if (st != BSP_OK) return st;
  SelectBatchT<kSelectBatch> B;
  for (int j0 = 0; j0 < n_jobs; j0 += kSelectBatch) {
    B.n_jobs = n_jobs - j0 < kSelectBatch ? n_jobs - j0 : kSelectBatch;
    B.block = block;
    for (int i = 0; i < B.n_jobs; ++i) {
      const bsp_layer_job& u = jobs[j0 + i];
      B.job[i] = select_job(u.W, u.cols, u.ldw, u.rows / block, u.cols, rates[j0 + i], u.ws, const_cast<float*>(u.threshold_dev));
    }
    B.cleared = 1;
    BSP_CUDA_TRY(launch_pdl(select_clear_kernel<kSelectBatch>, dim3(B.n_jobs), dim3(kSelThreads), 0, s, B));
    st = launch_sums_c(B, sms, s);
    if (st != BSP_OK) return st;
    st = launch_select(B, sms, s);
    if (st != BSP_OK) return st;
  }
  return BSP_OK;
}
