// bsp_prune_pack, bsp_apply_mask: Algorithm 1's keep decision per
// group, Algorithm 2's mask, and the compaction of the kept groups into the canonical
// block-structured storage (Section 3.1).
//
// Launches per pack: (1) one CTA per block decides its groups and counts the kept ones,
// (2) CTAs per block turn the counts before theirs into blk_ptr, list the kept indices in
// ascending order and gather the dense tile of kept values.  W is read from HBM once by (1);
// (2) re-reads it from L2.  Orientation C with 8-element alignment runs the vectorised
// two-stage kernels of bsp_fused.cu, orientation R goes by segments of a strip; this file holds
// the latter, the generic kernels, the keep-count kernel and the entry points.
#include <mutex>

#include "bsp_common.cuh"

namespace bsp {
namespace {

constexpr int kPackThreads = 256;
// Up to here the keep-count select ranks the groups of a block.  The call, ranking against digits: 768 x 64 in 16-row blocks
// 5.2 against 8.2 us, 768 x 192 7.0 against 7.6, 128 x 8103 in strips of three 24 against 40; 2048 x 256 12.3 against 9.0.
constexpr int kRankGroups = 192;
static_assert(kRankGroups <= 256, "a block of few groups is one segment");
constexpr int kSegment = 256;          // groups of a strip that one CTA packs (orientation R)
// Segments of a matrix up to which strips are packed by them: every CTA adds up the counts before its own.  With many
// strips, 4000 segments (1000 x 1000 in single columns) 26 us, 30 without; 8192 equal; 13870 (280 x 6935) 67, 51 without.
// With few, a CTA per strip leaves more to lose: 5115 (7928 x 2640 in strips of 16) 37, 57 without.
constexpr int kMaxSegments = 4096, kFewStrips = 512, kMaxSegmentsFew = 16384;

struct Geometry {
  int rows, cols, ldw, block, orient, n_blocks, n_groups;
  int vec;            // widest vector that reads whole pieces: of a group (R), of 8 adjacent columns (C)
};

// Pointer to element 0 of group g of block b, and the stride between the group's elements.
__device__ __forceinline__ const uint16_t* group_ptr(const uint16_t* W, const Geometry& G, int b, int g,
                                                     size_t* stride) {
  if (G.orient == BSP_ORIENT_C) {
    *stride = G.ldw;
    return W + static_cast<size_t>(b) * G.block * G.ldw + g;
  }
  *stride = 1;
  return W + static_cast<size_t>(g) * G.ldw + static_cast<size_t>(b) * G.block;
}

// Position of group g of block b in a per-group array ([rows/d, cols] for C, [rows, cols/h] for R).
__device__ __forceinline__ size_t group_slot(const Geometry& G, int b, int g) {
  return G.orient == BSP_ORIENT_C ? static_cast<size_t>(b) * G.n_groups + g
                                  : static_cast<size_t>(g) * G.n_blocks + b;
}

// Float32 sum of squares of group g of block b.
__device__ __forceinline__ float group_sum(const uint16_t* W, const Geometry& G, int b, int g) {
  size_t stride;
  const uint16_t* p = group_ptr(W, G, b, g, &stride);
  return G.orient == BSP_ORIENT_C ? group_sumsq_strided8(p, G.block, stride) : group_sumsq_contig(p, G.block, G.vec);
}

// n elements from stride to stride, four loads in flight.
template <class T>
__device__ __forceinline__ void copy_strided(T* dst, size_t dst_stride, const T* src, size_t src_stride, int n) {
  int left = n;
#pragma unroll 1
  for (; left >= 4; left -= 4) {
    T v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u, src += src_stride) v[u] = ld_global(src);
#pragma unroll
    for (int u = 0; u < 4; ++u, dst += dst_stride) *dst = v[u];
  }
#pragma unroll 1
  for (; left > 0; --left, src += src_stride, dst += dst_stride) *dst = ld_global(src);
}

// (1a) threshold mode, one CTA per block.
template <int T>
__global__ void __launch_bounds__(T)
flags_threshold_kernel(const uint16_t* W, Geometry G, float threshold,
                       const float* threshold_dev, uint8_t* keep,
                       int32_t* counts) {
  __shared__ int s_count;
  if (threadIdx.x == 0) s_count = 0;
  pdl_wait();
  pdl_launch_dependents();
  __syncthreads();
  const float t = threshold_dev ? *threshold_dev : threshold;
  const bool keep_all = t < 0.0f;
  const float t2 = __fmul_rn(t, t);
  const int b = blockIdx.x;
  int local = 0;
  for (int g = threadIdx.x; g < G.n_groups; g += blockDim.x) {
    const float S = group_sum(W, G, b, g);
    const bool k = keep_all || (S > t2);
    keep[group_slot(G, b, g)] = k ? 1 : 0;
    local += k ? 1 : 0;
  }
  local = warp_sum(local);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(&s_count, local);
  __syncthreads();
  if (threadIdx.x == 0) counts[b] = s_count;
}

// (1b) keep-count mode, one CTA per block: the keep_count largest sums, ties towards the lower index.  The
// block's sums stay in shared memory as float bit patterns (monotone, they are not negative); a radix
// select of three digits finds the smallest kept one, and a scan in index order decides which of its equals
// are kept.  O(groups) work per digit; ranking every sum against every other one (O(groups^2)) took
// 0.5-1 ms on the larger matrices.
// Blocks of 512 groups or more get 512 threads (orientation C, whose rows in flight take 64 registers) or 1024 (R): the
// digits are passes over the keys, and a GPU that is still busy with the launch before puts several of the smaller CTAs on
// one SM, where they share its issue slots.  Norms, packing and layout together, against 256 threads: 16 strips of 3072
// groups 105 -> 46 us, 64 strips of 768 28 -> 16, 11 row-blocks of 3072 44 -> 33, 192 of 768 22.6 -> 18.5.
constexpr int kTopkDigit = 11;                       // 31 bits = 11 + 10 + 10
constexpr int kTopkBins = 1 << kTopkDigit;
// (CTAs per SM that leave the registers for ten rows of eight columns in flight; left alone the compiler takes 32 and
// spills, and a block of 256 rows 2 x as long.)
template <int T>
__global__ void __launch_bounds__(T, T == 1024 ? 2 : T == 512 ? 3 : 6)
flags_topk_kernel(const uint16_t* W, Geometry G, int keep_count,
                  uint8_t* keep, int32_t* counts, int32_t* seg_counts) {
  extern __shared__ uint32_t s_key[];                // [n_groups]
  __shared__ int s_seg[BSP_TOPK_MAX_GROUPS / kSegment];
  __shared__ uint32_t hist[kTopkBins];
  __shared__ int s_warp[32];
  __shared__ uint32_t s_pick[3];
  constexpr int kPer = kTopkBins / T;
  const int b = blockIdx.x, n = G.n_groups;
  pdl_wait();
  pdl_launch_dependents();
  if (keep_count <= 0 || keep_count >= n) {
    const uint8_t all = keep_count > 0 ? 1 : 0;
    for (int g = threadIdx.x; g < n; g += T) keep[group_slot(G, b, g)] = all;
    if (threadIdx.x == 0) counts[b] = all ? n : 0;
    const int segments = (n + kSegment - 1) / kSegment;
    if (seg_counts != nullptr && static_cast<int>(threadIdx.x) < segments)
      seg_counts[b * segments + threadIdx.x] = all ? min(kSegment, n - static_cast<int>(threadIdx.x) * kSegment) : 0;
    return;
  }
  if (threadIdx.x < BSP_TOPK_MAX_GROUPS / kSegment) s_seg[threadIdx.x] = 0;
  if (G.orient == BSP_ORIENT_C && G.vec == 8) {
    for (int q = threadIdx.x; q < (n >> 3); q += T) {
      float acc[8];
      sumsq8<0>(W + static_cast<size_t>(b) * G.block * G.ldw + (q << 3), G.block, G.ldw, acc);
#pragma unroll
      for (int i = 0; i < 8; ++i) s_key[(q << 3) + i] = __float_as_uint(acc[i]);
    }
  } else {
    for (int g = threadIdx.x; g < n; g += T) s_key[g] = __float_as_uint(group_sum(W, G, b, g));
  }
  uint32_t want = static_cast<uint32_t>(n - keep_count + 1);   // the smallest kept sum is the want-th smallest
  uint32_t prefix = 0u;
  int shift = 31;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    const int bits = pass == 0 ? kTopkDigit : 10;
    const int above = shift;                         // bits above `above` are decided
    shift -= bits;
#pragma unroll
    for (int i = 0; i < kPer; ++i) hist[threadIdx.x + i * T] = 0u;
    __syncthreads();
    const uint32_t mask = (1u << bits) - 1u;
    for (int g = threadIdx.x; g < n; g += T) {
      const uint32_t u = s_key[g];
      if (above >= 31 || (u >> above) == prefix) atomicAdd(&hist[(u >> shift) & mask], 1u);
    }
    __syncthreads();
    uint32_t c[kPer], mine = 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) { c[i] = hist[threadIdx.x * kPer + i]; mine += c[i]; }
    int total;
    uint32_t before = static_cast<uint32_t>(block_exclusive_scan(static_cast<int>(mine), s_warp, &total));
    if (before < want && want <= before + mine) {    // exactly one thread
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        if (before < want && want <= before + c[i]) { s_pick[0] = threadIdx.x * kPer + i; s_pick[1] = want - before; s_pick[2] = c[i]; }
        before += c[i];
      }
    }
    __syncthreads();
    prefix = (prefix << bits) | s_pick[0];
    want = s_pick[1];
    __syncthreads();
  }
  // groups above the smallest kept sum stay; of the e groups equal to it the first e - want + 1 do
  // (the select counted want - 1 of them as smaller): all of them in most cases, which takes no ranking
  const bool all_equals = want == 1u;
  const int equals_kept = static_cast<int>(s_pick[2] - want) + 1;
  int seen = 0;
  for (int g0 = 0; g0 < n; g0 += T) {
    const int g = g0 + threadIdx.x;
    const uint32_t u = g < n ? s_key[g] : 0u;
    const int eq = g < n && u == prefix ? 1 : 0;
    int rank = 0;
    if (!all_equals) {
      int round;
      rank = seen + block_exclusive_scan(eq, s_warp, &round);
      seen += round;
    }
    const bool k = g < n && (u > prefix || (eq && rank < equals_kept));
    if (g < n) keep[group_slot(G, b, g)] = k ? 1 : 0;
    if (seg_counts != nullptr) {                     // (a warp's groups are in one segment)
      const unsigned kept = __ballot_sync(0xffffffffu, k);
      if ((threadIdx.x & 31) == 0 && kept != 0u) atomicAdd(&s_seg[g / kSegment], __popc(kept));
    }
  }
  if (threadIdx.x == 0) counts[b] = keep_count;
  if (seg_counts != nullptr) {
    __syncthreads();
    const int segments = (n + kSegment - 1) / kSegment;
    if (static_cast<int>(threadIdx.x) < segments) seg_counts[b * segments + threadIdx.x] = s_seg[threadIdx.x];
  }
}

// The same for blocks of few groups, by ranking every sum against every other one: the digits' passes over 2048 bins
// cost more there.
__global__ void __launch_bounds__(kRankGroups)
flags_rank_kernel(const uint16_t* W, Geometry G, int keep_count, uint8_t* keep, int32_t* counts, int32_t* seg_counts) {
  __shared__ float s_S[kRankGroups];
  const int b = blockIdx.x, g = threadIdx.x, n = G.n_groups;
  pdl_wait();
  pdl_launch_dependents();
  const float mine = g < n ? group_sum(W, G, b, g) : 0.0f;
  s_S[g] = mine;
  __syncthreads();
  if (g < n) {
    int rank = 0;
    for (int o = 0; o < n; ++o) {
      const float other = s_S[o];
      rank += (other > mine || (other == mine && o < g)) ? 1 : 0;
    }
    keep[group_slot(G, b, g)] = rank < keep_count ? 1 : 0;
  }
  if (g == 0) {
    counts[b] = min(keep_count, n);
    if (seg_counts != nullptr) seg_counts[b] = min(keep_count, n);   // (one segment)
  }
}

cudaError_t launch_topk(const uint16_t* w, const Geometry& G, int sms, int keep_count, uint8_t* flags, int32_t* counts, int32_t* seg_counts,
                        cudaStream_t s) {
  if (G.n_groups <= kRankGroups)
    return launch_pdl(flags_rank_kernel, dim3(G.n_blocks), dim3((G.n_groups + 31) / 32 * 32), 0, s, w, G, keep_count, flags, counts, seg_counts);
  const size_t smem = sizeof(uint32_t) * G.n_groups;
  auto launch = [&](auto kernel, int threads) {
    return launch_pdl(kernel, dim3(G.n_blocks), dim3(threads), smem, s, w, G, keep_count, flags, counts, seg_counts);
  };
  if (G.n_groups < 512) return launch(flags_topk_kernel<kPackThreads>, kPackThreads);
  if (G.orient == BSP_ORIENT_C) return launch(flags_topk_kernel<512>, 512);
  // 1024 threads where all strips run at once, and where a strip has so many groups that its passes count more than the
  // waves (512 strips of 8192 groups 136 us, 215 with 256 threads; 600 of 768 groups 25 against 22)
  return G.n_blocks <= 2 * sms || G.n_groups >= 4096 ? launch(flags_topk_kernel<1024>, 1024)
                                                         : launch(flags_topk_kernel<kPackThreads>, kPackThreads);
}

// (2) counts -> blk_ptr (exclusive scan) and the kept-weight total: matrices with more blocks than the
// compaction kernel adds up by itself.
__global__ void __launch_bounds__(1024)
scan_counts_kernel(const int32_t* counts, int n_blocks, int block,
                   int32_t* blk_ptr, int64_t* kept_weights) {
  __shared__ int s_warp[32];
  pdl_wait();
  pdl_launch_dependents();
  int running = 0;
  for (int base = 0; base < n_blocks; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int v = i < n_blocks ? counts[i] : 0;
    int total;
    const int excl = block_exclusive_scan(v, s_warp, &total);
    if (i < n_blocks) blk_ptr[i] = running + excl;
    running += total;
  }
  if (threadIdx.x == 0) {
    blk_ptr[n_blocks] = running;
    if (kept_weights) *kept_weights = static_cast<int64_t>(running) * block;
  }
}

// (3) compaction: ascending index list and the dense tile of kept values of one block.  With `counts` the
// CTA adds up the counts before its block itself and writes blk_ptr (one launch less; 4 bytes per block and
// CTA from L2), without it blk_ptr is there already.  Orientation R: a thread moves its whole group, by
// vectors of G.vec elements; the kept groups of a warp are neighbours in the tile.
template <int T>
__global__ void __launch_bounds__(T)
compact_kernel(const uint16_t* W, Geometry G, const uint8_t* keep, const int32_t* counts,
               int32_t* blk_ptr, int32_t* idx, uint16_t* vals,
               int64_t* kept_weights) {
  __shared__ int s_warp[32];
  const int b = blockIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  int base, kc;
  if (counts != nullptr) {
    int part = 0;
    for (int i = threadIdx.x; i < b; i += blockDim.x) part += counts[i];
    block_exclusive_scan(part, s_warp, &base);
    kc = counts[b];
    if (threadIdx.x == 0) {
      blk_ptr[b] = base;
      if (b == G.n_blocks - 1) {
        blk_ptr[G.n_blocks] = base + kc;
        if (kept_weights) *kept_weights = static_cast<int64_t>(base + kc) * G.block;
      }
    }
  } else {
    base = blk_ptr[b];
    kc = blk_ptr[b + 1] - base;
  }
  if (kc == 0) return;
  uint16_t* tile = vals + static_cast<size_t>(G.block) * base;
  // (values are stored at multiples of the block from an array that is only known to be 2-byte aligned)
  const int vec = G.orient == BSP_ORIENT_R && (reinterpret_cast<uintptr_t>(vals) & 15) == 0 ? G.vec : 1;
  int running = 0;
  for (int g0 = 0; g0 < G.n_groups; g0 += blockDim.x) {
    const int g = g0 + threadIdx.x;
    const int k = (g < G.n_groups) ? keep[group_slot(G, b, g)] : 0;
    int total;
    const int p = running + block_exclusive_scan(k, s_warp, &total);
    running += total;
    if (k) {
      idx[base + p] = g;
      size_t stride;
      const uint16_t* src = group_ptr(W, G, b, g, &stride);
      uint16_t* dst = tile + static_cast<size_t>(p) * G.block;
      if (G.orient == BSP_ORIENT_C) copy_strided(tile + p, kc, src, stride, G.block);   // tile [d, kc]: element r goes to row r
      else if (vec == 8) copy_strided(reinterpret_cast<uint4*>(dst), 1, reinterpret_cast<const uint4*>(src), 1, G.block >> 3);
      else if (vec == 4) copy_strided(reinterpret_cast<uint2*>(dst), 1, reinterpret_cast<const uint2*>(src), 1, G.block >> 2);
      else copy_strided(dst, 1, src, 1, G.block);
    }
  }
}

// Orientation R by segments of 256 groups (rows) of a strip, a CTA each: a few wide strips are only a few CTAs
// otherwise.  A segment's kept count goes to a list of its own, from which the compaction takes blk_ptr and the place of
// its part of the tile; there a CTA moves the kept groups as one run of vectors, coalesced on the packed side.
// Latency-bound.  3072 x 1024, the two launches: 64-column strips 30.8 -> 7.5 us, 16-column 15.7 -> 9.4; 768 x 768 in
// 12-column strips 8.2 -> 6.2.
__global__ void __launch_bounds__(kSegment)
flags_segment_kernel(const uint16_t* W, Geometry G, float threshold, const float* threshold_dev,
                     uint8_t* keep, int32_t* seg_counts) {
  __shared__ int s_warp[kSegment / 32];
  const int b = blockIdx.x, g = blockIdx.y * kSegment + threadIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  const float t = threshold_dev ? *threshold_dev : threshold;
  bool k = false;
  if (g < G.n_groups) {
    k = group_sum(W, G, b, g) > __fmul_rn(t, t) || t < 0.0f;
    keep[group_slot(G, b, g)] = k ? 1 : 0;
  }
  const unsigned kept = __ballot_sync(0xffffffffu, k);
  if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = __popc(kept);
  __syncthreads();
  if (threadIdx.x == 0) {
    int c = 0;
#pragma unroll
    for (int w = 0; w < kSegment / 32; ++w) c += s_warp[w];
    seg_counts[b * gridDim.y + blockIdx.y] = c;
  }
}

template <int VEC>
__global__ void __launch_bounds__(kSegment)
compact_segment_kernel(const uint16_t* W, Geometry G, const uint8_t* keep,
                       const int32_t* seg_counts, int32_t* blk_ptr, int32_t* idx,
                       uint16_t* vals, int64_t* kept_weights) {
  __shared__ int s_base[kSegment / 32], s_warp[kSegment / 32];
  __shared__ int s_group[kSegment];
  const int b = blockIdx.x, segments = gridDim.y, seg = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = seg * kSegment + threadIdx.x;
  pdl_wait();
  pdl_launch_dependents();
  const bool k = g < G.n_groups && keep[group_slot(G, b, g)] != 0;
  int part = 0;                                              // kept groups before this segment, in the order of the strips
  const int before = b * segments + seg;
  for (int i = threadIdx.x; i < before; i += kSegment) part += seg_counts[i];
  part = warp_sum(part);
  const unsigned kept = __ballot_sync(0xffffffffu, k);
  if (lane == 0) { s_base[warp] = part; s_warp[warp] = __popc(kept); }
  __syncthreads();
  int base = 0, p = 0, m = 0;
#pragma unroll
  for (int w = 0; w < kSegment / 32; ++w) {
    base += s_base[w];
    if (w < warp) p += s_warp[w];
    m += s_warp[w];
  }
  p += __popc(kept & ((1u << lane) - 1u));
  if (k) {
    idx[base + p] = g;
    s_group[p] = g;
  }
  if (threadIdx.x == 0) {
    if (seg == 0) blk_ptr[b] = base;
    if (before + 1 == G.n_blocks * segments) {               // the matrix's last segment
      blk_ptr[G.n_blocks] = base + m;
      if (kept_weights) *kept_weights = static_cast<int64_t>(base + m) * G.block;
    }
  }
  __syncthreads();
  const int per = G.block / VEC;
  const uint16_t* strip = W + static_cast<size_t>(b) * G.block;
  uint16_t* out = vals + static_cast<size_t>(G.block) * base;
  using Vec = vector_of<VEC>;
  for (int e0 = threadIdx.x; e0 < m * per; e0 += 4 * kSegment) {
    Vec v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = min(e0 + u * kSegment, m * per - 1);
      const int q = e / per, c = (e - q * per) * VEC;
      v[u] = ld_global(reinterpret_cast<const Vec*>(strip + static_cast<size_t>(s_group[q]) * G.ldw + c));
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = e0 + u * kSegment;
      if (e < m * per) *reinterpret_cast<Vec*>(out + static_cast<size_t>(e) * VEC) = v[u];
    }
  }
}

// Orientation C, 8 adjacent columns of a row per thread: nothing is read but the flags, and only pieces with a
// pruned group are written.  CTAs take pieces of one row, or of the matrix numbered through (kFlat) where a row has too
// few for a warp and there are many rows: 6272 x 80 a row per CTA 8.0 us, flat 3.3; 256 x 88 1.8 and 2.5, 3240 x 1848 15.5
// and 17.8 (two divisions a thread).
template <bool kFlat, typename Index>
__global__ void __launch_bounds__(256)
apply_mask_c_kernel(uint16_t* W, int rows, int cols, int ldw, int block, const uint8_t* keep) {
  const Index chunks = static_cast<Index>(cols >> 3);
  const Index item = static_cast<Index>(blockIdx.x) * blockDim.x + threadIdx.x;
  const Index i = kFlat ? item / chunks : static_cast<Index>(blockIdx.y);
  const Index q = kFlat ? item - i * chunks : item;
  const size_t c = static_cast<size_t>(q) << 3;
  const size_t b = static_cast<unsigned>(i) / static_cast<unsigned>(block);
  pdl_wait();
  pdl_launch_dependents();
  if (i >= static_cast<Index>(rows) || q >= chunks) return;
  const uint2 f = ld_global(reinterpret_cast<const uint2*>(keep + b * cols + c));
  if (((f.x - 0x01010101u) & ~f.x & 0x80808080u) == 0u && ((f.y - 0x01010101u) & ~f.y & 0x80808080u) == 0u) return;   // no zero byte
  uint16_t* w = W + static_cast<size_t>(i) * ldw + c;
  if ((f.x | f.y) == 0u) {
    *reinterpret_cast<uint4*>(w) = make_uint4(0u, 0u, 0u, 0u);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if ((((e < 4 ? f.x : f.y) >> (8 * (e & 3))) & 0xffu) == 0u) w[e] = 0;
  }
}
// Any geometry, a weight per thread.  It overlaps the kernel before it only where it has a CTA per SM or fewer: many short
// CTAs that take seats among those of the kernel before cost 13 % of a 7928 x 2640 matrix in orientation R (75.7 against
// 85.7 us), and a few save half a microsecond.
template <bool kOverlap>
__global__ void __launch_bounds__(256)
apply_mask_kernel(uint16_t* W, Geometry G, const uint8_t* keep) {
  if (kOverlap) {
    pdl_wait();
    pdl_launch_dependents();
  }
  const long long e = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (e >= static_cast<long long>(G.rows) * G.cols) return;
  const int i = static_cast<int>(e / G.cols), j = static_cast<int>(e - static_cast<long long>(i) * G.cols);
  const size_t slot = G.orient == BSP_ORIENT_C ? static_cast<size_t>(i / G.block) * G.cols + j
                                               : static_cast<size_t>(i) * (G.cols / G.block) + j / G.block;
  if (!ld_global(keep + slot)) W[static_cast<size_t>(i) * G.ldw + j] = 0;
}

// Fixed scratch for bsp_prune_pack_static: lives in the library's device image, so every GPU
// that loads the library holds these bytes until the process exits.
static __device__ __align__(256) unsigned char g_static_pack_scratch[BSP_STATIC_SCRATCH_BYTES];

}  // namespace
}  // namespace bsp

extern "C" int bsp_pack_bound(int rows, int cols, int block, int orient, size_t* idx_elems,
                              size_t* val_elems, size_t* ws_bytes) {
  using namespace bsp;
  if (rows <= 0 || cols <= 0 || block <= 0) return BSP_ERR_ARG;
  if (orient != BSP_ORIENT_C && orient != BSP_ORIENT_R) return BSP_ERR_ARG;
  int nb, ng;
  if (!geometry(rows, cols, block, orient, &nb, &ng)) return BSP_ERR_SHAPE;
  if (idx_elems) *idx_elems = static_cast<size_t>(nb) * ng;
  if (val_elems) *val_elems = static_cast<size_t>(rows) * cols;
  if (ws_bytes) *ws_bytes = ws_layout(nb, ng).total;
  return BSP_OK;
}

extern "C" int bsp_pack_scratch_bytes(int rows, int cols, int block, int orient, size_t* bytes) {
  using namespace bsp;
  if (rows <= 0 || cols <= 0 || block <= 0 || bytes == nullptr) return BSP_ERR_ARG;
  if (orient != BSP_ORIENT_C && orient != BSP_ORIENT_R) return BSP_ERR_ARG;
  int nb, ng;
  if (!geometry(rows, cols, block, orient, &nb, &ng)) return BSP_ERR_SHAPE;
  *bytes = ws_layout(nb, ng).sumsq_off;
  return BSP_OK;
}

extern "C" int bsp_prune_pack(const void* W, int rows, int cols, int ldw, int block, int orient,
                              float threshold, const float* threshold_dev, int keep_per_block,
                              uint8_t* keep, int32_t* blk_ptr, int32_t* idx, void* vals,
                              int64_t* kept_weights, void* ws, size_t ws_bytes, void* stream) {
  using namespace bsp;
  int st = check_matrix_args(W, rows, cols, ldw, block, orient);
  if (st != BSP_OK) return st;
  if (blk_ptr == nullptr || idx == nullptr || vals == nullptr || ws == nullptr) return BSP_ERR_ARG;
  if (!aligned_to(ws, 256) || !aligned_to(vals, 2) || !aligned_to(blk_ptr, 4) || !aligned_to(idx, 4)) return BSP_ERR_ARG;
  if (threshold != threshold) return BSP_ERR_ARG;  // NaN
  Geometry G{rows, cols, ldw, block, orient, 0, 0, 1};
  geometry(rows, cols, block, orient, &G.n_blocks, &G.n_groups);
  if (orient == BSP_ORIENT_R) G.vec = contig_vec(W, ldw, block);
  else if (cols % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16)) G.vec = 8;
  const WsLayout L = ws_layout(G.n_blocks, G.n_groups);
  if (ws_bytes < L.sumsq_off) return BSP_ERR_WORKSPACE;   // counts and flags; the float32 region is the percentile call's
  if (keep_per_block >= 0 && G.n_groups > BSP_TOPK_MAX_GROUPS) return BSP_ERR_UNSUPPORTED;

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* wsb = static_cast<char*>(ws);
  int32_t* counts = reinterpret_cast<int32_t*>(wsb + L.counts_off);
  uint8_t* flags = keep ? keep : reinterpret_cast<uint8_t*>(wsb + L.keep_off);
  const uint16_t* w = static_cast<const uint16_t*>(W);

  int sms = 0;                          // (two CTAs of 1024 threads fit one)
  BSP_TRY(sm_count(&sms));
  const bool fast = orient == BSP_ORIENT_C && fused_shape_ok(W, rows, cols, ldw, block) && aligned_to(flags, 8);
  if (fast) {
    // vectorised kernels of bsp_fused.cu: stage 1 for the flags (unless the keep-count kernel makes them), stage 2
    FusedJob j{w, rows, cols, ldw, G.n_blocks, threshold, threshold_dev, nullptr, nullptr, nullptr, nullptr, nullptr,
               flags, counts, blk_ptr, idx, static_cast<uint16_t*>(vals), kept_weights, nullptr};
    if (keep_per_block >= 0) {
      BSP_CUDA_TRY(launch_topk(w, G, sms, keep_per_block, flags, counts, nullptr, s));
    } else {
      st = fused_stage1(&j, 1, block, 0.0f, 0, s);
      if (st != BSP_OK) return st;
    }
    return fused_stage2(&j, 1, block, s);
  }
  const long long segments = (G.n_groups + kSegment - 1) / kSegment;
  const bool keep_in_ws = keep >= reinterpret_cast<uint8_t*>(wsb) && keep < reinterpret_cast<uint8_t*>(wsb) + ws_bytes;
  if (orient == BSP_ORIENT_R && keep != nullptr && !keep_in_ws && G.n_blocks * segments <= (G.n_blocks <= kFewStrips ? kMaxSegmentsFew : kMaxSegments) &&
      G.n_blocks * segments * sizeof(int32_t) <= L.sumsq_off - L.keep_off) {
    // (the flags go to the caller's array, so the workspace's flags are free for the segments' counts)
    int32_t* seg_counts = reinterpret_cast<int32_t*>(wsb + L.keep_off);
    const dim3 grid(G.n_blocks, static_cast<unsigned>(segments));
    if (keep_per_block >= 0) BSP_CUDA_TRY(launch_topk(w, G, sms, keep_per_block, flags, counts, seg_counts, s));
    else BSP_CUDA_TRY(launch_pdl(flags_segment_kernel, grid, dim3(kSegment), 0, s, w, G, threshold, threshold_dev, flags, seg_counts));
    const int vec = (reinterpret_cast<uintptr_t>(vals) & 15) == 0 ? G.vec : 1;
    BSP_CUDA_TRY(launch_pdl(vec == 8 ? compact_segment_kernel<8> : vec == 4 ? compact_segment_kernel<4> : compact_segment_kernel<1>, grid,
                            dim3(kSegment), 0, s, w, G, flags, seg_counts, blk_ptr, idx, static_cast<uint16_t*>(vals), kept_weights));
    return BSP_OK;
  }
  // A CTA per block, threads for its groups: up to 1024 of them, since a matrix of few wide blocks has few CTAs (768 x 5120
  // in 16-row blocks 27 us, 83 with 256 threads).  Many blocks fill the GPU by themselves and want CTAs that come and
  // go (5343 x 920 in single rows 47 us, 67 with 1024; 2204 x 1214 in fours 12.7 against 15; 7826 x 4759 in single columns
  // 650 against 730).
  const bool tall = G.n_blocks <= 2 * sms;
  const int threads = !tall ? 256 : G.n_groups >= 1024 ? 1024 : G.n_groups <= 128 ? 128 : (G.n_groups + 31) / 32 * 32;
  if (keep_per_block >= 0) {
    BSP_CUDA_TRY(launch_topk(w, G, sms, keep_per_block, flags, counts, nullptr, s));
  } else {
    BSP_CUDA_TRY(launch_pdl(tall ? flags_threshold_kernel<1024> : flags_threshold_kernel<256>, dim3(G.n_blocks), dim3(threads), 0, s, w, G,
                            threshold, threshold_dev, flags, counts));
  }
  // every CTA of the compaction adds up the counts before its block; past 4096 blocks that costs more than a
  // scan of its own (it grows with the square of the block count)
  const bool own_scan = G.n_blocks > 4096;
  if (own_scan) BSP_CUDA_TRY(launch_pdl(scan_counts_kernel, dim3(1), dim3(1024), 0, s, counts, G.n_blocks, block, blk_ptr, kept_weights));
  BSP_CUDA_TRY(launch_pdl(tall ? compact_kernel<1024> : compact_kernel<256>, dim3(G.n_blocks), dim3(threads), 0, s, w, G, flags,
                          own_scan ? nullptr : counts, blk_ptr, idx, static_cast<uint16_t*>(vals), kept_weights));
  return BSP_OK;
}

extern "C" int bsp_apply_mask(void* W, int rows, int cols, int ldw, int block, int orient,
                              const uint8_t* keep, void* stream) {
  using namespace bsp;
  int st = check_matrix_args(W, rows, cols, ldw, block, orient);
  if (st != BSP_OK) return st;
  if (keep == nullptr) return BSP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  uint16_t* w = static_cast<uint16_t*>(W);
  if (orient == BSP_ORIENT_C && cols % 8 == 0 && ldw % 8 == 0 && aligned_to(W, 16) && aligned_to(keep, 8)) {
    const int chunks = cols / 8;
    const long long ctas = (static_cast<long long>(rows) * chunks + 255) / 256;
    if (rows <= 65535 && (chunks >= 32 || rows < 2048)) {
      const dim3 grid((chunks + 255) / 256, rows), threads(chunks >= 256 ? 256 : (chunks + 31) / 32 * 32);
      BSP_CUDA_TRY(launch_pdl(apply_mask_c_kernel<false, unsigned>, grid, threads, 0, s, w, rows, cols, ldw, block, keep));
    } else if (ctas * 256 < (1LL << 32)) {
      BSP_CUDA_TRY(launch_pdl(apply_mask_c_kernel<true, unsigned>, dim3(static_cast<unsigned>(ctas)), dim3(256), 0, s, w, rows, cols, ldw, block, keep));
    } else {
      BSP_CUDA_TRY(launch_pdl(apply_mask_c_kernel<true, unsigned long long>, dim3(static_cast<unsigned>(ctas)), dim3(256), 0, s, w, rows, cols, ldw, block, keep));
    }
    return BSP_OK;
  }
  Geometry G{rows, cols, ldw, block, orient, 0, 0, 1};
  geometry(rows, cols, block, orient, &G.n_blocks, &G.n_groups);
  const long long elems = static_cast<long long>(rows) * cols;
  const dim3 grid(static_cast<unsigned>((elems + 255) / 256));
  int sms = 0;
  BSP_TRY(sm_count(&sms));
  if (grid.x <= static_cast<unsigned>(sms)) BSP_CUDA_TRY(launch_pdl(apply_mask_kernel<true>, grid, dim3(256), 0, s, w, G, keep));
  else apply_mask_kernel<false><<<grid, 256, 0, s>>>(w, G, keep);
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

extern "C" int bsp_prune_pack_static(const void* W, int rows, int cols, int ldw, int block, int orient,
                                     float threshold, const float* threshold_dev, int keep_per_block,
                                     uint8_t* keep, int32_t* blk_ptr, int32_t* idx, void* vals,
                                     int64_t* kept_weights, void* stream) {
  using namespace bsp;
  int st = check_matrix_args(W, rows, cols, ldw, block, orient);
  if (st != BSP_OK) return st;
  size_t need = 0;
  st = bsp_pack_scratch_bytes(rows, cols, block, orient, &need);
  if (st != BSP_OK) return st;
  if (need > static_cast<size_t>(BSP_STATIC_SCRATCH_BYTES)) return BSP_ERR_UNSUPPORTED;

  // In host code the array's name is only a handle; the device address has to be asked for,
  // once per device, while that device is current.
  static void* scratch_of_device[64] = {nullptr};
  static std::mutex guard;
  std::lock_guard<std::mutex> lock(guard);
  int dev = -1;
  BSP_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return BSP_ERR_UNSUPPORTED;
  if (scratch_of_device[dev] == nullptr) {
    void* ptr = nullptr;
    BSP_CUDA_TRY(cudaGetSymbolAddress(&ptr, g_static_pack_scratch));
    if (ptr == nullptr) return BSP_ERR_CUDA;
    scratch_of_device[dev] = ptr;
  }
  // Every byte of the scratch that the kernels read (per-block counts, per-group flags) is
  // written earlier in the same call, so nothing left over from the previous call is observed
  // and nothing needs clearing.
  return bsp_prune_pack(W, rows, cols, ldw, block, orient, threshold, threshold_dev, keep_per_block, keep, blk_ptr,
                        idx, vals, kept_weights, scratch_of_device[dev], BSP_STATIC_SCRATCH_BYTES, stream);
}
