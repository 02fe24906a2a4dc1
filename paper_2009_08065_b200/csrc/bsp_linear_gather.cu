// bsp_linear_gathered: the pruned linear layer with the pruned work skipped.  For a row-block of
// d output rows only the kept columns of X are fetched and multiplied (Section 3.1: only the
// non-zero columns of a block take part; Section 4.4: compact storage saves computation).
//
// Operands.  Per row-block the product is  Y[tile, block] = X[tile, kept columns] . vals^T  with
// 128 tokens as the M side of a tcgen05.mma, the d output rows as its N side and the kept columns
// as K.  Single columns of a row-major X are 2-byte pieces, useless for 16-byte copies, so the
// activations are taken TRANSPOSED, XT [k_in, tokens]: a kept column is then a contiguous row of
// 128 tokens (256 bytes), and TMA row gathers (tile::gather4: four rows of a 2-D tensor per
// instruction, box one row high) bring the kept rows straight into the tensor core's "MN-major"
// operand layout (8-row atoms of 64 tokens x 8 columns, 128-byte swizzle).  (A first version
// gathered with 16-byte cp.async copies; the load/store unit's limit on requests in flight held
// it to about 13 bytes per clock per SM.)  The weight
// side comes from a gather plan made once per pruned matrix: per pipeline stage (64 kept columns)
// the d x 64 tile already in the K-major 128-byte-swizzled layout (one bulk copy lands it), the
// 64 column numbers, and a byte that says how many 16-column groups are real and whether the stage
// starts or ends a row-block.
//
// Kernel.  Persistent CTAs walk units of (128-token tile) x (run of consecutive row-blocks); the
// stages of such a run are consecutive in the plan, so the producers just stream them.
//   warps 0-3 : producers, warp w filling every fourth stage; lane = (64-token half, four rows): one
//               gather4 per lane per stage, completion bytes counted on the stage's mbarrier;
//               lane 0 also issues the bulk copy of the weight tile and hands the stage's byte on;
//   warp 4    : one lane issues tcgen05.mma (M=128, N=d, K=16) into one of the TMEM accumulators,
//               commits stage release and, at the end of a row-block, accumulator ready;
//   warps 5.. : epilogue, two or four groups of four warps that take the row-blocks in turn (group =
//               accumulator); each warp reads its 32 TMEM lanes (tokens), adds bias, optional GELU, rounds to
//               bf16, and the group's 128 x 32 pieces leave through staging buffers as TMA stores (blocks of 16
//               rows: straight from registers).  A piece takes 1000 cycles, 1700 with GELU, nearly all of it
//               latency: one group storing from registers took 54 us for 4096 x 1024 with GELU at 8 times
//               compression and 8192 tokens, two groups 35, four 30; the gathering alone needs 19.
// Every wait is bounded; on expiry the role records BSP_ERR_TIMEOUT and leaves its loop.
//
// What bounds it: every gathered element crosses L2 -> shared memory once per row-block and feeds
// only d multiply-adds per token, so the operand traffic per flop is 1/d of a byte: the kernel
// pays off for tall blocks and high compression, where the zero-expanded dense route spends its
// time multiplying zeros.
#include "bsp_tc.cuh"

namespace bsp {

int check_linear_args(const void* a, const void* b, const void* c, int n_out, int k_in, int block,
                      const void* X, int tokens, int ldx, int act, const void* Y, int ldy);

using namespace tc;

namespace {

constexpr int gather_threads(int groups) { return 160 + 128 * groups; }   // 4 producer warps, MMA warp, epilogue groups
constexpr int kGStageK = 64;                // kept columns per pipeline stage
constexpr int kGStageA = kGStageK * kBlockM * 2;   // 16 KB: 64 rows of 128 tokens
constexpr int kGQueue = 12;                 // a producer warp loads its column numbers up to this many stages ahead
constexpr int kGPrefetch = kGQueue;         // the plan's column array is padded by this many stages

template <int D, int GROUPS>     // GROUPS epilogue groups of four warps, as many TMEM accumulators
struct GatherCfg {
  static constexpr int kStageB = D * 128;                       // d rows of 64 bf16
  static constexpr int kStage = kGStageA + kStageB;
  static constexpr bool kStaged = D >= kEpiCols;                // outputs leave through staging buffers and TMA stores
  static constexpr bool kFragments = GROUPS == 4;               // transposed pieces by fragments (see FragmentPiece)
  static constexpr int kStaging = kStaged ? kEpiBytes : 0;     // four buffers, shared out among the groups
  static constexpr int kFixed = 1024 /*alignment slack*/ + 512 /*barriers, stage bytes*/ + GROUPS * D * 2 /*bias, a block per group*/ + kStaging;
  static constexpr int kStagesRaw = (kSmemLimit - kFixed) / kStage;
  static constexpr int kStages = kStagesRaw > 12 ? 12 : kStagesRaw;
  static constexpr int kTmemCols = GROUPS * D;                  // a power of two, 32 ... 512
  static constexpr int kSmemBytes = kStages * kStage + kFixed;
};

// Layout of a gather plan in device memory (all regions 256-byte aligned):
//   soff  int32 [n_blocks + 1]   first stage of every row-block
//   meta  uint8 [stages]         bits 0-2: real 16-column groups (1..4), bit 4: first stage of its
//                                row-block, bit 5: last stage
//   cols  int16 [stages][64]     column of X for row r of the stage; -1 = zero row (padding inside a
//                                real group), -2 = beyond the real groups (not loaded, not multiplied)
//   tiles bf16  [stages][d][64]  weight tile, row n at byte n*128, 16-byte chunk c at (c ^ (n & 7))
struct GatherLayout {
  size_t soff_off, meta_off, cols_off, tiles_off, total;
  long long max_stages;
};
inline GatherLayout gather_layout(int n_out, int k_in, int block) {
  GatherLayout L;
  const long long nb = n_out / block;
  L.max_stages = nb * ((k_in + kGStageK - 1) / kGStageK);      // every row-block has at least one stage
  if (L.max_stages < nb) L.max_stages = nb;
  L.soff_off = 0;
  L.meta_off = round_up(sizeof(int32_t) * static_cast<size_t>(nb + 1), 256);
  L.cols_off = L.meta_off + round_up(static_cast<size_t>(L.max_stages) + 256, 256);
  L.tiles_off = L.cols_off + round_up(static_cast<size_t>(L.max_stages + kGPrefetch + 1) * kGStageK * 2, 256);
  L.total = L.tiles_off + round_up(static_cast<size_t>(L.max_stages) * block * 128, 256);
  return L;
}

// ---- plan construction -------------------------------------------------------------------
// soff[b] = number of stages of the row-blocks before b (one CTA, a running block-wide scan).
__global__ void __launch_bounds__(1024)
gather_plan_scan_kernel(const int32_t* __restrict__ blk_ptr, int n_blocks, int32_t* __restrict__ soff) {
  __shared__ int s_warp[32];
  int running = 0;
  for (int b0 = 0; b0 < n_blocks; b0 += blockDim.x) {
    const int b = b0 + threadIdx.x;
    int mine = 0;
    if (b < n_blocks) {
      const int kc = blk_ptr[b + 1] - blk_ptr[b];
      mine = kc > 0 ? (kc + kGStageK - 1) / kGStageK : 1;
    }
    int total;
    const int before = running + block_exclusive_scan(mine, s_warp, &total);
    if (b < n_blocks) soff[b] = before;
    running += total;
  }
  if (threadIdx.x == 0) soff[n_blocks] = running;
}

// One CTA per row-block: meta bytes, permuted column numbers and swizzled weight tiles of its stages.
__global__ void __launch_bounds__(256)
gather_plan_fill_kernel(const int32_t* __restrict__ blk_ptr, const int32_t* __restrict__ idx,
                        const uint16_t* __restrict__ vals, int block, const int32_t* __restrict__ soff,
                        uint8_t* __restrict__ meta, int16_t* __restrict__ cols, uint16_t* __restrict__ tiles) {
  const int b = blockIdx.x;
  const int lo = blk_ptr[b], kc = blk_ptr[b + 1] - lo;
  const int g0 = soff[b], n_st = soff[b + 1] - g0;
  const uint16_t* tile = vals + static_cast<size_t>(block) * lo;        // [block][kc]
  for (int s = threadIdx.x; s < n_st; s += blockDim.x) {
    const int left = kc - s * kGStageK;                                  // real columns from this stage on
    int groups = left <= 0 ? 1 : (left >= kGStageK ? 4 : (left + 15) / 16);
    meta[g0 + s] = static_cast<uint8_t>(groups | (s == 0 ? 0x10 : 0) | (s == n_st - 1 ? 0x20 : 0));
  }
  for (int e = threadIdx.x; e < n_st * kGStageK; e += blockDim.x) {
    const int s = e / kGStageK, r = e % kGStageK;
    const int k = s * kGStageK + r;
    const int left = kc - s * kGStageK;
    const int groups = left <= 0 ? 1 : (left >= kGStageK ? 4 : (left + 15) / 16);
    int16_t c = -2;
    if (r < groups * 16) c = k < kc ? static_cast<int16_t>(idx[lo + k]) : static_cast<int16_t>(-1);
    cols[static_cast<size_t>(g0 + s) * kGStageK + r] = c;
  }
  // weight tiles: one thread per 16-byte chunk (8 columns of one row)
  const int chunks = n_st * block * 8;
  for (int e = threadIdx.x; e < chunks; e += blockDim.x) {
    const int s = e / (block * 8), rem = e % (block * 8);
    const int n = rem >> 3, ch = rem & 7;
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int k0 = s * kGStageK + ch * 8 + 2 * i;
      const uint32_t v0 = k0 < kc ? tile[static_cast<size_t>(n) * kc + k0] : 0u;
      const uint32_t v1 = k0 + 1 < kc ? tile[static_cast<size_t>(n) * kc + k0 + 1] : 0u;
      w[i] = v0 | (v1 << 16);
    }
    uint16_t* dst = tiles + (static_cast<size_t>(g0 + s) * block + n) * 64 + ((ch ^ (n & 7)) << 3);
    *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// ---- transposed copy ---------------------------------------------------------------------
// XT[c, r] = X[r, c] for a row-major bf16 matrix; 64 x 64 tiles through shared memory, 16-byte
// global accesses on both sides (rows and cols multiples of 8).  Bound by memory (2 bytes in and out) once the shared
// memory side is cheap: a tile row is 32 words, turned by 4 words for every 8 rows, so that rows go in as 16-byte stores
// and a thread reads the words of two columns in 8 rows, both without bank conflicts, and sorts the halves into the
// two columns' 16-byte stores.  (By single elements, 16 stores and 16 loads a thread, 8192 x 1024 took 8.2 us, 6.9 now.)
__global__ void __launch_bounds__(256)
transpose_kernel(const uint16_t* X, int rows, int cols, int ldx, uint16_t* XT, int ldxt) {
  __shared__ __align__(16) uint32_t s_t[64][32];
  const int r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  pdl_wait();
  pdl_launch_dependents();
  uint4 v[2];
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (threadIdx.x >> 3) + 32 * u, q = threadIdx.x & 7;
    v[u] = make_uint4(0u, 0u, 0u, 0u);
    if (r0 + r < rows && c0 + q * 8 < cols) v[u] = ld_global(reinterpret_cast<const uint4*>(X + static_cast<size_t>(r0 + r) * ldx + c0 + q * 8));
  }
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (threadIdx.x >> 3) + 32 * u, q = threadIdx.x & 7;
    *reinterpret_cast<uint4*>(&s_t[r][(4 * q + 4 * (r >> 3)) & 31]) = v[u];
  }
  __syncthreads();
  const int q = threadIdx.x & 7, pair = threadIdx.x >> 3;      // source rows 8q..8q+7 of columns 2 pair, 2 pair + 1
  if (c0 + 2 * pair >= cols || r0 + 8 * q >= rows) return;
  uint32_t w[8], a[4], b[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) w[i] = s_t[8 * q + i][(pair + 4 * q) & 31];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    a[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x5410);        // the low halves: the even column
    b[i] = __byte_perm(w[2 * i], w[2 * i + 1], 0x7632);
  }
  uint16_t* out = XT + static_cast<size_t>(c0 + 2 * pair) * ldxt + r0 + 8 * q;
  *reinterpret_cast<uint4*>(out) = make_uint4(a[0], a[1], a[2], a[3]);
  *reinterpret_cast<uint4*>(out + ldxt) = make_uint4(b[0], b[1], b[2], b[3]);
}

// ---- the kernel --------------------------------------------------------------------------
struct GatherParams {
  const uint16_t* XT;
  int ldxt, tokens, n_out, k_in, act;
  const uint16_t* bias;
  uint16_t* Y;
  int ldy;
  int transposed;            // Y is [n_out, tokens] (leading dimension ldy spans the tokens)
  const int32_t* soff;
  const uint8_t* meta;
  const int16_t* cols;
  const uint16_t* tiles;
  int n_blocks, m_tiles, n_chunks, rb_per_chunk;
  int* status;
};

// MN-major operand tile with the 128-byte swizzle: 8-row atoms 1024 bytes apart along the
// contraction, the two 64-token halves of the tile 8 KB apart.
__device__ __forceinline__ uint64_t gather_desc_a(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3ffff) >> 4);
  d |= static_cast<uint64_t>((kGStageK * 128) >> 4) << 16;      // leading byte offset / 16
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                   // stride byte offset / 16
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}
// bf16 x bf16 -> float32, A MN-major (bit 15), B K-major, M = 128, N = d.
__host__ __device__ constexpr uint32_t gather_idesc(int d) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (static_cast<uint32_t>(d >> 3) << 17) |
         (static_cast<uint32_t>(kBlockM >> 4) << 24);
}
__device__ __forceinline__ void tmem_load_16cols(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}

// Four rows of XT x 64 tokens, for both 64-token halves of a tile, by an elected lane of a converged warp.
__device__ __forceinline__ void gather4_elect(uint32_t dst, const CUtensorMap* map, int x, int r0, int r1, int r2, int r3, uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t.reg .b32 d2, x2;\n\telect.sync _|e, 0xffffffff;\n\t"
      "add.u32 d2, %0, %8;\n\tadd.s32 x2, %2, 64;\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3, %4, %5, %6}], [%7];\n\t"
      "@e cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes "
      "[d2], [%1, {x2, %3, %4, %5, %6}], [%7];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(r0), "r"(r1), "r"(r2), "r"(r3), "r"(bar), "n"(kGStageK * 128)
      : "memory");
}
// The MMAs of one stage, one per real group of 16 columns, then the commit that frees it.
__device__ __forceinline__ void mma_gather_stage(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate,
                                                 uint32_t groups, uint32_t free_bar) {
  asm volatile(
      "{\n\t.reg .pred p, t, e, e1, e2, e3;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "setp.gt.and.u32 e1, %5, 1, e;\n\tsetp.gt.and.u32 e2, %5, 2, e;\n\tsetp.gt.and.u32 e3, %5, 3, e;\n\t"
      "add.s64 a1, %1, 128;\n\tadd.s64 a2, %1, 256;\n\tadd.s64 a3, %1, 384;\n\t"
      "add.s64 b1, %2, 2;\n\tadd.s64 b2, %2, 4;\n\tadd.s64 b3, %2, 6;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "@e1 tcgen05.mma.cta_group::1.kind::f16 [%0], a1, b1, %3, t;\n\t"
      "@e2 tcgen05.mma.cta_group::1.kind::f16 [%0], a2, b2, %3, t;\n\t"
      "@e3 tcgen05.mma.cta_group::1.kind::f16 [%0], a3, b3, %3, t;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%6];\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(groups), "r"(free_bar)
      : "memory");
}

// A 32-row piece of a TRANSPOSED output, [32 output rows][128 tokens].  The accumulator is read as 8 x 8 fragments (a lane
// holds two neighbouring output rows of a token), which stmatrix stores transposed: four instructions a warp and piece
// where the row-per-thread form of piece_store_transposed stores 32 16-bit values per thread.  The staging buffer is two
// halves of 64 tokens with the 128-byte swizzle, so that the eight rows of a fragment fall on different banks.  The
// epilogue of such a layer is bound by issue slots (58 % busy with four groups): 4096 x 1024 in 128-row blocks at 8x with
// GELU, 8192 tokens, 32.6 -> 30.7 us.  With two groups, which are not, a piece by itself takes longer (336 tokens, two linears
// of 896 features: 15.5 -> 15.7 us).  With 128-row blocks the kernel stands at the 80 registers that 672 threads leave and
// spills 16 bytes a thread; that is counted in the figures.
struct FragmentPiece {
  uint32_t v[32];            // [16-token half][8 output rows: 4][token, token + 8 by two output rows]
  uint32_t bias[4];          // of this lane's two rows of each 8
};
__device__ __forceinline__ void fragment_load(uint32_t taddr, uint32_t bias_smem, int lane, FragmentPiece& p) {
#pragma unroll
  for (int h = 0; h < 2; ++h)
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(p.v[16 * h]), "=r"(p.v[16 * h + 1]), "=r"(p.v[16 * h + 2]), "=r"(p.v[16 * h + 3]), "=r"(p.v[16 * h + 4]),
          "=r"(p.v[16 * h + 5]), "=r"(p.v[16 * h + 6]), "=r"(p.v[16 * h + 7]), "=r"(p.v[16 * h + 8]), "=r"(p.v[16 * h + 9]),
          "=r"(p.v[16 * h + 10]), "=r"(p.v[16 * h + 11]), "=r"(p.v[16 * h + 12]), "=r"(p.v[16 * h + 13]), "=r"(p.v[16 * h + 14]),
          "=r"(p.v[16 * h + 15])
        : "r"(taddr + (static_cast<uint32_t>(16 * h) << 16))
        : "memory");
#pragma unroll
  for (int j = 0; j < 4; ++j)
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(p.bias[j]) : "r"(bias_smem + 16u * j + 4u * (lane & 3)));
  tmem_load_wait();
  tmem_loaded<32>(p.v);
}
__device__ __forceinline__ void fragment_store(const FragmentPiece& p, int act, uint32_t buf, int quad, int lane) {
  // lane i of eight gives the address of output row 8 j + i; the four fragments of a store are the warp's 32 tokens
  const uint32_t i = lane & 7, chunk = static_cast<uint32_t>((quad & 1) * 4 + (lane >> 3));
  const uint32_t dst = buf + static_cast<uint32_t>(quad >> 1) * (kEpiStage / 2) + i * 128u + ((chunk ^ i) << 4);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned long long bias = pack_f32x2(__uint_as_float(p.bias[j] << 16), __uint_as_float(p.bias[j] & 0xffff0000u));
    uint32_t w[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t* v = &p.v[16 * (q >> 1) + 4 * j + 2 * (q & 1)];
      float f0, f1;
      unpack_f32x2(add_f32x2(pack_f32x2(__uint_as_float(v[0]), __uint_as_float(v[1])), bias), f0, f1);
      if (act == BSP_ACT_GELU) gelu_erf_pair(f0, f1);
      w[q] = pack_bf16x2(f0, f1);
    }
    asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(dst + j * 1024u), "r"(w[0]), "r"(w[1]),
                 "r"(w[2]), "r"(w[3]));
  }
}

// Named barriers of the epilogue groups: 1 + g, and 5 + g with a vote.
__device__ __forceinline__ void gather_group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); }
// The 128 threads of an epilogue group agree on whether all of their waits succeeded; also
// the barrier behind the group's bias writes.
__device__ __forceinline__ bool group_all_ok(int group, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, %2, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u), "r"(5 + group)
      : "memory");
  return r != 0u;
}

template <int D, int GROUPS>
__global__ void __launch_bounds__(gather_threads(GROUPS), 1)
linear_gather_kernel(const __grid_constant__ CUtensorMap map_xt, const __grid_constant__ CUtensorMap map_y,
                     const __grid_constant__ GatherParams P) {
  using Cfg = GatherCfg<D, GROUPS>;
  constexpr int kBuffers = kEpiBuffers / GROUPS;
  constexpr int S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  // [S stages: A 16 KB, B D*128][output staging][bias of a row-block per group][mbarriers][stage bytes][TMEM base]
  uint16_t* s_bias = reinterpret_cast<uint16_t*>(smem + S * Cfg::kStage + Cfg::kStaging);
  uint64_t* bars = reinterpret_cast<uint64_t*>(s_bias + GROUPS * D);
  // bars[0..S) full, [S..2S) empty, then per accumulator full, empty
  uint8_t* s_meta = reinterpret_cast<uint8_t*>(bars + 2 * S + 2 * GROUPS);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(s_meta + 16);
  volatile uint32_t* timed_out = tmem_holder + 1;     // set by a role whose wait expired

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
  auto acc_full_bar = [&](int a) { return bar_base + 8u * (2 * S + a); };
  auto acc_empty_bar = [&](int a) { return bar_base + 8u * (2 * S + GROUPS + a); };

  if (threadIdx.x == 0) {
    *timed_out = 0u;
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_xt)) : "memory");
    for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < GROUPS; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 4); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 4) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  const int total_units = P.m_tiles * P.n_chunks;
  pdl_wait();
  pdl_launch_dependents();

  if (warp < 4) {
    // ---------------------------------------------------------------- producers
    // Warp w fills the stages whose running number is w (mod 4).  Lane = (64-token half, group of
    // four consecutive rows): one TMA gather4 per lane brings four kept columns (rows of XT) x 64
    // tokens into the stage with the 128-byte swizzle.  A row number equal to k_in is out of range
    // and reads as zeros (padding rows); tokens beyond the end read as zeros too.
    const int quad4 = lane & 15;                     // this lane holds the numbers of columns 4 quad4 .. 4 quad4 + 3
    long long n0 = 0;                                // stages before this unit, over all units of this CTA
    bool ok = true;
    for (int unit = blockIdx.x; unit < total_units && ok; unit += gridDim.x) {
      const int m = unit / P.n_chunks, ch = unit - m * P.n_chunks;
      const int rb0 = ch * P.rb_per_chunk, rb1 = min(P.n_blocks, rb0 + P.rb_per_chunk);
      const int g_begin = ld_global(P.soff + rb0), g_end = ld_global(P.soff + rb1);
      const int x = m * kBlockM;
      const int first = g_begin + static_cast<int>(((warp - n0) % 4 + 4) % 4);   // this warp's first stage of the unit
      // column numbers and stage bytes are loaded two of the warp's stages (eight stages) ahead
      uint2 cq[2];
      uint32_t mq[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        cq[q] = ld_global(reinterpret_cast<const uint2*>(P.cols + static_cast<size_t>(first + 4 * q) * kGStageK + quad4 * 4));
        mq[q] = ld_global(P.meta + first + 4 * q);
      }
      for (int g0 = first; g0 < g_end && ok; g0 += 8) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int g = g0 + 4 * q;
          if (g < g_end && ok) {
            const long long n = n0 + (g - g_begin);
            const int stage = static_cast<int>(n % S);
            const uint32_t phase = static_cast<uint32_t>((n / S) & 1);
            if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; }
            if (ok) {
              const uint2 cv = cq[q];
              const uint32_t mt = mq[q];
              cq[q] = ld_global(reinterpret_cast<const uint2*>(P.cols + static_cast<size_t>(g + 8) * kGStageK + quad4 * 4));
              mq[q] = ld_global(P.meta + g + 8);
              const uint32_t a_dst = smem_base + stage * Cfg::kStage;
              const int groups = static_cast<int>(mt & 7u);
              if (lane == 0) {
                s_meta[stage] = static_cast<uint8_t>(mt);
                mbar_arrive_expect_tx(full_bar(stage), static_cast<uint32_t>(groups * 16 * kBlockM * 2 + Cfg::kStageB));
                asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                             ::"r"(a_dst + kGStageA), "l"(reinterpret_cast<uint64_t>(P.tiles + static_cast<size_t>(g) * D * 64)),
                               "r"(static_cast<uint32_t>(Cfg::kStageB)), "r"(full_bar(stage))
                             : "memory");
              }
              __syncwarp();
              int r01 = static_cast<int>(cv.x), r23 = static_cast<int>(cv.y);
              for (int q4 = 0; q4 < groups * 4; ++q4) {          // four rows of XT at a time, both 64-token halves
                const int c01 = __shfl_sync(0xffffffffu, r01, q4), c23 = __shfl_sync(0xffffffffu, r23, q4);
                int r0 = static_cast<int16_t>(c01 & 0xffff), r1 = c01 >> 16, r2 = static_cast<int16_t>(c23 & 0xffff), r3 = c23 >> 16;
                r0 = r0 < 0 ? P.k_in : r0;
                r1 = r1 < 0 ? P.k_in : r1;
                r2 = r2 < 0 ? P.k_in : r2;
                r3 = r3 < 0 ? P.k_in : r3;
                gather4_elect(a_dst + static_cast<uint32_t>(q4) * 512u, &map_xt, x, r0, r1, r2, r3, full_bar(stage));
              }
            }
          }
        }
      }
      n0 += g_end - g_begin;
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 4) {
    // ---------------------------------------------------------------- MMA issuer
    {
      constexpr uint32_t idesc = gather_idesc(D);
      int stage = 0;
      uint32_t phase = 0;
      uint32_t acc_phase = 0u;               // of every accumulator: they are used in turn
      int acc = 0;
      bool ok = true;
      for (int unit = blockIdx.x; unit < total_units && ok; unit += gridDim.x) {
        const int m = unit / P.n_chunks, ch = unit - m * P.n_chunks;
        const int rb0 = ch * P.rb_per_chunk, rb1 = min(P.n_blocks, rb0 + P.rb_per_chunk);
        const int g_begin = ld_global(P.soff + rb0), g_end = ld_global(P.soff + rb1);
        for (int g = g_begin; g < g_end; ++g) {
          if (!mbar_wait_warp(full_bar(stage), phase, P.status)) { ok = false; break; }
          tcgen05_fence_after();
          const uint32_t mt = s_meta[stage];
          const int groups = static_cast<int>(mt & 7u);
          const bool first = (mt & 0x10u) != 0, last = (mt & 0x20u) != 0;
          if (first) {
            if (!mbar_wait_warp(acc_empty_bar(acc), acc_phase ^ 1u, P.status)) { ok = false; break; }
            tcgen05_fence_after();
          }
          const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * D);
          const uint32_t a_addr = smem_base + stage * Cfg::kStage;
          const uint32_t b_addr = a_addr + kGStageA;
          mma_gather_stage(d_tmem, gather_desc_a(a_addr), smem_desc_sw128(b_addr), idesc, first ? 0u : 1u, static_cast<uint32_t>(groups),
                           empty_bar(stage));
          if (last) {
            tcgen05_commit_elect(acc_full_bar(acc));
            if (++acc == GROUPS) { acc = 0; acc_phase ^= 1u; }
          }
          if (++stage == S) { stage = 0; phase ^= 1u; }
        }
      }
      if (!ok && lane == 0) record_timeout(P.status, timed_out);
    }
  } else {
    // ---------------------------------------------------------------- epilogue
    const int group = (warp - 5) >> 2;       // takes accumulator `group`: every GROUPS-th row-block of this CTA's sequence
    const int quad = warp & 3;               // TMEM lanes [32*quad, 32*quad+32) belong to this warp
    const int row = quad * 32 + lane;
    const int tid = static_cast<int>(threadIdx.x) - 160 - group * 128;
    const bool issuer = tid == 0;            // the thread that owns the group's TMA stores
    const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(group * D);
    const uint32_t buf0 = smem_base + S * Cfg::kStage + static_cast<uint32_t>(group * kBuffers) * kEpiStage;
    uint16_t* my_bias = s_bias + group * D;
    uint32_t phase = 0u, piece_no = 0u;
    // position in this CTA's sequence of row-blocks
    struct {
      int unit, m, rb, rb1;
    } at{static_cast<int>(blockIdx.x), 0, 0, 0};
    auto enter = [&](auto& c) {
      if (c.unit >= total_units) return;
      const int ch = c.unit % P.n_chunks;
      c.m = c.unit / P.n_chunks;
      c.rb = ch * P.rb_per_chunk;
      c.rb1 = min(P.n_blocks, c.rb + P.rb_per_chunk);
    };
    auto advance = [&](auto& c) {
      if (c.unit < total_units && ++c.rb >= c.rb1) {
        c.unit += gridDim.x;
        enter(c);
      }
    };
    auto bias_of = [&](const auto& c) -> uint16_t {
      return tid < D && c.unit < total_units && P.bias != nullptr ? ld_global(P.bias + static_cast<size_t>(c.rb) * D + tid) : static_cast<uint16_t>(0);
    };
    enter(at);
    for (int g = 0; g < group; ++g) advance(at);
    uint16_t next_bias = bias_of(at);
    bool ok = true;
    while (at.unit < total_units) {
      const int m = at.m, rb = at.rb;
      // this block's bias was asked for a block ago (its slot's last readers are behind the group's last barrier)
      if (tid < D) my_bias[tid] = next_bias;
#pragma unroll
      for (int g = 0; g < GROUPS; ++g) advance(at);
      next_bias = bias_of(at);
      // one decision for the group: nobody is left alone at its barriers
      if (!group_all_ok(group, mbar_wait(acc_full_bar(group), phase, P.status))) { ok = false; break; }
      phase ^= 1u;
      tcgen05_fence_after();
      if constexpr (Cfg::kStaged) {
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += kEpiCols) {
          const uint32_t buf = buf0 + (piece_no % kBuffers) * kEpiStage;
          ++piece_no;
          auto acquire = [&] {                      // the buffer; and, after the last piece, the accumulator goes back
            if (issuer) tma_store_wait_read<kBuffers - 1>();   // the store that last used this buffer has read it
            gather_group_sync(group);
            if (c0 + kEpiCols >= D) {
              tcgen05_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(acc_empty_bar(group));
            }
          };
          if (Cfg::kFragments && P.transposed) {
            FragmentPiece piece;
            fragment_load(taddr + c0, smem_u32(my_bias + c0), lane, piece);
            acquire();
            fragment_store(piece, P.act, buf, quad, lane);
          } else {
            EpiloguePiece piece;
            piece_load(taddr + c0, smem_u32(my_bias + c0), piece);
            acquire();
            if (!Cfg::kFragments && P.transposed) piece_store_transposed(piece, P.act, buf, row);
            else piece_store(piece, P.act, buf + static_cast<uint32_t>(row) * 64u, static_cast<uint32_t>((row >> 1) & 3));
          }
          fence_async_smem();
          gather_group_sync(group);
          if (issuer) {
            if (P.transposed) {
              // (two boxes of 64 tokens, one bulk group; a tile may end within its first half)
              if (Cfg::kFragments && m * kBlockM + 64 < P.tokens)
                asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                             ::"l"(reinterpret_cast<uint64_t>(&map_y)), "r"(m * kBlockM + 64), "r"(rb * D + c0), "r"(buf + kEpiStage / 2)
                             : "memory");
              tma_store_2d(&map_y, m * kBlockM, rb * D + c0, buf);
            } else {
              tma_store_2d(&map_y, rb * D + c0, m * kBlockM, buf);
            }
          }
        }
      } else {
        uint32_t v[16];
        tmem_load_16cols(taddr, v);
        const uint4 b0 = ld_shared_v4(smem_u32(my_bias)), b1 = ld_shared_v4(smem_u32(my_bias) + 16u);
        tmem_load_wait();
        tmem_loaded<16>(v);
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty_bar(group));
        const uint32_t bw[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float f[16];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          f[2 * i] = __uint_as_float(v[2 * i]) + __uint_as_float(bw[i] << 16);
          f[2 * i + 1] = __uint_as_float(v[2 * i + 1]) + __uint_as_float(bw[i] & 0xffff0000u);
        }
        if (P.act == BSP_ACT_GELU) {
#pragma unroll
          for (int i = 0; i < 16; i += 2) gelu_erf_pair(f[i], f[i + 1]);
        }
        const int t = m * kBlockM + row;
        if (t < P.tokens) {
          uint32_t w[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) w[i] = pack_bf16x2(f[2 * i], f[2 * i + 1]);
          if (P.transposed) {
            // output row n = rb * D + i holds this thread's token in column t: the 32 lanes of a warp write 64
            // contiguous bytes per output row
            uint16_t* col = P.Y + static_cast<size_t>(rb) * D * P.ldy + t;
#pragma unroll
            for (int i = 0; i < 16; ++i) col[static_cast<size_t>(i) * P.ldy] = static_cast<uint16_t>(i & 1 ? w[i >> 1] >> 16 : w[i >> 1] & 0xffffu);
          } else {
            uint4* out = reinterpret_cast<uint4*>(P.Y + static_cast<size_t>(t) * P.ldy + static_cast<size_t>(rb) * D);
            out[0] = make_uint4(w[0], w[1], w[2], w[3]);
            out[1] = make_uint4(w[4], w[5], w[6], w[7]);
          }
        }
        gather_group_sync(group);                        // everyone has read the bias
      }
    }
    if (issuer) tma_store_wait_read<0>();
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  }

  tcgen05_fence_before();
  __syncthreads();
  quiet_period(timed_out);
  if (warp == 4) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
  }
}

template <int D, int GROUPS>
int launch_gather_groups(TcDevice* dev, const GatherParams& P, cudaStream_t s) {
  using Cfg = GatherCfg<D, GROUPS>;
  static_assert(Cfg::kStages >= 4, "pipeline too shallow");
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, linear_gather_kernel<D, GROUPS>, Cfg::kSmemBytes));
  CUtensorMap map_xt;      // XT as [k_in rows, tokens]; box = one row of 64 tokens, 128-byte swizzle, zeros out of range
  // (no L2 promotion: a gathered row is 128 bytes, and fetching 256 would read every line twice)
  if (!make_map(&map_xt, P.XT, P.tokens, P.k_in, P.ldxt, 1, 64, CU_TENSOR_MAP_L2_PROMOTION_L2_128B)) return BSP_ERR_CUDA;
  CUtensorMap map_y = map_xt;       // (blocks of 16 rows store without it)
  if (Cfg::kStaged) {
    if (P.transposed) {
      if (!make_map(&map_y, P.Y, P.tokens, P.n_out, P.ldy, kEpiCols, Cfg::kFragments ? 64 : kBlockM)) return BSP_ERR_CUDA;
    } else if (!make_map(&map_y, P.Y, P.n_out, P.tokens, P.ldy, kBlockM, kEpiCols)) {
      return BSP_ERR_CUDA;
    }
  }
  const int units = P.m_tiles * P.n_chunks;
  const int grid = units < dev->sms ? units : dev->sms;
  BSP_CUDA_TRY(launch_pdl(linear_gather_kernel<D, GROUPS>, dim3(grid), dim3(gather_threads(GROUPS)), Cfg::kSmemBytes, s, map_xt, map_y, P));
  return BSP_OK;
}

template <int D>
int launch_gather(TcDevice* dev, const GatherParams& P, cudaStream_t s) {
  if constexpr (D >= 64)
    if (gather_four_groups(D, P.act, static_cast<long long>(P.m_tiles) * P.n_blocks, dev->sms)) return launch_gather_groups<D, 4>(dev, P, s);
  return launch_gather_groups<D, 2>(dev, P, s);
}

bool gather_block_ok(int block) { return block == 16 || block == 32 || block == 64 || block == 128; }

}  // namespace
}  // namespace bsp

extern "C" int bsp_linear_gather_plan_bytes(int n_out, int k_in, int block, size_t* bytes) {
  using namespace bsp;
  if (n_out <= 0 || k_in <= 0 || block <= 0 || bytes == nullptr) return BSP_ERR_ARG;
  if (n_out % block) return BSP_ERR_SHAPE;
  if (!gather_block_ok(block) || k_in > 32767) return BSP_ERR_UNSUPPORTED;
  *bytes = gather_layout(n_out, k_in, block).total;
  return BSP_OK;
}

extern "C" int bsp_linear_gather_plan(const int32_t* blk_ptr, const int32_t* idx, const void* vals, int n_out,
                                      int k_in, int block, void* gplan, size_t gplan_bytes, void* stream) {
  using namespace bsp;
  if (blk_ptr == nullptr || idx == nullptr || vals == nullptr || gplan == nullptr) return BSP_ERR_ARG;
  size_t need;
  int st = bsp_linear_gather_plan_bytes(n_out, k_in, block, &need);
  if (st != BSP_OK) return st;
  if (!aligned_to(gplan, 256)) return BSP_ERR_ARG;
  if (gplan_bytes < need) return BSP_ERR_WORKSPACE;
  const GatherLayout L = gather_layout(n_out, k_in, block);
  char* base = static_cast<char*>(gplan);
  const int nb = n_out / block;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int32_t* soff = reinterpret_cast<int32_t*>(base + L.soff_off);
  gather_plan_scan_kernel<<<1, 1024, 0, s>>>(blk_ptr, nb, soff);
  BSP_LAUNCH_CHECK();
  gather_plan_fill_kernel<<<nb, 256, 0, s>>>(blk_ptr, idx, static_cast<const uint16_t*>(vals), block, soff,
                                             reinterpret_cast<uint8_t*>(base + L.meta_off),
                                             reinterpret_cast<int16_t*>(base + L.cols_off),
                                             reinterpret_cast<uint16_t*>(base + L.tiles_off));
  BSP_LAUNCH_CHECK();
  return BSP_OK;
}

extern "C" int bsp_transpose(const void* X, int rows, int cols, int ldx, void* XT, int ldxt, void* stream) {
  using namespace bsp;
  if (X == nullptr || XT == nullptr || rows < 0 || cols <= 0) return BSP_ERR_ARG;
  if (ldx < cols || ldxt < rows) return BSP_ERR_SHAPE;
  if (rows % 8 || cols % 8 || ldx % 8 || ldxt % 8 || !aligned_to(X, 16) || !aligned_to(XT, 16)) return BSP_ERR_UNSUPPORTED;
  if (rows == 0) return BSP_OK;
  const dim3 grid((cols + 63) / 64, (rows + 63) / 64);
  if (grid.y > 65535) return BSP_ERR_UNSUPPORTED;
  BSP_CUDA_TRY(launch_pdl(transpose_kernel, grid, dim3(256), 0, static_cast<cudaStream_t>(stream), static_cast<const uint16_t*>(X), rows,
                          cols, ldx, static_cast<uint16_t*>(XT), ldxt));
  return BSP_OK;
}

extern "C" int bsp_linear_gathered(const void* gplan, int n_out, int k_in, int block, const void* XT, int tokens,
                                   int ldxt, const void* bias, int act, void* Y, int ldy, void* stream) {
  return bsp_linear_gathered_ex(gplan, n_out, k_in, block, XT, tokens, ldxt, bias, act, Y, ldy, 0, stream);
}

extern "C" int bsp_linear_gathered_ex(const void* gplan, int n_out, int k_in, int block, const void* XT, int tokens,
                                      int ldxt, const void* bias, int act, void* Y, int ldy, int out_transposed,
                                      void* stream) {
  using namespace bsp;
  if (gplan == nullptr || XT == nullptr || Y == nullptr) return BSP_ERR_ARG;
  if (n_out <= 0 || k_in <= 0 || block <= 0 || tokens < 0) return BSP_ERR_ARG;
  if (act != BSP_ACT_NONE && act != BSP_ACT_GELU) return BSP_ERR_ARG;
  if (n_out % block) return BSP_ERR_SHAPE;
  if (ldxt < tokens || ldy < (out_transposed ? tokens : n_out)) return BSP_ERR_SHAPE;
  if (!gather_block_ok(block) || k_in > 32767) return BSP_ERR_UNSUPPORTED;
  if (!aligned_to(gplan, 256) || !aligned_to(XT, 16) || !aligned_to(Y, 16) || (bias != nullptr && !aligned_to(bias, 16)) ||
      tokens % 8 || ldxt % 8 || ldy % 8)
    return BSP_ERR_UNSUPPORTED;
  if (tokens == 0) return BSP_OK;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  const GatherLayout L = gather_layout(n_out, k_in, block);
  const char* base = static_cast<const char*>(gplan);
  GatherParams P;
  P.XT = static_cast<const uint16_t*>(XT);
  P.ldxt = ldxt;
  P.tokens = tokens;
  P.n_out = n_out;
  P.k_in = k_in;
  P.act = act;
  P.bias = static_cast<const uint16_t*>(bias);
  P.Y = static_cast<uint16_t*>(Y);
  P.ldy = ldy;
  P.transposed = out_transposed ? 1 : 0;
  P.soff = reinterpret_cast<const int32_t*>(base + L.soff_off);
  P.meta = reinterpret_cast<const uint8_t*>(base + L.meta_off);
  P.cols = reinterpret_cast<const int16_t*>(base + L.cols_off);
  P.tiles = reinterpret_cast<const uint16_t*>(base + L.tiles_off);
  P.n_blocks = n_out / block;
  const GatherUnits units = gather_units(tokens, P.n_blocks, dev->sms);
  P.m_tiles = units.m_tiles;
  P.rb_per_chunk = units.rb_per_chunk;
  P.n_chunks = units.n_chunks;
  P.status = dev->status;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  switch (block) {
    case 16: return launch_gather<16>(dev, P, s);
    case 32: return launch_gather<32>(dev, P, s);
    case 64: return launch_gather<64>(dev, P, s);
    default: return launch_gather<128>(dev, P, s);
  }
}
