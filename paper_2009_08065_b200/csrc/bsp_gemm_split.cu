// Split contraction for tensor-core products with fewer output tiles than SMs: a cluster of C CTAs shares one
// 128 x BN output tile, CTA r multiplies the r-th part of the contraction, and the partial tiles are added
// through distributed shared memory.  Two operand forms:
//   linear   Y = act(X plan^T + b): K-major operands, the contraction runs over the input features.  With few
//            tokens a layer's product has 12 to 60 tiles of 64 outputs; FFN-down at 8 tokens was 12 CTAs
//            working through 48 stages, 15.7 us of which nearly all was the latency of one CTA's loads.
//   tn       dW = (dY^T X) * Mask: MN-major operands, the contraction runs over the tokens; the 18 to 72 tiles
//            of 128 x 256 of a BERT-base weight left half to seven eighths of the SMs idle.
// A CTA: warps 0 and 10 TMA producers of the two operands, warp 1 MMA issuer, warps
// 2-9 the exchange and epilogue, in two groups of four warps (a warp per quarter of the TMEM lanes).  Each CTA owns
// BN / C columns of the tile.  Once a CTA's accumulator is complete it sends the others their columns as float32
// straight from tensor memory (st.async, 16 bytes per lane, 512 contiguous bytes per warp; only the warps whose rows
// exist), the owner counts the bytes on an mbarrier, adds them in rank order (the result does not depend on timing),
// applies bias, GELU or mask, and stores bf16 rows: by TMA where a warp group has 32 columns, from registers otherwise.
// The linear form has room for the receive buffers beside the stages, so nobody waits for the whole cluster; the
// weight-gradient form receives over its stages and therefore first meets the others at a cluster barrier.
// (Cluster barriers before and after plain remote stores: 1600 cycles of the 5600 of a 768 x 768 launch at 8 tokens.
// Bulk copies between the CTAs' shared memories instead of the stores: 0.6 us slower on the small tiles.)
// A CTA asks for more than half of an SM's shared memory even where a few stages would do: two CTAs of a cluster
// on one SM share its path to L2 (768 outputs x 768 inputs, C = 4: 4.2 us against 3.7).
// All waits are bounded.  A CTA whose wait ran out stays until the rest of its cluster has left: what they were still
// going to send arrives in memory that exists.
#include "bsp_tc.cuh"

namespace bsp {
using namespace tc;

namespace {

constexpr int kSplitThreads = 352;

struct SplitParams {
  int rows, cols;            // output matrix
  int n_tiles, k_blocks, stages;
  int a_bytes;               // bytes of one A copy: fewer than 128 rows where the matrix has fewer
  int recv_off, bars_off;    // offsets of the receive buffers and of the mbarriers
  int plan_stable, act;
  int transposed;            // linear: the output is written as [cols, rows]
  const uint16_t* bias;      // linear
  const uint8_t* keep;       // tn: per-group flags [rows / block, cols], or null
  int block;
  uint16_t* Y;
  int ldy;
  int* status;
};

// 16 bytes into another CTA's shared memory, counted on its mbarrier (both addresses from map_to_cta).
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%2, %3, %4, %5}, [%1];" ::"r"(addr), "r"(bar), "r"(a),
               "r"(b), "r"(c), "r"(d));
}
template <int N>
__device__ __forceinline__ void tmem_load_cols(uint32_t taddr, uint32_t (&v)[N]) {
  static_assert(N == 8 || N == 16 || N == 32, "columns per load");
  if constexpr (N == 32) {
    tmem_load_32cols(taddr, v);
  } else if constexpr (N == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]),
          "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
  } else {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "r"(taddr)
                 : "memory");
  }
}
template <int BN, int C, bool kTn>
__global__ void __launch_bounds__(kSplitThreads, 1)
gemm_split_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                  const __grid_constant__ CUtensorMap map_y, const __grid_constant__ SplitParams P) {
  constexpr int kStageA = kBlockM * kBlockK * 2, kStageB = BN * kBlockK * 2, kStage = kStageA + kStageB;
  constexpr uint32_t kTmemCols = BN;
  constexpr int W = BN / C;                            // columns a CTA owns: [rank * W, +W) of the tile
  constexpr int UW = W >= 16 ? W / 2 : 8;              // of these, the columns of one epilogue group (W = 8: group 0 only)
  constexpr int PC = UW < 32 / (C > 4 ? 2 : 1) ? UW : 32 / (C > 4 ? 2 : 1);   // columns a thread handles at a time
  constexpr uint32_t kSlot = kBlockM * W * 4;          // receive buffer of one source CTA
  constexpr bool kTmaStore = UW % kEpiCols == 0;
  static_assert(W % 8 == 0 && UW % PC == 0, "column pieces");
  constexpr uint32_t kIdesc = kTn ? (instr_desc_bf16(BN) | (1u << 15) | (1u << 16)) : instr_desc_bf16(BN);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + P.bars_off);       // [8] full, [8] empty, accumulator, received
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 18);
  float* s_bias = reinterpret_cast<float*>(bars + 20);                   // [W]
  volatile uint32_t* timed_out = tmem_holder + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = smem_u32(smem), bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (8 + s); };
  const uint32_t acc_bar = bar_base + 8u * 16, recv_bar = bar_base + 8u * 17;
  const int S = P.stages;
  const uint32_t rank = cluster_rank();
  const int tile = static_cast<int>(blockIdx.x) / C;
  const int m0 = (tile / P.n_tiles) * kBlockM, n0 = (tile % P.n_tiles) * BN;
  const int quads = (min(kBlockM, P.rows - m0) + 31) >> 5;   // quarters of the tile with rows that exist

  const int kb0 = static_cast<int>(static_cast<long long>(P.k_blocks) * rank / C);
  const int kb1 = static_cast<int>(static_cast<long long>(P.k_blocks) * (rank + 1) / C);
  const int ahead = min(S, kb1 - kb0);                 // stages that are filled without waiting for one to be free
  auto load_a = [&](int kb, int stage) {
    const uint32_t dst = smem_base + stage * kStage;
    if constexpr (kTn) {
      tma_stage_load(dst, &map_a, m0, kb * kBlockK, full_bar(stage), static_cast<uint32_t>(P.a_bytes));
      tma_load_2d_elect(dst + kAtomGroup, &map_a, m0 + 64, kb * kBlockK, full_bar(stage));
    } else {
      tma_stage_load(dst, &map_a, kb * kBlockK, m0, full_bar(stage), static_cast<uint32_t>(P.a_bytes));
    }
  };
  auto load_b = [&](int kb, int stage) {
    const uint32_t dst = smem_base + stage * kStage + kStageA;
    if constexpr (kTn) {
      tma_stage_load(dst, &map_b, n0, kb * kBlockK, full_bar(stage), kStageB);
#pragma unroll
      for (int g = 1; g < BN / 64; ++g) tma_load_2d_elect(dst + g * kAtomGroup, &map_b, n0 + 64 * g, kb * kBlockK, full_bar(stage));
    } else {
      tma_stage_load(dst, &map_b, kb * kBlockK, n0, full_bar(stage), kStageB);
    }
  };

  // The producers fill the first stages before the CTA meets: a cluster that found its SMs still taken by the kernel before
  // starts late, and its set-up (0.5 us) would lie ahead of its first operands (four linears of 768 features with 8 tokens 14.5
  // -> 14.1 us, an expansion and one linear with 128 tokens 6.47 -> 6.27).  The weights of a stable plan are older than
  // the kernel before this one: their producer does not wait (see launch_pdl).  The signal is left to the warp that allocates
  // this CTA's tensor memory, behind the allocation: a dependent that sat down on this SM before it could take that memory
  // first, and then wait for this grid while this CTA waits for the memory.
  if (warp == 0) {
    if (lane == 0) {
      *timed_out = 0u;
      for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }
      mbar_init(acc_bar, 1);
      mbar_init(recv_bar, 1);
      mbar_arrive_expect_tx(recv_bar, static_cast<uint32_t>((C - 1) * quads * 32 * W * 4));   // what the others will send
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    asm volatile("bar.arrive 6, 64;" ::: "memory");    // the mbarriers exist
    pdl_wait();
    for (int i = 0; i < ahead; ++i) load_a(kb0 + i, i);
  } else if (warp == 10) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_y)) : "memory");
    }
    __syncwarp();
    asm volatile("bar.sync 6, 64;" ::: "memory");
    if (!P.plan_stable) pdl_wait();
    for (int i = 0; i < ahead; ++i) load_b(kb0 + i, i);
  } else if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)), "r"(kTmemCols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    pdl_wait();
    pdl_launch_dependents();
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  cluster_arrive_relaxed();                      // this CTA runs and its mbarriers exist (fenced above)
  if (warp > 1 && warp != 10) pdl_wait();

  if (warp == 0 || warp == 10) {
    // ---------------------------------------------------------------- TMA producers of the A and the B tiles, further stages
    int stage = ahead == S ? 0 : ahead;
    uint32_t phase = ahead == S ? 1u : 0u;
    bool ok = true;
    for (int kb = kb0 + ahead; kb < kb1; ++kb) {
      if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
      if (warp == 0) load_a(kb, stage);
      else load_b(kb, stage);
      if (++stage == S) { stage = 0; phase ^= 1u; }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true, ready = false;
    for (int kb = kb0; kb < kb1; ++kb) {
      if (!mbar_wait_probed(ready, full_bar(stage), phase, P.status)) { ok = false; break; }
      tcgen05_fence_after();
      const int next = stage + 1 == S ? 0 : stage + 1;
      const uint32_t next_phase = next ? phase : phase ^ 1u;
      ready = kb + 1 < kb1 && mbar_try_wait(full_bar(next), next_phase);
      const uint32_t a_addr = smem_base + stage * kStage, b_addr = a_addr + kStageA;
      if constexpr (kTn)     // 16 contraction rows = two 8-row atoms = 2048 bytes per step
        mma_stage<128, 128>(tmem_base, smem_desc_mn_sw128(a_addr), smem_desc_mn_sw128(b_addr), kIdesc, kb != kb0 ? 1u : 0u, empty_bar(stage));
      else                   // 16 columns = 32 bytes
        mma_stage<2, 2>(tmem_base, smem_desc_sw128(a_addr), smem_desc_sw128(b_addr), kIdesc, kb != kb0 ? 1u : 0u, empty_bar(stage));
      stage = next;
      phase = next_phase;
    }
    if (ok) tcgen05_commit_elect(acc_bar);
    else if (lane == 0) record_timeout(P.status, timed_out);
  }
  __syncwarp();
  const bool epilogue = warp >= 2 && warp < 10;
  const int group = (warp - 2) >> 2, quad = warp & 3;
  const int row = quad * 32 + lane, m = m0 + row;
  const bool mine = epilogue && group * UW < W;        // this warp's group has columns
  const bool live = quad < quads;                      // this warp's rows exist
  const int n_own = n0 + static_cast<int>(rank) * W + group * UW;   // its first output column
  bool ok = true;
  uint2 flags[kTn ? UW / 8 : 1];
  if (epilogue) {
    if constexpr (!kTn) {
      const int c = static_cast<int>(threadIdx.x) - 64, n = n0 + static_cast<int>(rank) * W + c;
      if (c < W) s_bias[c] = P.bias != nullptr && n < P.cols ? bf16_bits_to_float(ld_global(P.bias + n)) : 0.0f;
    } else {
#pragma unroll
      for (int i = 0; i < UW / 8; ++i) {               // (cols is a multiple of 8: eight columns are inside or outside)
        flags[i] = make_uint2(0x01010101u, 0x01010101u);
        if (P.keep != nullptr && mine && m < P.rows && n_own + 8 * i < P.cols)
          flags[i] = ld_global(reinterpret_cast<const uint2*>(P.keep + static_cast<size_t>(m / P.block) * P.cols + n_own + 8 * i));
      }
    }
    ok = __all_sync(0xffffffffu, mbar_wait(acc_bar, 0u, P.status));
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
    tcgen05_fence_after();
  }
  __syncwarp();
  cluster_wait();                                // the others run
  if constexpr (kTn) {                                 // and no longer need their stages: their epilogue warps have seen the last MMA complete
    cluster_arrive_relaxed();
    cluster_wait();
  }

  const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
  // receive buffer of a CTA: [source, own rank left out][4-column group][row][4 floats]
  const uint32_t recv_base = smem_base + static_cast<uint32_t>(P.recv_off);
  const uint32_t row_at = static_cast<uint32_t>(row) * 16u;
  if (mine && live && ok) {
    // ---------------------------------------------------------------- partial columns to their owners
#pragma unroll 1
    for (int c0 = group * UW; c0 < (group + 1) * UW; c0 += PC) {
      uint32_t v[C - 1][PC];
#pragma unroll
      for (int o = 1; o < C; ++o) tmem_load_cols<PC>(taddr + ((rank + o) % C) * W + c0, v[o - 1]);
      tmem_load_wait();
#pragma unroll
      for (int o = 1; o < C; ++o) {
        tmem_loaded<PC>(v[o - 1]);
        const uint32_t q = (rank + o) % C, slot = rank < q ? rank : rank - 1;
        const uint32_t dst = map_to_cta(recv_base + slot * kSlot + static_cast<uint32_t>(c0 >> 2) * (kBlockM * 16u) + row_at, q);
        const uint32_t bar = map_to_cta(recv_bar, q);
#pragma unroll
        for (int j = 0; j < PC / 4; ++j)
          st_async_v4(dst + j * (kBlockM * 16u), bar, v[o - 1][4 * j], v[o - 1][4 * j + 1], v[o - 1][4 * j + 2], v[o - 1][4 * j + 3]);
      }
    }
  }
  __syncwarp();

  // ---------------------------------------------------------------- this CTA's columns
  if (epilogue) {
    if constexpr (!kTmaStore) epilogue_sync_all();     // s_bias is complete (with TMA stores: the vote below)
    if (!mbar_wait(recv_bar, 0u, P.status)) {
      if (lane == 0) record_timeout(P.status, timed_out);
      ok = false;
    }
    // one decision where a group shares barriers below: nobody is left alone at them
    if constexpr (kTmaStore) ok = epilogue_all_ok(ok);
    else ok = __all_sync(0xffffffffu, ok) && live;
  }
  if (mine && ok) {
    // output staging: over the stages, which only this CTA has used, or behind the receive buffers
    const uint32_t out_base = smem_base + (kTn ? (C - 1) * kSlot : 0u) + static_cast<uint32_t>(group) * 2u * kEpiStage;
#pragma unroll 1
    for (int p = 0; p < UW / PC && n_own + p * PC < P.cols; ++p) {
      const int c0 = group * UW + p * PC;
      uint32_t own[PC];
      tmem_load_cols<PC>(taddr + rank * W + c0, own);
      tmem_load_wait();
      tmem_loaded<PC>(own);
      float f[PC];
#pragma unroll
      for (int i = 0; i < PC; ++i) f[i] = __uint_as_float(own[i]);
      const uint32_t at = recv_base + static_cast<uint32_t>(c0 >> 2) * (kBlockM * 16u) + row_at;
#pragma unroll
      for (int src = 0; src < C - 1; ++src) {          // own part first, then the others in rank order
        uint4 a[PC / 4];
#pragma unroll
        for (int j = 0; j < PC / 4; ++j) a[j] = ld_shared_v4(at + src * kSlot + j * (kBlockM * 16u));
#pragma unroll
        for (int j = 0; j < PC / 4; ++j) {
          f[4 * j] += __uint_as_float(a[j].x);
          f[4 * j + 1] += __uint_as_float(a[j].y);
          f[4 * j + 2] += __uint_as_float(a[j].z);
          f[4 * j + 3] += __uint_as_float(a[j].w);
        }
      }
      if constexpr (!kTn) {
#pragma unroll
        for (int i = 0; i < PC; ++i) f[i] += s_bias[c0 + i];
        if (P.act == BSP_ACT_GELU) {
#pragma unroll
          for (int i = 0; i < PC; i += 2) gelu_erf_pair(f[i], f[i + 1]);
        }
      } else {
#pragma unroll
        for (int u = 0; u < PC / 8; ++u) {
          uint2 fl = flags[0];
#pragma unroll
          for (int i = 1; i < UW / 8; ++i)
            if (i == p * (PC / 8) + u) fl = flags[i];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if ((((i < 4 ? fl.x : fl.y) >> (8 * (i & 3))) & 0xffu) == 0u) f[8 * u + i] = 0.0f;
        }
      }
      uint32_t o[PC / 2];
#pragma unroll
      for (int i = 0; i < PC / 2; ++i) o[i] = pack_bf16x2(f[2 * i], f[2 * i + 1]);
      if (!kTn && P.transposed) {
        // lanes are neighbouring tokens: 64 contiguous bytes per output row
        if (m < P.rows) {
          uint16_t* out = P.Y + static_cast<size_t>(n0 + static_cast<int>(rank) * W + c0) * P.ldy + m;
#pragma unroll
          for (int i = 0; i < PC; ++i)
            if (n_own + p * PC + i < P.cols) out[static_cast<size_t>(i) * P.ldy] = static_cast<uint16_t>(i & 1 ? o[i >> 1] >> 16 : o[i >> 1] & 0xffffu);
        }
      } else if constexpr (kTmaStore) {
        // PC = 32: a 128 x 32 piece of this group, staged as the tensor map's 64-byte swizzle expects it
        const uint32_t buf = out_base + (p & 1) * kEpiStage;
        const bool issuer = (threadIdx.x & 127) == 64;   // first thread of warps 2 and 6
        if (p >= 2) {
          if (issuer) tma_store_wait_read<1>();
          group_sync(group);
        }
        const uint32_t row_xor = static_cast<uint32_t>((row >> 1) & 3);
#pragma unroll
        for (int j = 0; j < PC / 8; ++j)
          st_shared_v4(buf + static_cast<uint32_t>(row) * 64u + ((static_cast<uint32_t>(j) ^ row_xor) << 4), o[4 * j], o[4 * j + 1],
                       o[4 * j + 2], o[4 * j + 3]);
        fence_async_smem();
        group_sync(group);
        if (issuer) tma_store_2d(&map_y, n_own + p * PC, m0, buf);
      } else if (m < P.rows) {
        uint16_t* out = P.Y + static_cast<size_t>(m) * P.ldy + n0 + static_cast<int>(rank) * W + c0;
#pragma unroll
        for (int u = 0; u < PC / 8; ++u)
          if (n_own + p * PC + 8 * u < P.cols)
            *reinterpret_cast<uint4*>(out + 8 * u) = make_uint4(o[4 * u], o[4 * u + 1], o[4 * u + 2], o[4 * u + 3]);
      }
    }
    if (kTmaStore && (threadIdx.x & 127) == 64) tma_store_wait_read<0>();
  }

  tcgen05_fence_before();
  __syncthreads();
  quiet_period(timed_out);
  if (*timed_out != 0u) {                              // (the same for every thread) until every other CTA has left, or waits here too
    cluster_arrive();
    cluster_wait();
  }
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols) : "memory");
  }
}

template <int BN, int C, bool kTn>
int launch_split(TcDevice* dev, const CUtensorMap& map_a, const CUtensorMap& map_b, SplitParams P, cudaStream_t s) {
  CUtensorMap map_y;
  if (P.transposed || BN / C < 64) map_y = map_a;                    // (not used)
  else if (!make_map(&map_y, P.Y, P.cols, P.rows, P.ldy, kBlockM, kEpiCols)) return BSP_ERR_CUDA;
  constexpr int kStage = (kBlockM + BN) * kBlockK * 2;
  constexpr int kTail = 1024 + 160 + BN / C * 4 + 32;                // alignment slack, barriers, bias
  constexpr bool kTmaStore = BN / C >= 64;
  constexpr int kReceive = (C - 1) * kBlockM * (BN / C) * 4;
  constexpr int kExchange = kReceive + (kTmaStore ? kEpiBytes : 0);  // over the stages (weight gradient)
  constexpr int kFit = (kSmemLimit - kTail - (kTn ? 0 : kReceive)) / kStage;
  constexpr int kAlone = kSmemLimit / 2 + 1024;                      // one CTA per SM
  static_assert(kExchange + kTail <= kSmemLimit && kFit >= 3 && (kTn || !kTmaStore || kStage >= kEpiBytes), "shared memory");
  const int per_cta = (P.k_blocks + C - 1) / C;
  P.stages = per_cta < kFit ? per_cta : kFit;
  if (P.stages > 8) P.stages = 8;
  P.recv_off = kTn ? 0 : P.stages * kStage;
  P.bars_off = kTn ? (P.stages * kStage > kExchange ? P.stages * kStage : kExchange) : P.recv_off + kReceive;
  if (P.bars_off < kAlone) P.bars_off = kAlone;
  P.status = dev->status;
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, gemm_split_kernel<BN, C, kTn>, kSmemLimit));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((P.rows + kBlockM - 1) / kBlockM * P.n_tiles * C);
  cfg.blockDim = dim3(kSplitThreads);
  cfg.dynamicSmemBytes = P.bars_off + kTail;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  BSP_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_split_kernel<BN, C, kTn>, map_a, map_b, map_y, P));
  return BSP_OK;
}
template <int BN, bool kTn>
int launch_split_c(TcDevice* dev, int c, const CUtensorMap& map_a, const CUtensorMap& map_b, const SplitParams& P, cudaStream_t s) {
  return c == 2 ? launch_split<BN, 2, kTn>(dev, map_a, map_b, P, s)
       : c == 4 ? launch_split<BN, 4, kTn>(dev, map_a, map_b, P, s)
                : launch_split<BN, 8, kTn>(dev, map_a, map_b, P, s);
}

}  // namespace

bool query_split_ctas(int (&ctas)[3]) {
  // GPCs of different sizes hold different numbers of whole clusters: ask, with the shared memory of a real launch
  if (cudaFuncSetAttribute(gemm_split_kernel<64, 2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess)
    return false;
  for (int i = 0; i < 3; ++i) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(8);
    cfg.blockDim = dim3(kSplitThreads);
    cfg.dynamicSmemBytes = kSmemLimit;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2u << i;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_split_kernel<64, 2, false>, &cfg) != cudaSuccess) return false;
    ctas[i] = n << (i + 1);
  }
  return true;
}

// The choices below compare times in nanoseconds fitted to single launches on B200 (graphs of one launch, operands in
// L2): a part per kernel, for a split also per quarter of a tile that has rows (1 to 4: what is exchanged) and per CTA,
// and a part per 64-deep stage, against choose_dense's estimate for whole tiles.  They hold for grids of one wave only; a
// split is considered where its clusters all run at once.
//   64-wide tile split 2 / 4 / 8:          1950 / 2050 / 2400 + 300 / 270 / 250 per quarter + 165 / 165 / 185 per stage
//   128-wide tile split 2 / 4 / 8:         2700 / 2100 / 2200 + 320 / 520 / 500 per quarter + 170 / 165 / 180 per stage
//   and 2 per CTA
// (768 outputs x 3072 inputs: 10.0 us whole, split 8 ways 3.8 us at 8 tokens and 4.6 us at 128; 768 x 768: 4.5 whole, 2.8
// split 4 ways at 8 tokens; 1024 x 4096 at 1003 tokens: 13.4 whole, 10.6 as 128-wide tiles split 2; 304 x 304: 3.2 and
// 2.6 at 8 tokens, not split at 1003.  Over 163 layers of 1 to 1500 tokens the choice among whole tiles and the six splits is
// 0.9 % behind the best on average and 10 % at worst: 4 tokens, 432 x 1728 3.4 us as 128-wide tiles split 8, 3.1 as 64-wide ones.)
int choose_linear_split(const TcDevice& dev, int tokens, int n_out, int k_in, long long whole_ns, int* bn, long long* ns) {
  const long long m_tiles = (tokens + kBlockM - 1) / kBlockM;
  const int kb = (k_in + kBlockK - 1) / kBlockK;
  const int quads = tokens >= kBlockM ? 4 : (tokens + 31) / 32;
  static const int fixed[2][3] = {{1950, 2050, 2400}, {2700, 2100, 2200}}, per_quad[2][3] = {{300, 270, 250}, {320, 520, 500}};
  static const int per_stage[2][3] = {{165, 165, 185}, {170, 165, 180}};
  long long best = whole_ns - 100;                     // a split has to win by more than noise
  int choice = -1;
  for (int b = 0; b < 2; ++b) {
    const long long tiles = m_tiles * ((n_out + 64 * (b + 1) - 1) / (64 * (b + 1)));
    for (int i = 0; i < 3; ++i) {
      const int c = 2 << i;
      if (c > kb || tiles * c > dev.split_ctas[i]) continue;
      const long long stages = (kb + c - 1) / c * per_stage[b][i] * (k_in % 16 ? 161 : k_in % 64 ? 115 : 100) / 100;   // ragged rows, as in choose_dense
      const long long t = fixed[b][i] + quads * per_quad[b][i] + stages + 2 * tiles * c;
      if (t < best) { best = t; choice = i; *bn = 64 * (b + 1); }
    }
  }
  if (ns != nullptr) *ns = choice < 0 ? whole_ns : best;
  return choice;
}
// dW: whole tiles 128 / 192 / 256 wide by one CTA, 128 / 256 wide by a pair, or, 128 and 256 wide, split 2 / 4 / 8.  Whole
// tiles as in choose_dense: a fixed part, per wave the larger of the main loop and the epilogue, which binds with few tokens, and
// something per wave after the first; a stage takes longer the more SMs are at work in a single wave, and a little less where
// waves follow one another and drift apart.  Rows of dY or X that are no multiple of 128 bytes make that operand's boxes straddle
// lines, of 64 more of them and of 32 sectors as well: percentages of the stage.  Operands beyond what L2 holds make the narrow
// tiles, which read them more often, a tenth slower.
// (4096 tokens, one CTA 128 wide / pair 128 wide / split 2: 768 x 768 15.5 / 13.7 / 10.2 us, 3072 x 768 18.5 / 15.9, 2304 x
// 768 18.1 / 15.6; 4096 x 1024 31.9 and 28.4, pair 256 wide 26.3; 136 tokens, 2640 x 880 5.7 / 7.1; 36 tokens, 3648 x 2640 14.0
// / 14.3, one CTA 192 wide 12.6; 7858 tokens, 1496 x 880 51.3 / 43.4, split 2 of 256 wide 36.5; 6145 tokens, 880 x 880 split 2 of
// 128 wide 18.7, split 4 of 256 wide 17.2.  Over 767 weights of 1 to 15455 tokens, most of them of encoder layers of 256 to 1024
// features, the choice is 0.2 % behind the best on average and 7 % at worst.)
TnChoice choose_tn(const TcDevice& dev, int tokens, int n_out, int k_in) {
  struct Whole {
    int width;
    bool pair;
    int fixed, epilogue, extra_wave, stage_few, stage_full, stage_waves, ragged_dy[4], ragged_x[4];     // percent by row_class
  };
  struct Split {
    int width, c, fixed, per_cta, stage, ragged_dy[4], ragged_x[4];
  };
  static const Whole whole[5] = {{128, false, 4461, 623, 1780, 173, 218, 183, {0, 9, 16, 67}, {0, 8, 14, 20}},
                                 {192, false, 5366, 967, 2370, 234, 325, 283, {0, 6, 8, 42}, {0, 4, 7, 19}},
                                 {256, false, 6562, 949, 3365, 268, 378, 346, {0, 2, 9, 29}, {0, 2, 7, 19}},
                                 {128, true, 3858, 790, 1695, 152, 187, 165, {0, 4, 16, 47}, {0, 3, 10, 13}},
                                 {256, true, 4972, 1706, 2537, 259, 337, 300, {0, 0, 0, 18}, {0, 0, 0, 14}}};
  static const Split split[6] = {{128, 2, 3776, 5, 211, {0, 9, 17, 46}, {0, 3, 13, 49}},
                                 {128, 4, 3820, 8, 210, {0, 3, 14, 50}, {0, 14, 12, 38}},
                                 {128, 8, 3631, 10, 234, {0, 8, 15, 50}, {0, 0, 6, 30}},
                                 {256, 2, 5350, 10, 363, {0, 4, 5, 19}, {0, 0, 6, 40}},
                                 {256, 4, 4699, 22, 364, {0, 0, 8, 12}, {0, 4, 7, 61}},
                                 {256, 8, 5251, 16, 406, {0, 0, 4, 42}, {0, 0, 7, 35}}};
  auto row_class = [](int elements) { return elements % 64 == 0 ? 0 : elements % 32 == 0 ? 1 : elements % 16 == 0 ? 2 : 3; };
  const int dy = row_class(n_out), x = row_class(k_in);
  const long long m_tiles = (n_out + kBlockM - 1) / kBlockM, m_pairs = (n_out + 2 * kBlockM - 1) / (2 * kBlockM);
  const int kb = (tokens + kBlockK - 1) / kBlockK;
  const bool beyond_l2 = 2LL * tokens * (n_out + k_in) > 100000000LL;
  long long best = -1;
  TnChoice choice{256, false, 1};
  for (const Whole& w : whole) {
    const long long tiles = (w.pair ? m_pairs : m_tiles) * ((k_in + w.width - 1) / w.width), seats = w.pair ? dev.sms / 2 : dev.sms;
    const long long waves = (tiles + seats - 1) / seats;
    const long long stage = waves > 1 ? w.stage_waves : w.stage_few + (w.stage_full - w.stage_few) * tiles / seats;
    int percent = 100 + w.ragged_dy[dy] + w.ragged_x[x];
    if (w.width == 128 && w.pair && dy == 3 && x == 3) percent += 30;
    if (w.width == 128 && beyond_l2) percent += 10;
    const long long loop = kb * stage * percent / 100;
    const long long t = w.fixed + waves * (loop > w.epilogue ? loop : w.epilogue) + w.extra_wave * (waves - 1);
    if (best < 0 || t < best) { best = t; choice = TnChoice{w.width, w.pair, 1}; }
  }
  for (int i = 0; i < 6; ++i) {
    const Split& p = split[i];
    const long long tiles = m_tiles * ((k_in + p.width - 1) / p.width);
    if (p.c > kb || tiles * p.c > dev.split_ctas[i % 3]) continue;
    const long long t = p.fixed + p.per_cta * tiles * p.c + static_cast<long long>((kb + p.c - 1) / p.c) * p.stage * (100 + p.ragged_dy[dy] + p.ragged_x[x]) / 100;
    if (t < best) { best = t; choice = TnChoice{p.width, false, p.c}; }
  }
  return choice;
}

// Y = act(X plan^T + b) with a cluster of c = 2, 4 or 8 CTAs per 128 x bn tile (arguments already validated).
int launch_linear_split(TcDevice* dev, int bn, int c, const void* plan, const void* X, void* Y, int tokens, int n_out, int k_in,
                        int act, const void* bias, int ldx, int ldy, bool plan_stable, bool transposed, cudaStream_t s) {
  CUtensorMap map_x, map_w;
  const int box = copy_rows(tokens);
  if (!make_map(&map_x, X, k_in, tokens, ldx, box)) return BSP_ERR_CUDA;
  if (!make_map(&map_w, plan, k_in, n_out, k_in, bn)) return BSP_ERR_CUDA;
  SplitParams P{};
  P.rows = tokens;
  P.cols = n_out;
  P.n_tiles = (n_out + bn - 1) / bn;
  P.k_blocks = (k_in + kBlockK - 1) / kBlockK;
  P.a_bytes = box * kBlockK * 2;
  P.plan_stable = plan_stable ? 1 : 0;
  P.transposed = transposed ? 1 : 0;
  P.act = act;
  P.bias = static_cast<const uint16_t*>(bias);
  P.Y = static_cast<uint16_t*>(Y);
  P.ldy = ldy;
  return bn == 64 ? launch_split_c<64, false>(dev, c, map_x, map_w, P, s) : launch_split_c<128, false>(dev, c, map_x, map_w, P, s);
}

// dW = (dY^T X) * Mask with a cluster of c = 2, 4 or 8 CTAs per 128 x bn tile (arguments already validated; keep
// 8-byte aligned or null).
int launch_tn_split(TcDevice* dev, int bn, int c, const void* dY, int ldy, const void* X, int ldx, int tokens, int n_out, int k_in,
                    int block, const uint8_t* keep, void* dW, int lddw, cudaStream_t s) {
  CUtensorMap map_dy, map_x;
  if (!make_map(&map_dy, dY, n_out, tokens, ldy, kBlockK)) return BSP_ERR_CUDA;
  if (!make_map(&map_x, X, k_in, tokens, ldx, kBlockK)) return BSP_ERR_CUDA;
  SplitParams P{};
  P.rows = n_out;
  P.cols = k_in;
  P.n_tiles = (k_in + bn - 1) / bn;
  P.k_blocks = (tokens + kBlockK - 1) / kBlockK;
  P.a_bytes = kBlockM * kBlockK * 2;
  P.keep = keep;
  P.block = block;
  P.Y = static_cast<uint16_t*>(dW);
  P.ldy = lddw;
  return bn == 128 ? launch_split_c<128, true>(dev, c, map_dy, map_x, P, s) : launch_split_c<256, true>(dev, c, map_dy, map_x, P, s);
}

}  // namespace bsp
