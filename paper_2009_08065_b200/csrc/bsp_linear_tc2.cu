// Tensor-core products by CTA pairs (tcgen05 cta_group::2): the linear layer and the weight gradient.
//
// The one-CTA kernels (bsp_linear_tc.cu, bsp_gemm_tn.cu) stream (128 + BN) x 64 operand elements from L2 per
// 128 x BN x 64 block of multiply-adds, and at BERT shapes it is this L2 -> SM traffic, not the tensor pipe, that
// binds: they move 15 to 17 TB/s over all SMs (131 bytes per ns and SM, 19 TB/s, is the most that was seen, by the 256 x 128
// tiles of the weight gradient).  Here two CTAs of a cluster share one 256 x BN output
// tile: each loads its own 128 rows of A and HALF of the BN rows of B, and one tcgen05.mma.cta_group::2 (M = 256)
// issued by the leader CTA reads both CTAs' shared memory and writes rows 0..127 / 128..255 of the accumulator
// into the two CTAs' tensor memories.  Per CTA that is (128 + BN / 2) x 64 elements per block: a third less
// at BN = 256, 30 % at 192, a quarter at 128.
//
// Two operand forms:
//   linear   Y = act(X plan^T + b): A = X, B = plan, K-major;
//   tn       dW = (dY^T X) * Mask: A = dY, B = X, MN-major (see bsp_gemm_tn.cu), BN = 128 or 256.
//
// What bounds it: with operands in L2 the tensor pipe at the clock that the power limit leaves (4096 x 768 x 3072 in
// 256 x 192 tiles: a 64-deep stage every 240 ns, the pipe's 384 cycles at 1.6 GHz; the one-CTA kernel with as many CTAs
// 300 ns), and around it what every launch pays: 1.0 us from the last CTA of the launch before until its wait returns, 0.5
// to 1.3 us until the first operands are there, 1.3 to 2 us of epilogue behind the last MMA.  A cluster barrier that orders
// memory at both ends (0.5 to 0.8 us each) and arrivals of cluster scope in the epilogue (1 us) had made pairs no faster
// than single CTAs up to some 8192 tokens.
//
// Roles per CTA: warps 0 and 10 TMA producers of A and B (completion is counted on the leader's mbarrier), warp 1
// of the LEADER issues the MMAs and commits to both CTAs' barriers, warps 2..9 epilogue of the CTA's own 128 rows
// (as in the one-CTA kernels).
// No TMA multicast is used.  All mbarrier waits are bounded.
#include "bsp_tc.cuh"

namespace bsp {
using namespace tc;

namespace {

constexpr int kPairThreads = kThreads + 32;                // and the second producer
template <int BN>
struct PairCfg {
  static constexpr int kStageA = kBlockM * kBlockK * 2;        // this CTA's 128 rows of A
  static constexpr int kStageB = (BN / 2) * kBlockK * 2;       // this CTA's half of the rows of B
  static constexpr int kStage = kStageA + kStageB;
  static constexpr int kFixed = 1024 + kEpiBytes + 2 * BN * 2 + 256;   // as in TileCfg
  static constexpr int kStages = (kSmemLimit - kFixed) / kStage > 8 ? 8 : (kSmemLimit - kFixed) / kStage;
  static constexpr int kSmemBytes = kStages * kStage + kFixed;
  static constexpr int kTmemCols = 2 * BN <= 256 ? 256 : 512;
};

// TMA load whose completion bytes are counted on the leader's mbarrier (a cluster address); `arm` > 0: that many bytes
// are expected of both CTAs first (the leader's own copy of the barrier).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar_cluster,
                                                 uint32_t bar_own, uint32_t arm) {
  asm volatile(
      "{\n\t.reg .pred e, a;\n\telect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.and.u32 a, %6, 0, e;\n\t"
      "@a mbarrier.arrive.expect_tx.shared::cta.b64 _, [%5], %6;\n\t"
      "@e cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n\t}"
      ::"r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster), "r"(bar_own), "r"(arm)
      : "memory");
}
// Commits to the same barrier of both CTAs (by an elected lane of a converged warp).
__device__ __forceinline__ void tcgen05_commit_pair(uint32_t bar_own, uint32_t bar_peer) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%1];\n\t}" ::"r"(bar_own), "r"(bar_peer)
      : "memory");
}
// One pipeline stage for the pair: four K = 16 steps, then the commits that free the stage in both CTAs.
template <int STEP_A, int STEP_B>
__device__ __forceinline__ void mma_stage_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate,
                                               uint32_t free_own, uint32_t free_peer) {
  asm volatile(
      "{\n\t.reg .pred p, t, e;\n\t.reg .b64 a1, a2, a3, b1, b2, b3;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\tsetp.eq.b32 t, 0, 0;\n\t"
      "add.s64 a1, %1, %7;\n\tadd.s64 a2, a1, %7;\n\tadd.s64 a3, a2, %7;\n\t"
      "add.s64 b1, %2, %8;\n\tadd.s64 b2, b1, %8;\n\tadd.s64 b3, b2, %8;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a1, b1, %3, t;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a2, b2, %3, t;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], a3, b3, %3, t;\n\t"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%5];\n\t"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%6];\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate), "r"(free_own), "r"(free_peer), "n"(STEP_A), "n"(STEP_B)
      : "memory");
}
// An arrival on a barrier of either CTA.  What it reports, reads of tensor memory, is complete and behind a tcgen05 fence;
// ordering the thread's other accesses at cluster scope as well took 1 us of a tile's epilogue.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar_cluster) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
// bf16 x bf16 -> float32, M = 256 (128 rows in each CTA of the pair), N = BN; bits 15 and 16: MN-major operands.
template <int BN, bool kTn>
constexpr uint32_t kPairIdesc = (1u << 4) | (1u << 7) | (1u << 10) | (kTn ? (1u << 15) | (1u << 16) : 0u) |
                                (static_cast<uint32_t>(BN >> 3) << 17) | (static_cast<uint32_t>(256 >> 4) << 24);

struct PairParams {
  int rows, cols, contraction;   // output matrix, and what is summed over
  int act;                   // linear
  int plan_stable;           // linear: the plan was complete before the kernel preceding this one in the stream began
  const uint16_t* bias;      // linear
  const uint8_t* keep;       // tn: per-group flags [rows / block, cols], 8-byte aligned, or null
  int block;                 // tn
  int* status;
};

template <int BN, bool kTn>
__global__ void __launch_bounds__(kPairThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                 const __grid_constant__ CUtensorMap map_y, const __grid_constant__ PairParams P) {
  using Cfg = PairCfg<BN>;
  constexpr int S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  // [S operand stages][epilogue staging buffers][bias, bf16, for two tiles][mbarriers, TMEM base]
  uint16_t* s_bias = reinterpret_cast<uint16_t*>(smem + S * Cfg::kStage + kEpiBytes);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * Cfg::kStage + kEpiBytes + 2 * BN * 2);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * S + 4);
  volatile uint32_t* timed_out = tmem_holder + 1;     // set by a role of this CTA whose wait expired

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();          // 0 = leader of the pair
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };                 // used in the leader only
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };          // one per CTA
  auto acc_full_bar = [&](int a) { return bar_base + 8u * (2 * S + a); };   // one per CTA
  auto acc_empty_bar = [&](int a) { return bar_base + 8u * (2 * S + 2 + a); };   // used in the leader only

  if (threadIdx.x == 0) {
    *timed_out = 0u;
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_a)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_b)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_y)) : "memory");
    for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }   // two producers arm a stage
    for (int a = 0; a < 2; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 16); }   // 8 warps x 2 CTAs
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (kTn) {
    for (int c = threadIdx.x; c < 2 * BN; c += kPairThreads) s_bias[c] = 0;
  }
  if (warp == 1) {   // the same warp in both CTAs, same destination offset
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  cluster_arrive_relaxed();      // this CTA's barriers exist (fenced above) and its tensor memory is allocated
  tcgen05_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  // (the weights of a stable plan are older than the kernel before this one: their producer neither waits nor signals,
  // see launch_pdl)
  if (kTn || !(P.plan_stable && warp == 10)) {
    pdl_wait();
    pdl_launch_dependents();
  }
  cluster_wait();                // and so do the other's, before anything signals across the pair

  const int m_tiles = (P.rows + 255) / 256;
  const int n_tiles = (P.cols + BN - 1) / BN;
  const int total_tiles = m_tiles * n_tiles;
  const int k_blocks = (P.contraction + kBlockK - 1) / kBlockK;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of A (both CTAs)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles && ok; tile += n_pairs) {
      const int m0 = (tile / n_tiles) * 256 + static_cast<int>(rank) * kBlockM;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        const uint32_t dst = smem_base + stage * Cfg::kStage, leader_full = map_to_cta(full_bar(stage), 0);
        const uint32_t arm = rank == 0 ? 2u * Cfg::kStageA : 0u;               // both CTAs' bytes
        if constexpr (kTn) {
          tma_load_2d_pair(dst, &map_a, m0, kb * kBlockK, leader_full, full_bar(stage), arm);
          tma_load_2d_pair(dst + kAtomGroup, &map_a, m0 + 64, kb * kBlockK, leader_full, full_bar(stage), 0u);
        } else {
          tma_load_2d_pair(dst, &map_a, kb * kBlockK, m0, leader_full, full_bar(stage), arm);
        }
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    // the leader's commits that free the last stages arrive here while this CTA still exists
    for (int i = 0; i < S && ok; ++i) {
      ok = mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status);
      if (++stage == S) { stage = 0; phase ^= 1u; }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 10) {
    // ---------------------------------------------------------------- TMA producer of B (both CTAs)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles && ok; tile += n_pairs) {
      const int n0 = (tile % n_tiles) * BN + static_cast<int>(rank) * (BN / 2);
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        const uint32_t dst = smem_base + stage * Cfg::kStage + Cfg::kStageA, leader_full = map_to_cta(full_bar(stage), 0);
        const uint32_t arm = rank == 0 ? 2u * Cfg::kStageB : 0u;
        if constexpr (kTn) {
#pragma unroll
          for (int g = 0; g < BN / 128; ++g)
            tma_load_2d_pair(dst + g * kAtomGroup, &map_b, n0 + 64 * g, kb * kBlockK, leader_full, full_bar(stage), g == 0 ? arm : 0u);
        } else {
          tma_load_2d_pair(dst, &map_b, kb * kBlockK, n0, leader_full, full_bar(stage), arm);
        }
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 1 && rank == 0) {
    // ---------------------------------------------------------------- MMA issuer (leader CTA only)
    int stage = 0;
    uint32_t phase = 0;
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles && ok; tile += n_pairs) {
      if (!mbar_wait_warp(acc_empty_bar(acc), acc_phase[acc] ^ 1u, P.status)) { ok = false; break; }
      tcgen05_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * BN);
      bool ready = false;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_probed(ready, full_bar(stage), phase, P.status)) { ok = false; break; }
        tcgen05_fence_after();
        const int next = stage + 1 == S ? 0 : stage + 1;
        const uint32_t next_phase = next ? phase : phase ^ 1u;
        ready = kb + 1 < k_blocks && mbar_try_wait(full_bar(next), next_phase);
        const uint32_t a_addr = smem_base + stage * Cfg::kStage, b_addr = a_addr + Cfg::kStageA;
        // the stage is free in both CTAs once these MMAs have read it
        const uint32_t free_peer = map_to_cta(empty_bar(stage), 1);
        if constexpr (kTn)
          mma_stage_pair<128, 128>(d_tmem, smem_desc_mn_sw128(a_addr), smem_desc_mn_sw128(b_addr), kPairIdesc<BN, kTn>, kb != 0 ? 1u : 0u,
                                   empty_bar(stage), free_peer);
        else
          mma_stage_pair<2, 2>(d_tmem, smem_desc_sw128(a_addr), smem_desc_sw128(b_addr), kPairIdesc<BN, kTn>, kb != 0 ? 1u : 0u,
                               empty_bar(stage), free_peer);
        stage = next;
        phase = next_phase;
      }
      if (!ok) break;
      tcgen05_commit_pair(acc_full_bar(acc), map_to_cta(acc_full_bar(acc), 1));
      acc_phase[acc] ^= 1u;
      acc ^= 1;
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp >= 2 && warp < 10) {
    // ---------------------------------------------------------------- epilogue of this CTA's 128 rows
    const int group = (warp - 2) >> 2;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const int epi_tid = threadIdx.x - 64;
    const bool issuer = (epi_tid & 127) == 0;
    const uint32_t buf0 = smem_base + S * Cfg::kStage + group * 2 * kEpiStage;   // this group's two staging buffers
    uint32_t my_piece = 0;                   // pieces staged by this group so far: selects the buffer
    const uint32_t row_off = static_cast<uint32_t>(row) * 64u;
    const uint32_t row_xor = static_cast<uint32_t>((row >> 1) & 3);
    constexpr int kPieces = BN / kEpiCols / 2;   // pieces of a tile that a group takes
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = pair; tile < total_tiles && ok; tile += n_pairs) {
      const int m0 = (tile / n_tiles) * 256 + static_cast<int>(rank) * kBlockM, n0 = (tile % n_tiles) * BN;
      uint2 flags[kTn ? kPieces * 4 : 1];    // tn: the flags of this thread's pieces, asked for before the wait for the accumulator
      if constexpr (kTn) {
#pragma unroll
        for (int i = 0; i < kPieces * 4; ++i) {      // (cols is a multiple of 8: eight columns are inside or outside)
          const int n = n0 + (group + 2 * (i >> 2)) * kEpiCols + 8 * (i & 3);
          flags[i] = make_uint2(0x01010101u, 0x01010101u);
          if (P.keep != nullptr && m0 + row < P.rows && n < P.cols)
            flags[i] = ld_global(reinterpret_cast<const uint2*>(P.keep + static_cast<size_t>((m0 + row) / P.block) * P.cols + n));
        }
      } else {
        for (int c = epi_tid; c < BN; c += 256)
          s_bias[acc * BN + c] = (P.bias != nullptr && n0 + c < P.cols) ? ld_global(P.bias + n0 + c) : static_cast<uint16_t>(0);
        epilogue_sync_all();
      }
      // all 256 threads take the same decision, so nobody is left alone at a named barrier below
      if (!epilogue_all_ok(mbar_wait(acc_full_bar(acc), acc_phase[acc], P.status))) { ok = false; break; }
      tcgen05_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(acc * BN);
      const uint32_t leader_acc_empty = map_to_cta(acc_empty_bar(acc), 0);
      const int pieces = (min(BN, P.cols - n0) + kEpiCols - 1) / kEpiCols;
      // (the last two tiles' accumulators are not waited for again: no arrival that could come when the leader has left)
      bool released = tile + 2 * n_pairs >= total_tiles;
#pragma unroll (kTn ? kPieces : 1)
      for (int i = 0; i < kPieces; ++i) {
        const int pc = group + 2 * i;
        if (pc >= pieces) break;
        const int c0 = pc * kEpiCols;
        const uint32_t buf = buf0 + (my_piece & 1u) * kEpiStage;
        ++my_piece;
        EpiloguePiece piece;
        piece_load(taddr + c0, smem_u32(s_bias + acc * BN + c0), piece);
        if constexpr (kTn) {
          if (P.keep != nullptr) {
#pragma unroll
            for (int e = 0; e < kEpiCols; ++e) {
              const uint2 f = flags[i * 4 + (e >> 3)];
              if ((((e & 4 ? f.y : f.x) >> (8 * (e & 3))) & 0xffu) == 0u) piece.v[e] = 0u;
            }
          }
        }
        if (issuer) tma_store_wait_read<1>();   // the store issued two pieces ago has read this buffer
        group_sync(group);
        if (pc + 2 >= pieces && !released) { // this warp's last read of the accumulator
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(leader_acc_empty);
          released = true;
        }
        piece_store(piece, kTn ? BSP_ACT_NONE : P.act, buf + row_off, row_xor);
        fence_async_smem();
        group_sync(group);
        if (issuer) tma_store_2d(&map_y, n0 + c0, m0, buf);
      }
      if (!released) {
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(leader_acc_empty);
      }
      acc_phase[acc] ^= 1u;
      acc ^= 1;
    }
    if (issuer) tma_store_wait_read<0>();
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  }

  tcgen05_fence_before();
  __syncthreads();
  quiet_period(timed_out);
  // Neither CTA leaves, or frees its tensor memory, while the other may still touch them.  Nothing is in flight between
  // the two by now (every arrival from the other CTA has been waited for), so the barrier orders no memory.
  cluster_arrive_relaxed();
  cluster_wait();
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
  }
}

template <int BN, bool kTn>
int launch_pair(TcDevice* dev, const CUtensorMap& map_a, const CUtensorMap& map_b, const CUtensorMap& map_y, const PairParams& P,
                cudaStream_t s) {
  using Cfg = PairCfg<BN>;
  static_assert(Cfg::kStages >= 4 && Cfg::kStage % 1024 == 0 && (!kTn || BN % 128 == 0), "stages");
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, gemm_pair_kernel<BN, kTn>, Cfg::kSmemBytes));
  const long long tiles = static_cast<long long>((P.rows + 255) / 256) * ((P.cols + BN - 1) / BN);
  const int pairs = tiles < dev->sms / 2 ? static_cast<int>(tiles) : dev->sms / 2;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kPairThreads);
  cfg.dynamicSmemBytes = Cfg::kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  BSP_CUDA_TRY(cudaLaunchKernelEx(&cfg, gemm_pair_kernel<BN, kTn>, map_a, map_b, map_y, P));
  return BSP_OK;
}

}  // namespace

// Launch of the CTA-pair kernel with tiles 256 x bn (arguments already validated by the caller).
int launch_tc_pair(TcDevice* dev, int bn, const void* plan, const void* X, void* Y, int tokens, int n_out, int k_in, int act,
                   const void* bias, int ldx, int ldy, bool plan_stable, cudaStream_t s) {
  CUtensorMap map_x, map_w, map_y;
  if (!make_map(&map_x, X, k_in, tokens, ldx, kBlockM)) return BSP_ERR_CUDA;
  if (!make_map(&map_w, plan, k_in, n_out, k_in, bn / 2)) return BSP_ERR_CUDA;
  if (!make_map(&map_y, Y, n_out, tokens, ldy, kBlockM, kEpiCols)) return BSP_ERR_CUDA;
  const PairParams P{tokens, n_out, k_in, act, plan_stable ? 1 : 0, static_cast<const uint16_t*>(bias), nullptr, 1, dev->status};
  return bn == 128   ? launch_pair<128, false>(dev, map_x, map_w, map_y, P, s)
         : bn == 192 ? launch_pair<192, false>(dev, map_x, map_w, map_y, P, s)
                     : launch_pair<256, false>(dev, map_x, map_w, map_y, P, s);
}

// dW = (dY^T X) * Mask with tiles 256 x bn, bn = 128 or 256 (arguments already validated; keep 8-byte aligned or null).
int launch_tn_pair(TcDevice* dev, int bn, const void* dY, int ldy, const void* X, int ldx, int tokens, int n_out, int k_in,
                   int block, const uint8_t* keep, void* dW, int lddw, cudaStream_t s) {
  CUtensorMap map_dy, map_x, map_dw;
  if (!make_map(&map_dy, dY, n_out, tokens, ldy, kBlockK)) return BSP_ERR_CUDA;
  if (!make_map(&map_x, X, k_in, tokens, ldx, kBlockK)) return BSP_ERR_CUDA;
  if (!make_map(&map_dw, dW, k_in, n_out, lddw, kBlockM, kEpiCols)) return BSP_ERR_CUDA;
  const PairParams P{n_out, k_in, tokens, BSP_ACT_NONE, 0, nullptr, keep, block, dev->status};
  return bn == 128 ? launch_pair<128, true>(dev, map_dy, map_x, map_dw, P, s) : launch_pair<256, true>(dev, map_dy, map_x, map_dw, P, s);
}

}  // namespace bsp
