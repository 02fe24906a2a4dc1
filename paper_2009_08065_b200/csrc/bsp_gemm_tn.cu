// bsp_linear_backward_weight: the weight gradient of the masked layer that Algorithm 2 retrains
// (W = W * Mask):  dW = (dY^T X) * Mask,  dY [tokens, n_out], X [tokens, k_in], dW [n_out, k_in].
//
// The contraction runs over tokens, the slow dimension of both operands, so the tensor-core tiles
// are "MN-major": a pipeline stage holds 64 token rows of dY (128 output-row elements wide) and of
// X (128, 192 or 256 columns wide), each loaded as boxes of 64 elements x 64 token rows with the 128-byte
// swizzle; in shared memory that is a stack of 1024-byte atoms (8 token rows x 64 elements), 8 KB
// from one 64-element column group to the next, which is what the MN-major form of the tcgen05
// shared-memory descriptor describes (leading byte offset = distance between 64-element groups,
// stride byte offset = distance between 8-row groups).  Everything else (persistent CTAs, TMA
// producers, one MMA-issuing thread, two TMEM accumulators, two epilogue groups, TMA stores,
// bounded waits) is the pipeline of bsp_linear_tc.cu with a 128 x BN output tile.
// The epilogue applies the mask (pruned groups of dW are written as zero).  Most weights go to the CTA pairs of
// bsp_linear_tc2.cu or, with fewer tiles than SMs, to the split contraction of bsp_gemm_split.cu instead (choose_tn).
#include "bsp_tc.cuh"

namespace bsp {
using namespace tc;

namespace {

constexpr int kTnThreads = kThreads + 32;          // producer A, MMA, 8 epilogue warps, producer B

// bf16 x bf16 -> float32, both operands MN-major (bits 15 and 16), M = 128, N = BN.
__host__ __device__ constexpr uint32_t tn_idesc(int bn) { return instr_desc_bf16(bn) | (1u << 15) | (1u << 16); }

struct TnParams {
  int tokens, n_out, k_in;
  const uint8_t* keep;       // per-group flags [n_out / block, k_in], 8-byte aligned, or null
  int block;
  int* status;
};

template <int BN>
__global__ void __launch_bounds__(kTnThreads, 1)
gemm_tn_kernel(const __grid_constant__ CUtensorMap map_dy, const __grid_constant__ CUtensorMap map_x,
               const __grid_constant__ CUtensorMap map_dw, TnParams P) {
  using Cfg = TileCfg<BN>;
  constexpr int S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint16_t* s_zero = reinterpret_cast<uint16_t*>(smem + S * Cfg::kStage + kEpiBytes);       // zero "bias"
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * Cfg::kStage + kEpiBytes + 2 * BN * 2);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 2 * S + 4);
  volatile uint32_t* timed_out = tmem_holder + 1;     // set by a role whose wait expired

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t bar_base = smem_u32(bars);
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (S + s); };
  auto acc_full_bar = [&](int a) { return bar_base + 8u * (2 * S + a); };
  auto acc_empty_bar = [&](int a) { return bar_base + 8u * (2 * S + 2 + a); };

  if (threadIdx.x == 0) {
    *timed_out = 0u;
    for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 8); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  for (int c = threadIdx.x; c < 2 * BN; c += blockDim.x) s_zero[c] = 0;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = *tmem_holder;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // output tile (mt, nt): rows [128 mt, +128) of dW (output features), columns [256 nt, +256) (input features)
  const int m_tiles = (P.n_out + kBlockM - 1) / kBlockM;
  const int n_tiles = (P.k_in + BN - 1) / BN;
  const int total_tiles = m_tiles * n_tiles;
  const int k_blocks = (P.tokens + kBlockK - 1) / kBlockK;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the dY tiles
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile / n_tiles) * kBlockM;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        const uint32_t a_dst = smem_base + stage * Cfg::kStage;
        tma_stage_load(a_dst, &map_dy, m0, kb * kBlockK, full_bar(stage), Cfg::kStageA);
        tma_load_2d_elect(a_dst + kAtomGroup, &map_dy, m0 + 64, kb * kBlockK, full_bar(stage));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 10) {
    // ---------------------------------------------------------------- TMA producer of the X tiles
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int n0 = (tile % n_tiles) * BN;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        const uint32_t b_dst = smem_base + stage * Cfg::kStage + Cfg::kStageA;
        tma_stage_load(b_dst, &map_x, n0, kb * kBlockK, full_bar(stage), Cfg::kStageB);
#pragma unroll
        for (int g = 1; g < BN / 64; ++g)
          tma_load_2d_elect(b_dst + g * kAtomGroup, &map_x, n0 + 64 * g, kb * kBlockK, full_bar(stage));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    int stage = 0;
    uint32_t phase = 0;
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      if (!mbar_wait_warp(acc_empty_bar(acc), acc_phase[acc] ^ 1u, P.status)) { ok = false; break; }
      tcgen05_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(acc * BN);
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(full_bar(stage), phase, P.status)) { ok = false; break; }
        tcgen05_fence_after();
        const uint32_t a_addr = smem_base + stage * Cfg::kStage;
        const uint32_t b_addr = a_addr + Cfg::kStageA;
        // 16 token rows = two 8-row atoms = 2048 bytes per step
        mma_stage<128, 128>(d_tmem, smem_desc_mn_sw128(a_addr), smem_desc_mn_sw128(b_addr), tn_idesc(BN), kb != 0 ? 1u : 0u, empty_bar(stage));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
      if (!ok) break;
      tcgen05_commit_elect(acc_full_bar(acc));
      acc_phase[acc] ^= 1u;
      acc ^= 1;
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp >= 2 && warp < 10) {
    // ---------------------------------------------------------------- epilogue (as in bsp_linear_tc.cu, no bias)
    const int group = (warp - 2) >> 2;
    const int quad = warp & 3;
    const int row = quad * 32 + lane;
    const int epi_tid = threadIdx.x - 64;
    const bool issuer = (epi_tid & 127) == 0;
    const uint32_t buf0 = smem_base + S * Cfg::kStage + group * 2 * kEpiStage;
    uint32_t my_piece = 0;
    const uint32_t row_off = static_cast<uint32_t>(row) * 64u;
    const uint32_t row_xor = static_cast<uint32_t>((row >> 1) & 3);
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile / n_tiles) * kBlockM, n0 = (tile % n_tiles) * BN;
      // all 256 threads take the same decision, so nobody is left alone at a named barrier below
      if (!epilogue_all_ok(mbar_wait(acc_full_bar(acc), acc_phase[acc], P.status))) { ok = false; break; }
      tcgen05_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(acc * BN);
      const int pieces = (min(BN, P.k_in - n0) + kEpiCols - 1) / kEpiCols;
      bool released = false;
#pragma unroll 1
      for (int pc = group; pc < pieces; pc += 2) {
        const int c0 = pc * kEpiCols;
        const uint32_t buf = buf0 + (my_piece & 1u) * kEpiStage;
        ++my_piece;
        if (issuer) tma_store_wait_read<1>();
        group_sync(group);
        EpiloguePiece piece;
        uint2 flags[kEpiCols / 8];
#pragma unroll
        for (int j = 0; j < kEpiCols / 8; ++j) {     // (k_in is a multiple of 8: eight columns are inside or outside)
          flags[j] = make_uint2(0x01010101u, 0x01010101u);
          const int n = n0 + c0 + 8 * j;
          if (P.keep != nullptr && m0 + row < P.n_out && n < P.k_in)
            flags[j] = ld_global(reinterpret_cast<const uint2*>(P.keep + static_cast<size_t>((m0 + row) / P.block) * P.k_in + n));
        }
        piece_load(taddr + c0, smem_u32(s_zero), piece);
        if (P.keep != nullptr) {
#pragma unroll
          for (int i = 0; i < kEpiCols; ++i)
            if ((((i & 4 ? flags[i >> 3].y : flags[i >> 3].x) >> (8 * (i & 3))) & 0xffu) == 0u) piece.v[i] = 0u;
        }
        if (pc + 2 >= pieces) {
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty_bar(acc));
          released = true;
        }
        piece_store(piece, BSP_ACT_NONE, buf + row_off, row_xor);
        fence_async_smem();
        group_sync(group);
        if (issuer) {
          tma_store_2d(&map_dw, n0 + c0, m0, buf);
        }
      }
      if (!released) {
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty_bar(acc));
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
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
  }
}

template <int BN>
int launch_tn(TcDevice* dev, const CUtensorMap& map_dy, const CUtensorMap& map_x, const CUtensorMap& map_dw, const TnParams& P,
              cudaStream_t s) {
  using Cfg = TileCfg<BN>;
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, gemm_tn_kernel<BN>, Cfg::kSmemBytes));
  const int tiles = ((P.n_out + kBlockM - 1) / kBlockM) * ((P.k_in + BN - 1) / BN);
  BSP_CUDA_TRY(launch_pdl(gemm_tn_kernel<BN>, dim3(tiles < dev->sms ? tiles : dev->sms), dim3(kTnThreads), Cfg::kSmemBytes, s, map_dy,
                          map_x, map_dw, P));
  return BSP_OK;
}

}  // namespace
}  // namespace bsp

extern "C" int bsp_linear_backward_weight(const void* dY, int ldy, const void* X, int ldx, int tokens, int n_out,
                                          int k_in, int block, const uint8_t* keep, void* dW, int lddw, void* stream) {
  using namespace bsp;
  if (dY == nullptr || X == nullptr || dW == nullptr) return BSP_ERR_ARG;
  if (tokens <= 0 || n_out <= 0 || k_in <= 0 || block <= 0) return BSP_ERR_ARG;
  if (n_out % block) return BSP_ERR_SHAPE;
  if (ldy < n_out || ldx < k_in || lddw < k_in) return BSP_ERR_SHAPE;
  if (!aligned_to(dY, 16) || !aligned_to(X, 16) || !aligned_to(dW, 16) || ldy % 8 || ldx % 8 || lddw % 8 || n_out % 8 ||
      k_in % 8)
    return BSP_ERR_UNSUPPORTED;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  // (flags that are not 8-byte aligned are applied by the mask kernel afterwards)
  const uint8_t* flags = keep != nullptr && aligned_to(keep, 8) ? keep : nullptr;
  const TnChoice choice = choose_tn(*dev, tokens, n_out, k_in);
  const int bn = choice.bn;
  if (choice.pair || choice.cluster > 1) {
    const int st = choice.pair ? launch_tn_pair(dev, bn, dY, ldy, X, ldx, tokens, n_out, k_in, block, flags, dW, lddw, s)
                               : launch_tn_split(dev, bn, choice.cluster, dY, ldy, X, ldx, tokens, n_out, k_in, block, flags, dW, lddw, s);
    if (st != BSP_OK || keep == flags) return st;
    return bsp_apply_mask(dW, n_out, k_in, lddw, block, BSP_ORIENT_C, keep, stream);
  }
  // operands as [token rows, features]: inner dimension = features, boxes of 64 features x 64 token rows
  CUtensorMap map_dy, map_x, map_dw;
  if (!make_map(&map_dy, dY, n_out, tokens, ldy, kBlockK)) return BSP_ERR_CUDA;
  if (!make_map(&map_x, X, k_in, tokens, ldx, kBlockK)) return BSP_ERR_CUDA;
  if (!make_map(&map_dw, dW, k_in, n_out, lddw, kBlockM, kEpiCols)) return BSP_ERR_CUDA;
  const TnParams P{tokens, n_out, k_in, flags, block, dev->status};
  const int st = bn == 128   ? launch_tn<128>(dev, map_dy, map_x, map_dw, P, s)
                 : bn == 192 ? launch_tn<192>(dev, map_dy, map_x, map_dw, P, s)
                             : launch_tn<256>(dev, map_dy, map_x, map_dw, P, s);
  if (st != BSP_OK) return st;
  if (keep != flags) return bsp_apply_mask(dW, n_out, k_in, lddw, block, BSP_ORIENT_C, keep, stream);
  return BSP_OK;
}
