// bsp_linear / bsp_linear_plan / bsp_linear_planned: the pruned linear layer on the B200 tensor
// cores (tcgen05.mma with float32 accumulators in tensor memory, operands staged by TMA).
//
// Execution layout ("plan").  A row-block's kept-column list differs from its neighbours', and a
// tcgen05 operand tile addresses K in contiguous 16-byte pieces, so single columns cannot be
// picked from a resident X tile by the hardware.  Re-gathering X per row-block would move
// 2 bytes through shared memory per `block` multiply-adds, which caps the tensor pipe at about
// block/64 of its peak.  The plan therefore scatters the packed values back to their natural
// column positions, zero elsewhere: a [n_out, k_in] bf16 matrix that TMA can tile directly,
// with X read in its natural order and reused by a whole 128 x BN output tile.  The packed form
// stays the storage format; the plan is private scratch derived from it.
//
// Kernel.  Persistent CTAs (one per SM) walk output tiles of 128 tokens x BN outputs.
//   warps 0 and 10   : TMA producers, X tile [128 x 64] and W tile [BN x 64] per pipeline stage
//                      (128-byte swizzle), completion on an mbarrier;
//   warp 1           : issues tcgen05.mma (M=128, N=BN, K=16) into one of two TMEM accumulators
//                      and commits stage release / accumulator ready to mbarriers;
//   warps 2..9       : epilogue, two groups of four warps; group g takes the 32-column pieces of
//                      the tile with index = g (mod 2).  Each warp tcgen05.ld's its 32 TMEM lanes
//                      (= 32 tokens), adds bias, optional GELU, rounds to bf16, writes its rows
//                      into the group's swizzled staging buffer, and one thread hands the
//                      128 x 32 piece to a TMA store (full-line writes, tails clipped by the
//                      tensor map).  The epilogue runs concurrently with the next tile's main
//                      loop on the other accumulator.
// Every wait is bounded by a wall-clock deadline (bsp_set_wait_limit_ms); on expiry the role records
// BSP_ERR_TIMEOUT in the status word and leaves its loop, the other roles then time out on their
// own waits (the epilogue threads by a common vote), and the CTA waits a millisecond for whatever
// it still has in flight, frees its tensor memory and exits.
#include <mutex>
#include <cstring>

#include "bsp_tc.cuh"

namespace bsp {

int check_linear_args(const void* a, const void* b, const void* c, int n_out, int k_in, int block,
                      const void* X, int tokens, int ldx, int act, const void* Y, int ldy);
int launch_tc_pair(TcDevice* dev, int bn, const void* plan, const void* X, void* Y, int tokens, int n_out, int k_in, int act,
                   const void* bias, int ldx, int ldy, bool plan_stable, cudaStream_t s);

using namespace tc;

namespace {

// [0]: 0, or BSP_ERR_TIMEOUT once a bounded wait expired; [1]: a counter nothing ever bumps (self-test);
// [2..3]: the limit of one wait in nanoseconds; [4]: waits that ran out in the last self-test;
// [6..7]: how long its mbarrier wait lasted, nanoseconds
__device__ __align__(16) int g_linear_status[8] = {0, 0, static_cast<int>(kDefaultWaitLimitNs & 0xffffffffull),
                                                   static_cast<int>(kDefaultWaitLimitNs >> 32), 0, 0, 0, 0};


struct LinearParams {
  int tokens, n_out, k_in, act;
  int plan_stable;      // the plan was complete before the kernel preceding this one in the stream began
  int a_bytes;          // bytes of one copy of an activation tile (copy_rows)
  int transposed;       // the output is written as [n_out, tokens] (map_y describes that matrix)
  const uint16_t* bias;
  int* status;
};

// Epilogue groups of four warps (one warp per quarter of the TMEM lanes), two staging buffers each.
// Four groups with one buffer each (the same 32 KB; the exposed epilogue of a CTA's last tile then takes
// two pieces per group instead of four) were measured 1.5 us slower per four-GEMM layer at 4096 tokens:
// sixteen warps contend for the shared memory that the operand copies and the tensor core keep busy.
constexpr int kGroups = 2;
constexpr int kEpiThreads = 128 * kGroups;
constexpr int kBufPerGroup = kEpiBuffers / kGroups;
constexpr int kWeightWarp = 2 + 4 * kGroups;            // the second TMA producer warp, for the weight tiles
constexpr int kThreadsTc = 32 * (kWeightWarp + 1);

// Named barriers of this kernel's epilogue: 5 + g among the 128 threads of group g, 3 and 4 among all of them.
__device__ __forceinline__ void tc_group_sync(int g) { asm volatile("bar.sync %0, 128;" ::"r"(5 + g) : "memory"); }
__device__ __forceinline__ void tc_epilogue_sync_all() { asm volatile("bar.sync 3, %0;" ::"n"(kEpiThreads) : "memory"); }
__device__ __forceinline__ bool tc_epilogue_all_ok(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, 4, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(ok ? 1u : 0u), "n"(kEpiThreads)
      : "memory");
  return r != 0u;
}

template <int BN>
__global__ void __launch_bounds__(kThreadsTc, 1)
linear_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                 const __grid_constant__ CUtensorMap map_y, LinearParams P) {
  using Cfg = TileCfg<BN>;
  constexpr int S = Cfg::kStages;
  extern __shared__ uint8_t smem_raw[];
  // operand stages need 1024-byte alignment for the 128-byte swizzle pattern
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  // [S operand stages][2 epilogue staging buffers][bias, bf16, for two tiles][mbarriers, TMEM base]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + S * Cfg::kStage + kEpiBytes + 2 * BN * 2);
  // bars[0..S) full, [S..2S) empty, [2S..2S+2) accumulator full, [2S+2..2S+4) accumulator empty
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
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_w)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_y)) : "memory");
    for (int s = 0; s < S; ++s) { mbar_init(full_bar(s), 2); mbar_init(empty_bar(s), 1); }   // two producers arm a stage
    for (int a = 0; a < 2; ++a) { mbar_init(acc_full_bar(a), 1); mbar_init(acc_empty_bar(a), 4 * kGroups); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                 "r"(static_cast<uint32_t>(Cfg::kTmemCols)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  // Programmatic dependent launch: everything above touched only this CTA's shared and tensor
  // memory and overlaps the tail of the previous kernel in the stream.  From here on the kernel
  // reads memory that kernel may have written (X, the plan), so wait for it to finish; and let
  // the next kernel in the stream start its own prologue as soon as SMs become free.  When the
  // caller vouches that the plan is older than the previous kernel, the weight producer does not
  // wait: its first tiles are on their way while the previous kernel finishes writing X.  It leaves
  // the signal to the warps that have waited: one thread's signal counts for its CTA, and the kernel
  // that it lets in may read weights at once in the same way (see launch_pdl).
  if (!(P.plan_stable && warp == kWeightWarp)) {
    pdl_wait();
    pdl_launch_dependents();
  }

  const int m_tiles = (P.tokens + kBlockM - 1) / kBlockM;
  const int n_tiles = (P.n_out + BN - 1) / BN;
  const int total_tiles = m_tiles * n_tiles;
  const int k_blocks = (P.k_in + kBlockK - 1) / kBlockK;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer of the X tiles
    // (the two operands of a stage are issued by two warps, this one and the last one, so neither waits
    // behind the other's copy)
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile / n_tiles) * kBlockM;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        const uint32_t a_dst = smem_base + stage * Cfg::kStage;
        tma_stage_load(a_dst, &map_x, kb * kBlockK, m0, full_bar(stage), static_cast<uint32_t>(P.a_bytes));
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == kWeightWarp) {
    // ---------------------------------------------------------------- TMA producer of the weight tiles
    int stage = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int n0 = (tile % n_tiles) * BN;
      for (int kb = 0; kb < k_blocks; ++kb) {
        if (!mbar_wait_warp(empty_bar(stage), phase ^ 1u, P.status)) { ok = false; break; }
        tma_stage_load(smem_base + stage * Cfg::kStage + Cfg::kStageA, &map_w, kb * kBlockK, n0, full_bar(stage), Cfg::kStageB);
        if (++stage == S) { stage = 0; phase ^= 1u; }
      }
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    constexpr uint32_t idesc = instr_desc_bf16(BN);
    int stage = 0;
    uint32_t phase = 0;
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
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
        const uint32_t a_addr = smem_base + stage * Cfg::kStage;
        const uint32_t b_addr = a_addr + Cfg::kStageA;
        // the stage is reusable once these MMAs have read it
        mma_stage<2, 2>(d_tmem, smem_desc_sw128(a_addr), smem_desc_sw128(b_addr), idesc, kb != 0 ? 1u : 0u, empty_bar(stage));
        stage = next;
        phase = next_phase;
      }
      if (!ok) break;
      tcgen05_commit_elect(acc_full_bar(acc));   // accumulator complete
      acc_phase[acc] ^= 1u;
      acc ^= 1;
    }
    if (!ok && lane == 0) record_timeout(P.status, timed_out);
  } else if (warp >= 2 && warp < kWeightWarp) {
    // ---------------------------------------------------------------- epilogue
    const int group = (warp - 2) >> 2;
    const int quad = warp & 3;               // TMEM lanes [32*quad, 32*quad+32) belong to this warp
    const int row = quad * 32 + lane;        // token row of this thread inside the tile
    const int epi_tid = threadIdx.x - 64;    // index among the epilogue threads
    const bool issuer = (epi_tid & 127) == 0;  // the thread of each group that owns its TMA stores
    const uint32_t buf0 = smem_base + S * Cfg::kStage + group * kBufPerGroup * kEpiStage;   // this group's staging buffers
    uint32_t my_piece = 0;                   // pieces staged by this group so far: selects the buffer
    uint16_t* s_bias = reinterpret_cast<uint16_t*>(smem + S * Cfg::kStage + kEpiBytes);  // [2][BN] bf16
    const uint32_t row_off = static_cast<uint32_t>(row) * 64u;
    const uint32_t row_xor = static_cast<uint32_t>((row >> 1) & 3);
    uint32_t acc_phase[2] = {0u, 0u};
    int acc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < total_tiles && ok; tile += gridDim.x) {
      const int m0 = (tile / n_tiles) * kBlockM, n0 = (tile % n_tiles) * BN;
      // Bias of this tile's columns, in the half of s_bias that belongs to this accumulator.  The
      // other group can lag by at most one tile (it has to reach the barrier below for this tile),
      // so the values it may still be reading are in the other half.
      for (int c = epi_tid; c < BN; c += kEpiThreads)
        s_bias[acc * BN + c] = (P.bias != nullptr && n0 + c < P.n_out) ? ld_global(P.bias + n0 + c) : static_cast<uint16_t>(0);
      tc_epilogue_sync_all();
      // all epilogue threads take the same decision, so nobody is left alone at a named barrier below
      if (!tc_epilogue_all_ok(mbar_wait(acc_full_bar(acc), acc_phase[acc], P.status))) { ok = false; break; }
      tcgen05_fence_after();
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(quad * 32) << 16) + static_cast<uint32_t>(acc * BN);
      const int pieces = (min(BN, P.n_out - n0) + kEpiCols - 1) / kEpiCols;
      bool released = false;
#pragma unroll 1
      for (int pc = group; pc < pieces; pc += kGroups) {
        const int c0 = pc * kEpiCols;
        const uint32_t buf = buf0 + (my_piece % kBufPerGroup) * kEpiStage;
        ++my_piece;
        EpiloguePiece piece;
        piece_load(taddr + c0, smem_u32(s_bias + acc * BN + c0), piece);
        if (issuer) tma_store_wait_read<kBufPerGroup - 1>();   // the store that last used this buffer has read it
        tc_group_sync(group);
        if (pc + kGroups >= pieces) {        // this warp's last read of the accumulator
          tcgen05_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty_bar(acc));
          released = true;
        }
        if (P.transposed) piece_store_transposed(piece, P.act, buf, row);
        else piece_store(piece, P.act, buf + row_off, row_xor);
        fence_async_smem();                  // make the staged piece visible to the TMA engine
        tc_group_sync(group);
        if (issuer) {
          // rows beyond `tokens` / columns beyond `n_out` are clipped by the tensor map
          if (P.transposed) tma_store_2d(&map_y, m0, n0 + c0, buf);
          else tma_store_2d(&map_y, n0 + c0, m0, buf);
        }
      }
      if (!released) {                       // a group without a piece in this tile still releases the accumulator
        tcgen05_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty_bar(acc));
      }
      acc_phase[acc] ^= 1u;
      acc ^= 1;
    }
    if (issuer) tma_store_wait_read<0>();   // shared memory must outlive the reads; the writes complete with the grid
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

// Self-test of the bail-out path: one CTA sets up what the tensor-core kernels set up (an mbarrier,
// tensor memory), then two of its threads wait through the same helpers on a barrier and on a
// counter that nothing ever signals.  Both waits run out at the configured limit, the roles record
// it, the CTA sits out the quiet period, frees its tensor memory and returns by itself.
__global__ void __launch_bounds__(128, 1) wait_selftest_kernel(int* status) {
  __shared__ __align__(8) uint64_t s_bar;
  __shared__ uint32_t s_tmem[2];
  volatile uint32_t* timed_out = s_tmem + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    *timed_out = 0u;
    status[4] = 0;
    mbar_init(smem_u32(&s_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(32u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tcgen05_fence_before();
  __syncthreads();
  tcgen05_fence_after();
  const uint32_t tmem_base = s_tmem[0];
  if (warp == 0 && lane == 0) {
    const unsigned long long t0 = global_timer_ns();
    if (!mbar_wait(smem_u32(&s_bar), 0u, status)) {
      record_timeout(status, timed_out);
      atomicAdd(status + 4, 1);
    }
    const unsigned long long dt = global_timer_ns() - t0;
    *reinterpret_cast<volatile unsigned long long*>(status + 6) = dt;
  } else if (warp == 2 && lane == 0) {
    if (!wait_counter(status + 1, 1, status)) {
      record_timeout(status, timed_out);
      atomicAdd(status + 4, 1);
    }
  }
  tcgen05_fence_before();
  __syncthreads();
  quiet_period(timed_out);
  if (warp == 1) {
    tcgen05_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(32u) : "memory");
  }
}

// Plan: put the packed tiles of one row-block back at their natural column positions, zero
// elsewhere.  grid = (row-blocks, row ranges); a CTA brings its rows' packed values (one contiguous run) and the
// index list into shared memory together, makes a column -> kept-position table, and each thread produces 8
// adjacent columns of a row (one 16-byte store).  Latency-bound: block pointers, then values and list, then stores.
// Looking the values up in global memory instead, eight dependent 2-byte loads per store, took 4.2 us for a
// 3072 x 768 matrix of 16-row blocks.
__device__ __forceinline__ unsigned grid_piece() { return blockIdx.z * gridDim.y + blockIdx.y; }   // see grid_of
constexpr int kPlanSmem = 48 * 1024;
__host__ __device__ inline int plan_rows_per_cta(int k_in) {
  const int r = kPlanSmem / (2 * k_in) - 1;     // rows of at most k_in values, and the table
  const int want = k_in >= 512 ? 4 : 2048 / k_in;   // four rows, or a piece of 8 columns for every thread
  return r > want ? want : r < 1 ? 1 : r;
}
__global__ void __launch_bounds__(256)
plan_expand_kernel(const int32_t* blk_ptr, const int32_t* idx,
                   const uint16_t* vals, int k_in, int block, uint16_t* Wx) {
  extern __shared__ __align__(16) int16_t s_pos[];   // [k_in] column -> position in the kept list, or -1 (k_in < 32768)
  const int b = blockIdx.x;
  const int rows_per = plan_rows_per_cta(k_in);
  const unsigned at = grid_piece() * static_cast<unsigned>(rows_per);
  if (at >= static_cast<unsigned>(block)) return;
  const int r_lo = static_cast<int>(at), n_rows = min(rows_per, block - r_lo);
  uint16_t* s_val = reinterpret_cast<uint16_t*>(s_pos + k_in);   // [n_rows][kc]
  const int chunks = k_in >> 3;
  for (int k = threadIdx.x; k < chunks; k += 256) reinterpret_cast<uint4*>(s_pos)[k] = make_uint4(~0u, ~0u, ~0u, ~0u);
  pdl_wait();
  pdl_launch_dependents();
  const int lo = ld_global(blk_ptr + b), kc = ld_global(blk_ptr + b + 1) - lo;
  const uint16_t* run = vals + static_cast<size_t>(block) * lo + static_cast<size_t>(r_lo) * kc;
  int col[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) col[u] = static_cast<int>(threadIdx.x) + u * 256 < kc ? ld_global(idx + lo + threadIdx.x + u * 256) : -1;
  const int n_val = n_rows * kc;
  for (int e0 = threadIdx.x; e0 < n_val; e0 += 8 * 256) {
    uint16_t v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u * 256 < n_val) v[u] = ld_global(run + e0 + u * 256);
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (e0 + u * 256 < n_val) s_val[e0 + u * 256] = v[u];
  }
  __syncthreads();                                   // the table is cleared
#pragma unroll
  for (int u = 0; u < 4; ++u)
    if (col[u] >= 0) s_pos[col[u]] = static_cast<int16_t>(threadIdx.x + u * 256);
  for (int j = threadIdx.x + 1024; j < kc; j += 256) s_pos[ld_global(idx + lo + j)] = static_cast<int16_t>(j);
  __syncthreads();
  for (int e = threadIdx.x; e < n_rows * chunks; e += 256) {
    const int r = e / chunks, q = e - r * chunks;
    const uint4 pos4 = *reinterpret_cast<const uint4*>(s_pos + (q << 3));
    const uint32_t pw[4] = {pos4.x, pos4.y, pos4.z, pos4.w};
    const uint16_t* row = s_val + r * kc;
    uint32_t out[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p0 = static_cast<int16_t>(pw[i] & 0xffffu), p1 = static_cast<int16_t>(pw[i] >> 16);
      const uint32_t v0 = p0 >= 0 ? row[p0] : 0u;
      const uint32_t v1 = p1 >= 0 ? row[p1] : 0u;
      out[i] = v0 | (v1 << 16);
    }
    *reinterpret_cast<uint4*>(Wx + (static_cast<size_t>(b) * block + r_lo + r) * k_in + (q << 3)) =
        make_uint4(out[0], out[1], out[2], out[3]);
  }
}

// Plan from the orientation-R packed form (vertical strips of h columns, kept ROWS per strip, tiles
// [kc][h]).  One CTA per strip and 256 rows: a table row -> kept position, then every row segment is
// written, its values or zeros, by vectors of VEC elements; nothing has to be zeroed beforehand.  Bound by
// latency on the paper's matrices (a 768 x 768 one is 192 CTAs); a launch per strip that scattered the
// kept segments after a clearing pass took 8.8 + 1.2 us there.
constexpr int kPlanRRows = 256;
template <int VEC>
__global__ void __launch_bounds__(256)
plan_expand_r_kernel(const int32_t* blk_ptr, const int32_t* row_idx,
                     const uint16_t* vals, int first_row, int n_out, int k_in, int h, uint16_t* Wx) {
  __shared__ int s_pos[kPlanRRows];
  const int a = blockIdx.x, r0 = first_row + blockIdx.y * kPlanRRows;
  const int n_rows = min(kPlanRRows, n_out - r0);
  s_pos[threadIdx.x] = -1;
  pdl_wait();
  pdl_launch_dependents();
  const int lo = blk_ptr[a], kc = blk_ptr[a + 1] - lo;
  __syncthreads();
  for (int j0 = threadIdx.x; j0 < kc; j0 += 4 * 256) {
    int r[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) r[u] = ld_global(row_idx + lo + min(j0 + u * 256, kc - 1)) - r0;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u * 256 < kc && r[u] >= 0 && r[u] < n_rows) s_pos[r[u]] = j0 + u * 256;
  }
  __syncthreads();
  const uint16_t* tile = vals + static_cast<size_t>(h) * lo;
  uint16_t* out = Wx + static_cast<size_t>(r0) * k_in + static_cast<size_t>(a) * h;
  const int per_row = h / VEC;
  // (the places come from this kernel's own loads, so these are behind the wait; unlike ordinary loads they may pass the
  // stores of the element before)
#pragma unroll 4
  for (int e = threadIdx.x; e < n_rows * per_row; e += 256) {
    const int r = e / per_row, c = (e - r * per_row) * VEC;
    const int p = s_pos[r];
    uint16_t* dst = out + static_cast<size_t>(r) * k_in + c;
    const uint16_t* src = tile + static_cast<size_t>(p) * h + c;
    if (VEC == 8) {
      *reinterpret_cast<uint4*>(dst) = p >= 0 ? __ldcg(reinterpret_cast<const uint4*>(src)) : make_uint4(0u, 0u, 0u, 0u);
    } else if (VEC == 4) {
      *reinterpret_cast<uint2*>(dst) = p >= 0 ? __ldcg(reinterpret_cast<const uint2*>(src)) : make_uint2(0u, 0u);
    } else {
      *dst = p >= 0 ? __ldcg(src) : static_cast<uint16_t>(0);
    }
  }
}

// The same for strips of a few columns, by scattering the kept segments over a cleared plan: a CTA of the kernel above has
// 256 short segments there and little else, and there are as many CTAs as strips.
__global__ void __launch_bounds__(256)
plan_scatter_r_kernel(const int32_t* __restrict__ blk_ptr, const int32_t* __restrict__ row_idx,
                      const uint16_t* __restrict__ vals, int k_in, int h, uint16_t* __restrict__ Wx) {
  const int a = blockIdx.x;                       // strip
  const int lo = blk_ptr[a], kc = blk_ptr[a + 1] - lo;
  const uint16_t* tile = vals + static_cast<size_t>(h) * lo;
  for (int e = threadIdx.x; e < kc * h; e += 256) {
    const int p = e / h, c = e - p * h;
    Wx[static_cast<size_t>(row_idx[lo + p]) * k_in + static_cast<size_t>(a) * h + c] = tile[e];
  }
}

// Transposed plan from the orientation-C packed form: PT[k, n] = (W * Mask)[n, k], for the product
// dX = dY (W * Mask).  A CTA makes the piece of 64 plan rows (columns k of W) x up to 64 plan columns (rows
// n of W: as many whole row-blocks as fit, or 64 rows of a taller one).  Per row-block a table column -> kept
// position; the values are read along k, where neighbours in the packed tile are neighbours in memory, turned
// in shared memory (33-word rows: no bank conflicts either way) and written along n, 128 contiguous bytes a
// plan row, zeros included.  Bound by a chain of four trips to memory (block pointers, index list, values,
// stores) and, with four CTAs per SM, by issue slots: all of a thread's values are asked for at once, the unit's
// values are fetched into L2 while the lists are read, and a warp takes adjacent rows so that the table and the
// block's place are looked up once per row-block.  (Looked up per element, with a division each, the values took 4 us
// even from L2.)  Between the products of a backward pass (768 features, 16-row blocks, cold operands) a 3072 x 768
// matrix takes 5.4 us, 7.3 scattered over a cleared plan; a 768 x 3072 one 5.4 and 33.
constexpr int kPlanTK = 64, kPlanTN = 64, kPlanTMaxBlocks = 32, kPlanTThreads = 512;
struct PlanTGeometry {
  int n_out, k_in, block;
  int blocks_per_unit;      // whole row-blocks of a unit, 1 where a block is cut into segments
  int segments;             // 64-row segments of a row-block taller than 64 rows, else 1
};
__global__ void __launch_bounds__(kPlanTThreads, 4)
plan_expand_t_kernel(const int32_t* blk_ptr, const int32_t* idx,
                     const uint16_t* vals, PlanTGeometry G, uint16_t* PT) {
  __shared__ int32_t s_col_pos[kPlanTMaxBlocks][kPlanTK];
  __shared__ uint16_t s_t[kPlanTK][kPlanTN + 2];
  __shared__ int32_t s_ptr[kPlanTMaxBlocks + 1];
  const unsigned piece = grid_piece(), pieces = gridDim.y * gridDim.z;
  if (piece * kPlanTK >= static_cast<unsigned>(G.k_in)) return;
  const int k0 = static_cast<int>(piece) * kPlanTK, nk = min(kPlanTK, G.k_in - k0);
  const int b0 = static_cast<int>(blockIdx.x) / G.segments * G.blocks_per_unit;
  const int seg = static_cast<int>(blockIdx.x) % G.segments;
  const int nb = min(G.blocks_per_unit, G.n_out / G.block - b0);
  const int rows_per_block = G.segments > 1 ? min(kPlanTN, G.block - seg * kPlanTN) : G.block;
  const int n0 = b0 * G.block + seg * kPlanTN;
  const int n_rows = nb * rows_per_block;
  for (int e = threadIdx.x; e < nb * kPlanTK; e += kPlanTThreads) s_col_pos[0][e] = -1;
  if (threadIdx.x == 0) prefetch_line(blk_ptr + b0);
  pdl_wait();
  pdl_launch_dependents();
  if (static_cast<int>(threadIdx.x) <= nb) s_ptr[threadIdx.x] = ld_global(blk_ptr + b0 + threadIdx.x);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  {
    // the unit's values are one run too: its CTAs fetch a share of it each into L2 while the lists are read
    const int lo = s_ptr[0], kept = s_ptr[nb] - lo;
    const char* run = reinterpret_cast<const char*>(vals + static_cast<size_t>(G.block) * lo + static_cast<size_t>(seg) * kPlanTN * kept);
    const long long bytes = 2LL * rows_per_block * kept, step = 128LL * kPlanTThreads * pieces;
    for (long long at = 128LL * (static_cast<long long>(threadIdx.x) * pieces + piece); at < bytes; at += step) prefetch_line(run + at);
  }
  // A warp lists a row-block's columns of the tile.  A longer list is narrowed down by 32 samples first: one trip to
  // memory more, but every CTA reading its blocks' whole lists took as many instructions as moving the values (a backward
  // pass of 944 features, 8-row blocks, 4508 tokens: 242 -> 236 us).
  for (int q = warp; q < nb; q += kPlanTThreads / 32) {
    const int lo = s_ptr[q], kc = s_ptr[q + 1] - lo;
    int first = 0, last = kc;                                  // where columns of the tile can stand
    if (kc > 256) {
      const int col = ld_global(idx + lo + static_cast<int>(static_cast<long long>(kc) * lane >> 5));
      const int below = __popc(__ballot_sync(0xffffffffu, col < k0)), upto = __popc(__ballot_sync(0xffffffffu, col < k0 + nk));
      if (below > 0) first = static_cast<int>(static_cast<long long>(kc) * (below - 1) >> 5);
      if (upto < 32) last = static_cast<int>(static_cast<long long>(kc) * upto >> 5);
    }
    for (int j0 = first + lane; j0 < last; j0 += 8 * 32) {
      int k[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) k[u] = j0 + u * 32 < last ? ld_global(idx + lo + j0 + u * 32) - k0 : -1;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (static_cast<unsigned>(k[u]) < static_cast<unsigned>(nk)) s_col_pos[q][k[u]] = j0 + u * 32;
    }
  }
  __syncthreads();
  // a warp takes adjacent rows, a lane two columns: their places in the packed tile change only with the row-block
  constexpr int kRows = kPlanTN / (kPlanTThreads / 32);
  const int n_first = warp * kRows;
  int q = n_first / rows_per_block, r = n_first - q * rows_per_block, kc = 0, p0 = -1, p1 = -1;
  const uint16_t* row = vals;
  auto enter = [&]() {
    if (q >= nb) return;
    const int lo = s_ptr[q];
    kc = s_ptr[q + 1] - lo;
    row = vals + static_cast<size_t>(G.block) * lo + static_cast<size_t>(r + seg * kPlanTN) * kc;
    p0 = s_col_pos[q][lane];
    p1 = s_col_pos[q][lane + 32];
  };
  enter();
  uint32_t v[kRows][2];
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    v[i][0] = v[i][1] = 0u;
    if (n_first + i >= n_rows) continue;
    if (p0 >= 0) v[i][0] = ld_global(row + p0);
    if (p1 >= 0) v[i][1] = ld_global(row + p1);
    row += kc;
    if (++r == rows_per_block) { r = 0; ++q; enter(); }
  }
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    s_t[lane][n_first + i] = static_cast<uint16_t>(v[i][0]);
    s_t[lane + 32][n_first + i] = static_cast<uint16_t>(v[i][1]);
  }
  __syncthreads();
  uint16_t* out = PT + static_cast<size_t>(k0) * G.n_out + n0;
  if (n_rows % 8 == 0 && n0 % 8 == 0 && G.n_out % 8 == 0) {
    const int per_row = n_rows >> 3;
    for (int e = threadIdx.x; e < nk * per_row; e += kPlanTThreads) {
      const int k = e / per_row, c = (e - k * per_row) << 3;
      const uint32_t* w = reinterpret_cast<const uint32_t*>(&s_t[k][c]);
      *reinterpret_cast<uint4*>(out + static_cast<size_t>(k) * G.n_out + c) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  } else {
    for (int e = threadIdx.x; e < nk * n_rows; e += kPlanTThreads) {
      const int k = e / n_rows, c = e - k * n_rows;
      out[static_cast<size_t>(k) * G.n_out + c] = s_t[k][c];
    }
  }
}

// The same by scattering the kept columns over a cleared plan, one CTA per row-block: consecutive threads take consecutive
// rows of a kept column.
__global__ void __launch_bounds__(256)
plan_scatter_t_kernel(const int32_t* __restrict__ blk_ptr, const int32_t* __restrict__ idx,
                      const uint16_t* __restrict__ vals, int n_out, int block, uint16_t* __restrict__ PT) {
  const int b = blockIdx.x;
  const int lo = blk_ptr[b], kc = blk_ptr[b + 1] - lo;
  const uint16_t* tile = vals + static_cast<size_t>(block) * lo;
  for (int e = threadIdx.x; e < kc * block; e += 256) {
    const int j = e / block, r = e - j * block;
    PT[static_cast<size_t>(idx[lo + j]) * n_out + static_cast<size_t>(b) * block + r] = tile[static_cast<size_t>(r) * kc + j];
  }
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
// A grid of x by `pieces`, the pieces spread over y and z where y alone (65535) does not hold them.
// Which transposed layouts are scattered: rows whose number is no multiple of 8 would be stored one element at a time by
// the one-pass kernel (1126 x 1320, 2-row blocks 8.7 us against 4.6; 4668 x 3288, 12-row 59 against 50; not tall blocks,
// of which there are too few to scatter), and past a thousand row-blocks the scattering has its CTAs
// (7048 x 2160, 4-row 36 against 15).  Otherwise the one pass wins between the products of a backward step (3072 x 768,
// 16-row 5.4 against 7.3, 768 x 3072 5.4 against 33, 6360 x 432, 8-row 7.6 against 8.5).
bool transposed_by_scatter(int n_out, int block) {
  return (n_out % 8 != 0 && block < 16) || n_out / block > 1024;
}
dim3 grid_of(int x, long long pieces) {
  const long long z = (pieces + 65534) / 65535;
  return dim3(x, static_cast<unsigned>((pieces + z - 1) / z), static_cast<unsigned>(z));
}
}  // namespace
// Tile width, one CTA or a pair, for a product of whole tiles: the least estimated time.  A launch costs a fixed
// part (start-up, first operands, the last tile's epilogue), per wave of tiles the larger of its main loop and its
// epilogue (with GELU also a part of the smaller one: they contend for issue slots), and something per wave after the
// first.  A 64-deep stage takes longer the more SMs are drawing operands from L2 (two times per width, for a few CTAs
// and for all of them), and where rows of X and the plan are no multiple of 128 bytes; more so where they are no multiple
// of 32 either (every row then straddles sectors, the narrow tiles' most: 12891 x 3856 x 3080 with GELU by one CTA 256 wide 325
// us, by pairs 128, 192 and 256 wide 328, 279 and 260; over 120 such layers the choice is 0.2 % behind the best on average and 7 %
// at worst).  Fitted to launches of 8 to
// 32768 tokens (nanoseconds; one CTA 64 / 128 / 192 / 256 wide, pairs 128 / 192 / 256): over 64 layers of 256 to 1024
// features the choice is 0.4 % behind the best of the seven on average and 6 % at worst.  Best one-CTA kernel / best pair:
// 4096 tokens x 768 outputs x 3072 inputs 19.9 / 16.5 us, 2304 x 768 14.4 / 13.2, 3072 x 768 with GELU 20.7 / 19.8, 4096 x
// 1024 with GELU 30.9 / 26.2, 768 x 768 7.0 / 7.2; 1003 tokens x 3072 x 1024 8.0 / 8.1, 512 x 768 x 3072 10.6 / 10.9.
DenseChoice choose_dense(const TcDevice& dev, int tokens, int n_out, int k_in, int act, DenseKinds kinds) {
  constexpr int kKinds = 7, kFirstPair = 4;
  static const int width[kKinds] = {64, 128, 192, 256, 128, 192, 256};
  static const int fixed[kKinds] = {2830, 3200, 3750, 4400, 3600, 4070, 4560}, extra_wave[kKinds] = {500, 700, 300, 800, 540, 450, 240};
  static const int stage_few[kKinds] = {158, 168, 250, 320, 150, 200, 270}, stage_all[kKinds] = {176, 210, 335, 370, 190, 250, 330};
  static const int ragged_percent[2][kKinds] = {{114, 130, 103, 110, 111, 106, 106}, {165, 192, 170, 167, 173, 155, 135}};
  static const int epilogue[2][kKinds] = {{500, 950, 1500, 1750, 570, 610, 1170}, {900, 1600, 2600, 2950, 1570, 3160, 3660}};
  static const int gelu_tail[kKinds] = {150, 500, 450, 600, 660, 530, 900};
  const long long kb = (k_in + kBlockK - 1) / kBlockK;
  const bool gelu = act == BSP_ACT_GELU;
  DenseChoice best{128, false, -1};
  for (int c = kinds == DenseKinds::kPairs ? kFirstPair : 0; c < (kinds == DenseKinds::kOneCta ? kFirstPair : kKinds); ++c) {
    const bool pair = c >= kFirstPair;
    const int rows = pair ? 2 * kBlockM : kBlockM;
    const long long tiles = ((tokens + rows - 1) / rows) * static_cast<long long>((n_out + width[c] - 1) / width[c]);
    const long long seats = pair ? dev.sms / 2 : dev.sms;
    const long long waves = (tiles + seats - 1) / seats;
    const long long busy = tiles < seats ? tiles : seats;
    long long main_ns = kb * (stage_few[c] + (stage_all[c] - stage_few[c]) * busy / seats);
    if (k_in % 64) main_ns = main_ns * ragged_percent[k_in % 16 != 0][c] / 100;
    const long long epi_ns = epilogue[gelu][c];
    long long tile_ns = main_ns > epi_ns ? main_ns : epi_ns;
    if (gelu) {
      const long long less = main_ns > epi_ns ? epi_ns : main_ns;
      tile_ns += less * less / tile_ns / 8;
    }
    const long long ns = fixed[c] + waves * tile_ns + (waves - 1) * extra_wave[c] + (gelu ? gelu_tail[c] : 0);
    if (best.ns < 0 || ns < best.ns) best = DenseChoice{width[c], pair, ns};
  }
  return best;
}
namespace {

template <int BN>
int launch_tc(TcDevice* dev, const void* plan, const void* X, void* Y, const LinearParams& P, int ldx,
              int ldy, cudaStream_t s) {
  using Cfg = TileCfg<BN>;
  static_assert(Cfg::kStages >= 3, "pipeline too shallow");
  static_assert(BN % kEpiCols == 0, "tile width must be a multiple of the epilogue piece");
  CUtensorMap map_x, map_w, map_y;
  if (!make_map(&map_x, X, P.k_in, P.tokens, ldx, copy_rows(P.tokens))) return BSP_ERR_CUDA;
  if (!make_map(&map_w, plan, P.k_in, P.n_out, P.k_in, BN)) return BSP_ERR_CUDA;
  if (P.transposed) {     // Y is [n_out, tokens]: pieces of 32 output rows x 128 tokens
    if (!make_map(&map_y, Y, P.tokens, P.n_out, ldy, kEpiCols, kBlockM)) return BSP_ERR_CUDA;
  } else if (!make_map(&map_y, Y, P.n_out, P.tokens, ldy, kBlockM, kEpiCols)) {
    return BSP_ERR_CUDA;
  }
  static OncePerDevice once;
  BSP_TRY(allow_dynamic_smem(once, linear_tc_kernel<BN>, Cfg::kSmemBytes));
  const int m_tiles = (P.tokens + kBlockM - 1) / kBlockM;
  const int n_tiles = (P.n_out + BN - 1) / BN;
  const int tiles = m_tiles * n_tiles;
  const int grid = tiles < dev->sms ? tiles : dev->sms;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreadsTc);
  cfg.dynamicSmemBytes = Cfg::kSmemBytes;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // start while the previous kernel drains
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  BSP_CUDA_TRY(cudaLaunchKernelEx(&cfg, linear_tc_kernel<BN>, map_x, map_w, map_y, P));
  return BSP_OK;
}

bool tc_path_ok(const void* plan, int n_out, int k_in, const void* X, int ldx, const void* Y, int ldy) {
  return aligned_to(plan, 16) && aligned_to(X, 16) && aligned_to(Y, 16) && k_in % 8 == 0 && ldx % 8 == 0 &&
         ldy % 8 == 0 && n_out % 8 == 0 && k_in <= 12288;
}

}  // namespace

TcDevice* tc_device() {
  static TcDevice info[64];
  static std::mutex guard;             // first calls from several host threads must not race on the set-up
  std::lock_guard<std::mutex> lock(guard);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  TcDevice& d = info[dev];
  if (d.sms == 0) {
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return nullptr;
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_linear_status) != cudaSuccess) return nullptr;
    if (!query_split_ctas(d.split_ctas)) return nullptr;
    d.status = static_cast<int*>(p);
    d.sms = sms;
  }
  return &d;
}

}  // namespace bsp

extern "C" int bsp_linear_plan_bytes(int n_out, int k_in, int block, size_t* bytes) {
  if (n_out <= 0 || k_in <= 0 || block <= 0 || bytes == nullptr) return BSP_ERR_ARG;
  if (n_out % block) return BSP_ERR_SHAPE;
  *bytes = bsp::round_up(static_cast<size_t>(n_out) * k_in * 2, 256);
  return BSP_OK;
}

extern "C" int bsp_linear_plan(const int32_t* blk_ptr, const int32_t* idx, const void* vals, int n_out,
                               int k_in, int block, void* plan, size_t plan_bytes, void* stream) {
  using namespace bsp;
  if (blk_ptr == nullptr || idx == nullptr || vals == nullptr || plan == nullptr) return BSP_ERR_ARG;
  size_t need;
  int st = bsp_linear_plan_bytes(n_out, k_in, block, &need);
  if (st != BSP_OK) return st;
  if (!aligned_to(plan, 256)) return BSP_ERR_ARG;
  if (plan_bytes < need) return BSP_ERR_WORKSPACE;
  if (k_in > 12288) return BSP_ERR_UNSUPPORTED;
  if (k_in % 8) return BSP_ERR_UNSUPPORTED;
  const int rows_per = plan_rows_per_cta(k_in);
  const dim3 grid = grid_of(n_out / block, (static_cast<long long>(block) + rows_per - 1) / rows_per);
  BSP_CUDA_TRY(launch_pdl(plan_expand_kernel, grid, dim3(256), static_cast<size_t>(k_in) * 2 * (1 + rows_per),
                          static_cast<cudaStream_t>(stream), blk_ptr, idx, static_cast<const uint16_t*>(vals), k_in, block,
                          static_cast<uint16_t*>(plan)));
  return BSP_OK;
}

extern "C" int bsp_linear_plan_r(const int32_t* blk_ptr, const int32_t* row_idx, const void* vals, int n_out,
                                 int k_in, int block, void* plan, size_t plan_bytes, void* stream) {
  using namespace bsp;
  if (blk_ptr == nullptr || row_idx == nullptr || vals == nullptr || plan == nullptr) return BSP_ERR_ARG;
  if (n_out <= 0 || k_in <= 0 || block <= 0) return BSP_ERR_ARG;
  if (k_in % block) return BSP_ERR_SHAPE;
  if (!aligned_to(plan, 256)) return BSP_ERR_ARG;
  const size_t need = round_up(static_cast<size_t>(n_out) * k_in * 2, 256);
  if (plan_bytes < need) return BSP_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const long long pieces = (static_cast<long long>(n_out) + kPlanRRows - 1) / kPlanRRows;
  int sms = 0;
  BSP_TRY(sm_count(&sms));
  // Strips narrower than 8 columns in more CTAs than the GPU holds at once (eight per SM) are scattered, a clearing pass
  // more: 1216 x 6264 in single columns 15 us against 75, 1168 x 2152 in fours 5.0 against 6.8.  Not below that (536 x 1964
  // in fours 4.9 against 4.7) and not in eights (5328 x 1648 14.8 against 10.9).
  if (block < 8 && k_in / block * pieces > 8LL * sms) {
    BSP_CUDA_TRY(cudaMemsetAsync(plan, 0, static_cast<size_t>(n_out) * k_in * 2, s));
    plan_scatter_r_kernel<<<k_in / block, 256, 0, s>>>(blk_ptr, row_idx, static_cast<const uint16_t*>(vals), k_in, block,
                                                       static_cast<uint16_t*>(plan));
    BSP_LAUNCH_CHECK();
    return BSP_OK;
  }
  // widest vector: every segment starts at a multiple of `block` in rows of k_in elements (a multiple of it too)
  const int vec = block % 8 == 0 && aligned_to(vals, 16) ? 8 : block % 4 == 0 && aligned_to(vals, 8) ? 4 : 1;
  // (a launch takes 16.7 million rows; numbering the pieces over two grid dimensions cost the short launches 0.6 us)
  for (long long done = 0; done < pieces; done += 65535) {
    const dim3 grid(k_in / block, static_cast<unsigned>(pieces - done < 65535 ? pieces - done : 65535));
    BSP_CUDA_TRY(launch_pdl(vec == 8 ? plan_expand_r_kernel<8> : vec == 4 ? plan_expand_r_kernel<4> : plan_expand_r_kernel<1>,
                            grid, dim3(256), 0, s, blk_ptr, row_idx, static_cast<const uint16_t*>(vals),
                            static_cast<int>(done * kPlanRRows), n_out, k_in, block, static_cast<uint16_t*>(plan)));
  }
  return BSP_OK;
}

extern "C" int bsp_linear_plan_t(const int32_t* blk_ptr, const int32_t* idx, const void* vals, int n_out, int k_in,
                                 int block, void* plan_t, size_t plan_bytes, void* stream) {
  using namespace bsp;
  if (blk_ptr == nullptr || idx == nullptr || vals == nullptr || plan_t == nullptr) return BSP_ERR_ARG;
  size_t need;
  int st = bsp_linear_plan_bytes(n_out, k_in, block, &need);
  if (st != BSP_OK) return st;
  if (!aligned_to(plan_t, 256)) return BSP_ERR_ARG;
  if (plan_bytes < need) return BSP_ERR_WORKSPACE;
  if (transposed_by_scatter(n_out, block)) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    BSP_CUDA_TRY(cudaMemsetAsync(plan_t, 0, static_cast<size_t>(n_out) * k_in * 2, s));
    plan_scatter_t_kernel<<<n_out / block, 256, 0, s>>>(blk_ptr, idx, static_cast<const uint16_t*>(vals), n_out, block,
                                                        static_cast<uint16_t*>(plan_t));
    BSP_LAUNCH_CHECK();
    return BSP_OK;
  }
  PlanTGeometry G{n_out, k_in, block, 1, 1};
  if (block > kPlanTN) {
    G.segments = (block + kPlanTN - 1) / kPlanTN;
  } else {
    // whole row-blocks up to 64 rows, preferably a multiple of 8 rows (16-byte stores)
    G.blocks_per_unit = kPlanTN / block < kPlanTMaxBlocks ? kPlanTN / block : kPlanTMaxBlocks;
    for (int m = G.blocks_per_unit; m > 1; --m)
      if (m * block % 8 == 0) { G.blocks_per_unit = m; break; }
  }
  const int nb = n_out / block;
  const int units = (nb + G.blocks_per_unit - 1) / G.blocks_per_unit * G.segments;
  const dim3 grid = grid_of(units, (static_cast<long long>(k_in) + kPlanTK - 1) / kPlanTK);
  BSP_CUDA_TRY(launch_pdl(plan_expand_t_kernel, grid, dim3(kPlanTThreads), 0, static_cast<cudaStream_t>(stream), blk_ptr, idx,
                          static_cast<const uint16_t*>(vals), G, static_cast<uint16_t*>(plan_t)));
  return BSP_OK;
}

extern "C" int bsp_linear_planned_ex(const void* plan, int n_out, int k_in, int block, const void* X, int tokens,
                                     int ldx, const void* bias, int act, void* Y, int ldy, int algo, void* stream) {
  using namespace bsp;
  const int algo_flags = algo & ~0xff;
  algo &= 0xff;
  if (algo < BSP_LINEAR_AUTO || algo > BSP_LINEAR_CTA_PAIR || (algo_flags & ~(BSP_LINEAR_PLAN_STABLE | BSP_LINEAR_OUT_TRANSPOSED)))
    return BSP_ERR_ARG;
  const bool transposed = (algo_flags & BSP_LINEAR_OUT_TRANSPOSED) != 0;
  if (transposed && algo == BSP_LINEAR_CTA_PAIR) return BSP_ERR_UNSUPPORTED;     // only the one-CTA kernel writes transposed
  // (a transposed output is [n_out, tokens]: its leading dimension spans the tokens)
  int st = check_linear_args(plan, plan, plan, n_out, k_in, block, X, tokens, ldx, act, Y, transposed ? n_out : ldy);
  if (st != BSP_OK) return st;
  if (transposed && ldy < tokens) return BSP_ERR_SHAPE;
  if (!tc_path_ok(plan, n_out, k_in, X, ldx, Y, ldy)) return BSP_ERR_UNSUPPORTED;
  if (tokens == 0) return BSP_OK;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const DenseKinds kinds = algo == BSP_LINEAR_CTA_PAIR ? DenseKinds::kPairs
                           : algo == BSP_LINEAR_AUTO && !transposed ? DenseKinds::kAll : DenseKinds::kOneCta;
  const DenseChoice choice = choose_dense(*dev, tokens, n_out, k_in, act, kinds);
  const bool plan_stable = (algo_flags & BSP_LINEAR_PLAN_STABLE) != 0;
  if (algo == BSP_LINEAR_AUTO) {
    // few output tiles: a cluster of CTAs per tile, each with a part of the contraction
    int bn_split = 0;
    const int c = choose_linear_split(*dev, tokens, n_out, k_in, choice.ns, &bn_split);
    if (c >= 0)
      return launch_linear_split(dev, bn_split, 2 << c, plan, X, Y, tokens, n_out, k_in, act, bias, ldx, ldy,
                                 plan_stable, transposed, s);
  }
  if (choice.pair) return launch_tc_pair(dev, choice.bn, plan, X, Y, tokens, n_out, k_in, act, bias, ldx, ldy, plan_stable, s);
  LinearParams P{tokens, n_out, k_in, act, plan_stable ? 1 : 0, copy_rows(tokens) * kBlockK * 2,
                 transposed ? 1 : 0,
                 static_cast<const uint16_t*>(bias), dev->status};
  switch (choice.bn) {
    case 256: return launch_tc<256>(dev, plan, X, Y, P, ldx, ldy, s);
    case 192: return launch_tc<192>(dev, plan, X, Y, P, ldx, ldy, s);
    case 128: return launch_tc<128>(dev, plan, X, Y, P, ldx, ldy, s);
    default: return launch_tc<64>(dev, plan, X, Y, P, ldx, ldy, s);
  }
}

extern "C" int bsp_linear_planned(const void* plan, int n_out, int k_in, int block, const void* X, int tokens,
                                  int ldx, const void* bias, int act, void* Y, int ldy, void* stream) {
  return bsp_linear_planned_ex(plan, n_out, k_in, block, X, tokens, ldx, bias, act, Y, ldy, BSP_LINEAR_AUTO, stream);
}

extern "C" int bsp_linear(const int32_t* blk_ptr, const int32_t* idx, const void* vals, int n_out, int k_in,
                          int block, const void* X, int tokens, int ldx, const void* bias, int act, void* Y,
                          int ldy, void* ws, size_t ws_bytes, void* stream) {
  using namespace bsp;
  int st = check_linear_args(blk_ptr, idx, vals, n_out, k_in, block, X, tokens, ldx, act, Y, ldy);
  if (st != BSP_OK) return st;
  if (ws == nullptr || !aligned_to(ws, 256) || !tc_path_ok(ws, n_out, k_in, X, ldx, Y, ldy))
    return bsp_linear_cuda_core(blk_ptr, idx, vals, n_out, k_in, block, X, tokens, ldx, bias, act, Y, ldy, stream);
  st = bsp_linear_plan(blk_ptr, idx, vals, n_out, k_in, block, ws, ws_bytes, stream);
  if (st != BSP_OK) return st;
  return bsp_linear_planned(ws, n_out, k_in, block, X, tokens, ldx, bias, act, Y, ldy, stream);
}

extern "C" int bsp_set_wait_limit_ms(int ms) {
  using namespace bsp;
  if (ms < 1 || ms > 600000) return BSP_ERR_ARG;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  const unsigned long long ns = static_cast<unsigned long long>(ms) * 1000000ull;
  BSP_CUDA_TRY(cudaDeviceSynchronize());         // kernels in flight keep the limit they started with
  BSP_CUDA_TRY(cudaMemcpy(dev->status + 2, &ns, sizeof(ns), cudaMemcpyHostToDevice));
  return BSP_OK;
}

extern "C" int bsp_wait_selftest(int* expired, long long* waited_ns, void* stream) {
  using namespace bsp;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  wait_selftest_kernel<<<1, 128, 0, s>>>(dev->status);
  BSP_LAUNCH_CHECK();
  int report[4] = {0, 0, 0, 0};
  BSP_CUDA_TRY(cudaMemcpyAsync(report, dev->status + 4, sizeof(report), cudaMemcpyDeviceToHost, s));
  BSP_CUDA_TRY(cudaStreamSynchronize(s));
  if (expired) *expired = report[0];
  if (waited_ns) memcpy(waited_ns, &report[2], sizeof(long long));
  return BSP_OK;
}

extern "C" int bsp_linear_status(void* stream) {
  using namespace bsp;
  TcDevice* dev = tc_device();
  if (dev == nullptr) return BSP_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int flag = 0;
  BSP_CUDA_TRY(cudaMemcpyAsync(&flag, dev->status, sizeof(int), cudaMemcpyDeviceToHost, s));
  BSP_CUDA_TRY(cudaStreamSynchronize(s));
  if (flag != 0) {
    BSP_CUDA_TRY(cudaMemsetAsync(dev->status, 0, sizeof(int), s));
    return BSP_ERR_TIMEOUT;
  }
  return BSP_OK;
}
