// bsp_linear_route / bsp_linear_run / bsp_linear_tune: one front door for the pruned linear layer.
//
// The library has two ways to run Y = act(X (W * Mask)^T + b): the zero-expanded route
// (bsp_linear_planned_ex: dense tcgen05 tiles over W with zeros in the pruned places; executes
// 2 T N K flops whatever the compression) and the gathering route (bsp_linear_gathered_ex: only the
// kept columns are fetched and multiplied; its time per 64 kept columns does not depend on the
// block height).  Which is faster depends on the block height, the compression, the shape and the
// activation.  The caller describes what it has (which layouts of the weights, which layouts of the
// activations, which layout it wants out) and either names a route, lets a cost estimate fitted to
// measurements choose, or has both timed on the spot.
#include <math.h>

#include "bsp_tc.cuh"

namespace bsp {
namespace {

bool gather_block(int block) { return block == 16 || block == 32 || block == 64 || block == 128; }

bool can_zero_expanded(const bsp_linear_call& c) { return c.plan != nullptr && c.X != nullptr; }
bool can_gathered(const bsp_linear_call& c) { return c.gplan != nullptr && c.XT != nullptr && gather_block(c.block); }

int check_call(const bsp_linear_call* c) {
  if (c == nullptr) return BSP_ERR_ARG;
  if (c->n_out <= 0 || c->k_in <= 0 || c->block <= 0 || c->tokens < 0) return BSP_ERR_ARG;
  if (c->n_out % c->block) return BSP_ERR_SHAPE;
  if ((c->Y == nullptr) == (c->YT == nullptr)) return BSP_ERR_ARG;          // exactly one output layout
  if (c->X == nullptr && c->XT == nullptr) return BSP_ERR_ARG;
  if (c->plan == nullptr && c->gplan == nullptr) return BSP_ERR_ARG;
  return BSP_OK;
}

// Estimated nanoseconds of the two routes.  Zero-expanded: what the kernel choice of bsp_linear_planned_ex expects, and a
// microsecond that it leaves out for all of its kernels alike.  Gathering: a launch, and per row-block that the busiest CTA
// works through 87 ns for every 16 kept columns (the TMA row gather is the bound, whatever the block height; a stage that a
// row-block leaves with one group of 16 takes the time of two) and, per 32 rows of the block, its epilogue: 213 ns, with GELU
// 400 by two epilogue groups, by four 300, or 260 where these write transposed pieces.  Fitted to 562 layers by both routes,
// 64 to 32768 tokens, 224 to 4096 features, blocks of 16 to 128 rows at 2 to 10 times compression: the gathering estimate is
// off by 6 % (rms), the choice costs 0.2 % over the better route on average and 11 % at worst (8192 tokens, 768 x 768 in 64-row
// blocks at 5x 11.3 us zero-expanded, 12.5 gathered).  With 301 ns for every GELU and 3 % in favour of the zero-expanded route
// it was 0.5 % and 27 %: 368 tokens, 800 x 3000 in 32-row blocks at 4.9x 9.5 us and 7.5; 32768 tokens, 3072 x 1024 in 128-row
// blocks at 3x 127 and 116.
void estimate_ns(const bsp_linear_call& c, const TcDevice& dev, double* zero_expanded, double* gathered) {
  long long ns = choose_dense(dev, c.tokens, c.n_out, c.k_in, c.act, c.YT == nullptr ? DenseKinds::kAll : DenseKinds::kOneCta).ns;
  int bn;
  choose_linear_split(dev, c.tokens, c.n_out, c.k_in, ns, &bn, &ns);
  *zero_expanded = static_cast<double>(ns) + 1000.0;
  const long long blocks = c.n_out / c.block;
  const GatherUnits u = gather_units(c.tokens, static_cast<int>(blocks), dev.sms);
  const double kept_per_block = c.kept_weights >= 0 ? static_cast<double>(c.kept_weights) / c.block / blocks : c.k_in;
  double groups = kept_per_block > 16.0 ? ceil(kept_per_block / 16.0) : 1.0;
  if (fmod(groups, 4.0) == 1.0) groups += 1.0;
  double epilogue = 213.0;
  if (c.act == BSP_ACT_GELU) {
    const bool four = gather_four_groups(c.block, c.act, u.m_tiles * blocks, dev.sms);
    epilogue = !four ? 400.0 : c.YT != nullptr ? 260.0 : 300.0;
  }
  const double block_ns = 87.0 * groups + epilogue * (c.block > 32 ? c.block / 32 : 1);
  const long long units = static_cast<long long>(u.m_tiles) * u.n_chunks;
  *gathered = 4550.0 + static_cast<double>((units + dev.sms - 1) / dev.sms * u.rb_per_chunk) * block_ns;
}

int choose(const bsp_linear_call& c) {
  const bool z = can_zero_expanded(c), g = can_gathered(c);
  if (z && !g) return BSP_ROUTE_ZERO_EXPANDED;
  if (g && !z) return BSP_ROUTE_GATHERED;
  if (!z && !g) return 0;
  if (c.tokens == 0) return BSP_ROUTE_ZERO_EXPANDED;
  TcDevice host;                                             // without a device: a B200
  host.sms = 148;
  host.split_ctas[0] = 148;
  host.split_ctas[1] = 144;
  host.split_ctas[2] = 128;
  const TcDevice* dev = tc_device();
  if (dev == nullptr) dev = &host;
  double tz, tg;
  estimate_ns(c, *dev, &tz, &tg);
  return tg < tz ? BSP_ROUTE_GATHERED : BSP_ROUTE_ZERO_EXPANDED;
}

int run_route(const bsp_linear_call& c, int route, cudaStream_t s) {
  void* out = c.Y ? c.Y : c.YT;
  const int ldo = c.Y ? c.ldy : c.ldyt;
  if (route == BSP_ROUTE_ZERO_EXPANDED) {
    if (!can_zero_expanded(c)) return BSP_ERR_ARG;
    const int algo = BSP_LINEAR_AUTO | (c.plan_stable ? BSP_LINEAR_PLAN_STABLE : 0) | (c.YT ? BSP_LINEAR_OUT_TRANSPOSED : 0);
    return bsp_linear_planned_ex(c.plan, c.n_out, c.k_in, c.block, c.X, c.tokens, c.ldx, c.bias, c.act, out, ldo, algo, s);
  }
  if (route == BSP_ROUTE_GATHERED) {
    if (!can_gathered(c)) return BSP_ERR_ARG;
    return bsp_linear_gathered_ex(c.gplan, c.n_out, c.k_in, c.block, c.XT, c.tokens, c.ldxt, c.bias, c.act, out, ldo,
                                  c.YT ? 1 : 0, s);
  }
  return BSP_ERR_ARG;
}

}  // namespace
}  // namespace bsp

extern "C" int bsp_linear_route(const bsp_linear_call* call, int* route) {
  using namespace bsp;
  int st = check_call(call);
  if (st != BSP_OK) return st;
  if (route == nullptr) return BSP_ERR_ARG;
  *route = choose(*call);
  return *route == 0 ? BSP_ERR_ARG : BSP_OK;       // no route: the layouts given do not fit together
}

extern "C" int bsp_linear_run(const bsp_linear_call* call, int route, int* route_taken, void* stream) {
  using namespace bsp;
  int st = check_call(call);
  if (st != BSP_OK) return st;
  if (route < BSP_ROUTE_AUTO || route > BSP_ROUTE_GATHERED) return BSP_ERR_ARG;
  if (route == BSP_ROUTE_AUTO) route = choose(*call);
  if (route == 0) return BSP_ERR_ARG;
  if (route_taken) *route_taken = route;
  return run_route(*call, route, static_cast<cudaStream_t>(stream));
}

extern "C" int bsp_linear_tune(const bsp_linear_call* call, int reps, int* best_route, float* ms_zero_expanded,
                               float* ms_gathered, void* stream) {
  using namespace bsp;
  int st = check_call(call);
  if (st != BSP_OK) return st;
  if (best_route == nullptr || reps < 1 || reps > 1000) return BSP_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float ms[3] = {0.0f, -1.0f, -1.0f};
  cudaEvent_t a, b;
  BSP_CUDA_TRY(cudaEventCreate(&a));
  if (cudaEventCreate(&b) != cudaSuccess) { cudaEventDestroy(a); return BSP_ERR_CUDA; }
  for (int route = BSP_ROUTE_ZERO_EXPANDED; route <= BSP_ROUTE_GATHERED && st == BSP_OK; ++route) {
    if (route == BSP_ROUTE_ZERO_EXPANDED ? !can_zero_expanded(*call) : !can_gathered(*call)) continue;
    st = run_route(*call, route, s);                                 // one untimed launch first
    if (st != BSP_OK) break;
    if (cudaEventRecord(a, s) != cudaSuccess) { st = BSP_ERR_CUDA; break; }
    for (int i = 0; i < reps && st == BSP_OK; ++i) st = run_route(*call, route, s);
    if (st != BSP_OK) break;
    if (cudaEventRecord(b, s) != cudaSuccess || cudaEventSynchronize(b) != cudaSuccess ||
        cudaEventElapsedTime(&ms[route], a, b) != cudaSuccess) { st = BSP_ERR_CUDA; break; }
    ms[route] /= static_cast<float>(reps);
  }
  cudaEventDestroy(a);
  cudaEventDestroy(b);
  if (st != BSP_OK) return st;
  if (ms[1] < 0.0f && ms[2] < 0.0f) return BSP_ERR_ARG;
  *best_route = (ms[2] >= 0.0f && (ms[1] < 0.0f || ms[2] < ms[1])) ? BSP_ROUTE_GATHERED : BSP_ROUTE_ZERO_EXPANDED;
  if (ms_zero_expanded) *ms_zero_expanded = ms[1];
  if (ms_gathered) *ms_gathered = ms[2];
  return BSP_OK;
}
