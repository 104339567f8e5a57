// The extension launches of one call with the launch of the given number failing.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>

extern int g_fail_at;
cudaError_t fake_launch(cudaStream_t st);

#include "xt_api.cu"

namespace xt {
cudaError_t launch_lane(const Batch*, const Score&, const Work&, const Launch&, int, void*,
                        cudaStream_t st) {
  return fake_launch(st);
}
cudaError_t launch_queue(const Batch*, const Score&, const Work&, const Launch&, int, int2*,
                         cudaStream_t st) {
  return fake_launch(st);
}
cudaError_t launch_band(const Batch*, const Score&, int32_t, const Work&, const Launch&, int, int,
                        cudaStream_t st) {
  return fake_launch(st);
}
cudaError_t launch_near(const Batch*, const Score&, int32_t, int, const Work&, int, cudaStream_t st) {
  return fake_launch(st);
}
}  // namespace xt

int main(int, char** argv) {
  g_fail_at = std::atoi(argv[1]);
  xt_ctx* ctx = new xt_ctx();
  ctx->branches = std::atoi(argv[2]);
  for (size_t b = 0; b < kMaxBranches; ++b) {
    ctx->aux[b] = (cudaStream_t)(100 + b);
    ctx->join_ev[b] = (cudaEvent_t)(200 + b);
  }
  ctx->fork_ev = (cudaEvent_t)300;
  ctx->near_ev = (cudaEvent_t)301;
  Plan pl;
  pl.near_pairs = 10000;
  pl.near_grid = 10;
  for (pl.n_launch = 0; pl.n_launch < 5; ++pl.n_launch) {
    Launch& L = pl.launch[pl.n_launch];
    L.lane = pl.n_launch % 2;
    L.band = pl.n_launch == 4;
    L.cls = pl.n_launch < 2 ? CLS_NARROW : CLS_NEAR;
    L.grid = 1;
  }
  Score sc = {};
  Work w = {};
  int dp = 0;
  const cudaError_t e = enqueue_dp(ctx, false, pl, 0, sc, w, nullptr, 1024, (cudaStream_t)1, &dp);
  std::printf("status %d\n", (int)e);
  return 0;
}
