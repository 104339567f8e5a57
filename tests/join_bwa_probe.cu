// A BWA-compatible call of several classes with the class launch of the given number
// failing.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <new>

extern int g_fail_at;

#include "xt_bwa.cu"

namespace xt {
xt_status ctx_fail(xt_ctx*, xt_status s, const char*) { return s; }
xt_status ctx_cuda_fail(xt_ctx*, cudaError_t, const char*) { return XT_ECUDA; }
xt_status ctx_alloc(xt_ctx*, void** p, size_t*, size_t want) {
  *p = ::operator new(want);
  return XT_OK;
}
xt_status ctx_codes(xt_ctx*, const uint8_t**, int64_t*, const uint8_t**, int64_t*, cudaStream_t) {
  return XT_OK;
}
}  // namespace xt

int main(int, char** argv) {
  g_fail_at = std::atoi(argv[1]);
  xt_ctx* ctx = new xt_ctx();
  ctx->num_sms = 152;
  ctx->branches = std::atoi(argv[2]);
  static int32_t host[kSegHostWords];
  ctx->seg_host = host;
  ctx->seg_ev = (cudaEvent_t)302;
  for (size_t b = 0; b < kMaxBranches; ++b) {
    ctx->aux[b] = (cudaStream_t)(100 + b);
    ctx->join_ev[b] = (cudaEvent_t)(200 + b);
  }
  ctx->fork_ev = (cudaEvent_t)300;
  static uint8_t bytes[16];
  static int64_t o64[4];
  static int32_t o32[4];
  static xt_result out[4];
  const xt_bwa_scoring sc = {1, -4, -1, 6, 1, 6, 1, 100, 100, 5};
  const xt_status s = xt_extend_batch_bwa(ctx, bytes, 16, o64, o32, bytes, 16, o64, o32, o32, 4, &sc, out,
                                          nullptr, (void*)1);
  std::printf("status %d\n", (int)s);
  return 0;
}
