// Runs the library's planner on pair counts without a GPU (tests/test_plan.py).
// Each case on standard input: a line "w match mismatch gap_open gap_extend zdrop
// n_score n hopeful budget near_ok tunings counts", then `tunings` lines "j batch_class P R"
// and `counts` lines "class j pairs"; one JSON line out per case.
#include "xt_api.cu"

#include <iostream>

int main() {
  xt_scoring s;
  int64_t n, hopeful, budget, near_ok, tunings, counts;
  while (std::cin >> s.w >> s.match >> s.mismatch >> s.gap_open >> s.gap_extend >> s.zdrop >>
         s.n_score >> n >> hopeful >> budget >> near_ok >> tunings >> counts) {
    xt_ctx* ctx = new xt_ctx();
    ctx->num_sms = 152;
    ctx->smem_optin = 227 * 1024;
    ctx->budget = (size_t)budget;
    ctx->match = s.match;
    if (tunings) {
      ctx->tuning.push_back(TuneEntry());
      ctx->tuning.back().w = s.w;
    }
    for (int k = 0; k < tunings; ++k) {
      int j, small, P, R;
      std::cin >> j >> small >> P >> R;
      BucketSched& b = small ? ctx->tuning.back().small[j] : ctx->tuning.back().b[j];
      b.P = P;
      b.R = R;
    }
    int32_t cnt[kNumClasses][kNumJ] = {};
    for (int k = 0; k < counts; ++k) {
      int c, j, v;
      std::cin >> c >> j >> v;
      cnt[c][j] = v;
    }
    const Score sc = make_score(&s);
    JFlags jf;
    bool lane_ok[kNumJ];
    batched_flags(ctx, sc, (int32_t)n, &jf, lane_ok);
    Plan pl;
    plan_counts(ctx, sc, cnt, (int32_t)hopeful, near_ok != 0, jf, lane_ok, &pl);
    const size_t pool = layout_pool(ctx, &pl);
    std::printf("{\"bad\": %d, \"near_pairs\": %d, \"near_grid\": %d, \"signature\": \"%016llx\", "
                "\"pool\": %zu, \"max_launches\": %d, \"launches\": [",
                (int)pl.bad, pl.near_pairs, pl.near_grid, (unsigned long long)plan_signature(pl), pool,
                kMaxLaunches);
    for (int i = 0; i < pl.n_launch; ++i) {
      const Launch& L = pl.launch[i];
      std::printf("%s{\"engine\": \"%s\", \"cls\": %d, \"cls2\": %d, \"j_lo\": %d, \"j_hi\": %d, \"P\": %d, "
                  "\"R\": %d, \"grid\": %d, \"near_hw\": %d, \"after_prev\": %d, \"global_ring\": %d, "
                  "\"lanes_from\": %d, \"lanes_left\": %d}",
                  i ? ", " : "", L.band ? "band" : (L.lane ? "lane" : "group"), L.cls, L.cls2, L.j_lo,
                  L.j_hi, L.P, L.R, L.grid, L.near_hw, (int)L.after_prev, (int)L.global_ring, L.lanes_from, (int)L.lanes_left);
    }
    std::printf("], \"flags\": [");
    for (int j = 0; j < kNumJ; ++j) std::printf("%s%d", j ? ", " : "", jf.f[j]);
    std::printf("]}\n");
    delete ctx;
  }
  return 0;
}
