// xt_band.cu -- the band engine: the whole band of a pair in registers.
//
// The band's 2w + 1 diagonals are spread over the P lanes of a group, K
// neighbouring diagonals ("slots") a lane, and the group walks down the rows.
// In these coordinates the diagonal neighbour (i-1, j-1) of a cell has its
// slot, the one above (i-1, j) the next slot and the one to the left (i, j-1)
// the one before, so a row needs no boundary row in memory, no strips and no
// masks at the band's edges; all that is read is the two sequences.
//
// Lane p is one row behind lane p - 1 (step t: row t - p).  Per step a lane
// hands E past its last slot to the next lane, which needs it for the same
// row one step later, and F above its first slot to the lane before it, which
// needs it for its last slot within the same step (the shuffle is issued
// after the first slot and consumed by the last).  The row maximum travels
// along the lanes with its row, so the last lane sees the rows in order and
// keeps the extension's state (best, z-drop, end-to-end score).
//
// Every register holds two pairs, one per 16-bit half (scores below 2^15 / 2^k
// for the anchoring multiplier 2^k > match).  Row maxima with their column:
// a slot's key is (H - base) * 32 + slot with H - base clamped at 0, base a
// lower bound of the row's maximum from the last row seen: a row's maximum
// falls by at most max(alpha, -mismatch, -n_score) a row (its cell goes on
// down, or diagonally at the band's left edge) and rises by at most match.
//
// Bounded by the integer ALU pipe: about 12 instructions (9 on that pipe) per
// slot of two pairs and 160 a row besides.  250k long reads (1,000-10,000
// bases, w = 500) 528 -> 320 ms a call against one lane per pair in 32 bits,
// whose boundary rows went through DRAM; 3,001 of them 21.0 -> 8.2 ms against
// 32-lane strips.  The slot's tag is added as the key's maximum is taken (one
// instruction with the tag as an immediate): a multiply-add needed the tag in
// a register and took 378 ms.  With few slots and one warp per scheduler a row's
// dependent instructions (330 with 8 slots) bound it, 0.57 us: 1,000 pairs of 100
// bases 85 us (so queries that short stay on the group engine).  A narrow band
// first: 5,000 pairs of 1,024 bases, w = 1,024, 4.90 -> 1.43 ms a call on 512
// diagonals.
#include <algorithm>

#include "xt_kernels.cuh"
#include "xt_lane.cuh"
#include "xt_near.cuh"

namespace xt {
namespace {

constexpr int kBandThreads = 128;
// CTAs per SM: 32 slots take up to 168 registers a thread, fewer slots less.
__host__ __device__ constexpr int band_blocks(int K) { return K <= 14 ? 4 : 3; }
constexpr int kKeyBits = 5;     // slots of a lane
constexpr int kBaseSteps = 8;   // steps between two bases

// Base of a pair that is done, whose rows go on without meaning: above every
// H, so that its keys stay 0 and cannot run over into the other pair's half.
constexpr int32_t kNoKey = 16383;

// Rows between the row a base was taken from and the last one it is used for.
__host__ __device__ constexpr int base_age(int P) { return P + kBaseSteps; }

// NEAR: the P * K slots hold diagonals |i - j| <= hw of a wider band (hw <
// sc.w); a pair is settled only where the bounds of xt_bounds.cuh prove its
// outputs, and the others are marked in near_tmp, at their place in the queue.
template <int P, int K, bool NEAR>
__global__ void __launch_bounds__(kBandThreads, band_blocks(K))
    k_band(const Batch* __restrict__ bd, Score sc, Work w, int cls, int j_lo, int j_hi,
           int head_id, int32_t match, uint32_t mcm, uint32_t kmul, int32_t fall,
           int sms, const int32_t hw) {
  static_assert(K % 2 == 0 && K <= 32 && P <= 32, "slot index fits the key");
  constexpr int kWords = (K + 7) / 8;          // window words a row's slots span
  constexpr int kWin = (K + 7 + 7) / 8;        // and over the eight rows of a reload
  constexpr int kGroups = 32 / P;              // per warp
  constexpr int kCheck = P < 8 ? 8 : P;        // steps between two looks at the end
  constexpr int kAge = base_age(P);
  // few slots: selects instead of branches and shared memory (with 32 slots the
  // code they add cost 3,001 long pairs 8.2 -> 9.8 ms)
  constexpr bool kFew = K <= 14;
  __shared__ Batch s_b;
  __shared__ uint32_t s_tbl[8];
  __shared__ uint32_t s_row[K][kBandThreads];  // a lane's row, to take a slot by its number
  if (threadIdx.x == 0) {
    s_b = *bd;
#pragma unroll
    for (int c = 0; c < 5; ++c) s_tbl[c] = sc.prof[c];
  }
  __syncthreads();
  const Batch& b = s_b;
  const int lane = threadIdx.x & 31;
  const int p = lane % P;
  const int32_t begin = w.seg_begin[cls * kNumJ + j_hi];
  const int32_t end = w.seg_end[cls * kNumJ + j_lo];
  // the grid is rounded up: the CTAs that hold no pair are the last ones
  constexpr int kPerCta = 2 * kBandThreads / P;
  const int ctas = min((int)gridDim.x, (end - begin + kPerCta - 1) / kPerCta);
  if ((int)blockIdx.x >= ctas) return;
  int32_t* head = w.heads + head_id;
  const int32_t alpha = sc.alpha, beta = sc.beta;
  const int32_t pad = P * K - (2 * hw + 1);    // dead slots before the band's first
  const int32_t u0 = p * K;                    // slot u of the group: column i - hw - pad + u
  const uint32_t na2 = pack16(-alpha, -alpha), nb2 = pack16(-beta, -beta);
  const uint32_t nn = (sc.nnnn & 0xFFu) | (kPadScore << 8);
  const uint32_t kill = (pad > 0 && (pad - 1) / K == p) ? 0u : 0xFFFFFFFFu;
  const int kill_s = pad > 0 ? (pad - 1) % K : -1;
  const unsigned full = 0xffffffffu;
  const int32_t mid = hw + pad;                // slot of the seed's diagonal
  const uint32_t mid2 = (uint32_t)mid * 0x00010001u, u02 = (uint32_t)u0 * 0x00010001u;
  // a row this far below the best may stop the extension; half + z_off2 is
  // negative from there on
  const int32_t zlim = sc.zdrop > 0 ? min(sc.zdrop, 32766) : 32766;
  const uint32_t z_off2 = (uint32_t)(32767 - zlim) * 0x00010001u;
  // The first pairs of every warp are set by its place: block b most likely
  // shares its SM with b + SMs, b + 2 SMs, and the queue is longest first, so
  // every other row of blocks takes its pairs in reverse (3,001 long pairs, one
  // wave of warps: 9.8 -> 8.2 ms against first come, first served).  Later
  // pairs come from the queue.
  const int row = blockIdx.x / sms, col = blockIdx.x - row * sms;
  const int cols = min(sms, ctas - row * sms);
  const int place = row * sms + (row & 1 ? cols - 1 - col : col);
  int32_t next = (place * (kBandThreads / 32) + (int)(threadIdx.x >> 5)) * (2 * kGroups);
  for (bool first = true;; first = false) {
    if (!first) {
      if (lane == 0)
        next = ctas * (kBandThreads / 32) * (2 * kGroups) +
               atomicAdd(head, 2 * kGroups);
      next = __shfl_sync(full, next, 0);
    }
    const int32_t base_idx = begin + next;
    if (base_idx >= end) break;
    int32_t kk[2], ql[2], tl[2], h0[2];
    ByteStream qs[2], ts[2];
    bool act[2];
    const int32_t qpos0 = u0 - p - mid;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int32_t idx = base_idx + 2 * (lane / P) + h;
      int32_t k = idx < end ? w.order[idx] : -1;
      if ((uint32_t)k >= (uint32_t)b.n) k = -1;  // a corrupt workspace: no pair
      kk[h] = k;
      ql[h] = k >= 0 ? b.q_len[k] : 1;
      tl[h] = k >= 0 ? b.t_len[k] : 1;
      h0[h] = k >= 0 ? b.h0[k] : 1;
      qs[h].init(b.q_seq, b.q_seq + b.q_bytes, b.q_seq + (k >= 0 ? b.q_off[k] : 0) + qpos0);
      ts[h].init(b.t_seq, b.t_seq + b.t_bytes, b.t_seq + (k >= 0 ? b.t_off[k] : 0) - p);
      act[h] = k >= 0;
    }
    uint32_t H[K], F[K];  // F: of the row to come (the last slot's comes from the next lane)
#pragma unroll
    for (int s = 0; s < K; ++s) H[s] = F[s] = 0;
    auto row_m1_2 = [&](int32_t c, const int32_t (&hh)[2]) -> uint32_t {
      int32_t v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        v[h] = c == -1 ? hh[h] : ((uint32_t)c < (uint32_t)min(ql[h], hw) ? max(0, hh[h] - alpha - beta * c) : 0);
      return pack16(v[0], v[1]);
    };
    // state of the extension, in the group's last lane, both pairs packed:
    // best and the slot of its cell, the largest offset of a raising row
    uint32_t best2 = pack16(h0[0], h0[1]), bu2 = mid2, off2 = 0;
    int32_t brow[2] = {-1, -1}, g[2] = {-1, -1}, grow[2] = {0, 0};
    int32_t live_row[2] = {-1, -1}, dead_row[2] = {-2, -2}, bound[2], row_end[2];
    // the row maximum so far and its slot, G2 the last column's cell, E past the lane
    uint32_t M2 = 0, U2 = 0, G2 = 0, Eout = 0, nbase2 = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bound[h] = INT32_MAX;  // of every cell computed from the last look on
      row_end[h] = min(tl[h] - 1, ql[h] - 1 + hw);
    }
    const int32_t ends_from = __reduce_min_sync(full, min(ql[0], ql[1])) - 1 - hw;
    auto half = [](uint32_t v, int h) -> int32_t { return h ? hi16(v) : lo16(v); };
    // NEAR: whether the cells off the narrow band leave the results alone, row i
    // the last one seen (the rows since was_best was taken against that best,
    // those to come against the last); a failed pair is left
    int32_t was_best[2] = {h0[0], h0[1]};
    const int32_t at = base_idx + 2 * (lane / P);
    auto leave = [&](int h) {
      act[h] = false;
      w.near_tmp[at + h] = 1;
    };
    auto settled = [&](int h, int32_t i) -> bool {
      const int32_t top = half(best2, h), cap = min(tl[h] - 1, ql[h] - 1 + sc.w);
      return g[h] > 0 && near_row_ok(i, ql[h], h0[h], match, hw, was_best[h], sc) &&
             near_row_ok(cap, ql[h], h0[h], match, hw, top, sc) &&
             near_end_ok(g[h], ql[h], tl[h], h0[h], match, hw, sc);
    };
    auto finish = [&](int h, int32_t last) {
      act[h] = false;
      if (NEAR) w.near_tmp[at + h] = 0;
      const int32_t d = mid - half(bu2, h);  // diagonal of the best
      write_result(b, kk[h], half(best2, h), brow[h] - d + 1, brow[h] + 1, g[h],
                   g[h] > 0 ? grow[h] + 1 : 0, half(off2, h), XT_OK,
                   band_cells_upto(last, ql[h], sc.w));
    };
    uint32_t win[2][kWin], tw[2] = {0, 0};
    int32_t qpos = qpos0;
#pragma unroll
    for (int u = 0; u < kWin; ++u, qpos += 8)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        win[h][u] = nibbles(qs[h].next(b.q_seq, b.q_seq + b.q_bytes), ql[h] - qpos);
    bool more = true;
    for (int32_t t8 = 0; more; t8 += 8) {
#pragma unroll
      for (int h = 0; h < 2; ++h) tw[h] = nibbles(ts[h].next(b.t_seq, b.t_seq + b.t_bytes), 8);
      // the base of the next steps' keys, from the last row the last lane saw
      {
        int32_t v[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int32_t m = t8 - p > 0 ? half(M2, h) : h0[h];
          v[h] = act[h] ? -max(0, m - kAge * fall - 1) : -kNoKey;
        }
        nbase2 = pack16(v[0], v[1]);
        if (P > 1) nbase2 = __shfl_sync(full, nbase2, P - 1, P);
      }
      const uint32_t base2 = pack16(-lo16(nbase2), -hi16(nbase2));
#pragma unroll 1
      for (int r8 = 0; r8 < 8; ++r8) {
        const int32_t t = t8 + r8, i = t - p;
        const int sh = 4 * r8;
        // a lane that has not started, or starts now, is at row -1
        if (t < P && i <= 0) {
          // (opaque copies: the row is built here, not kept in registers throughout)
          int32_t hh[2] = {h0[0], h0[1]};
          asm volatile("" : "+r"(hh[0]), "+r"(hh[1]));
#pragma unroll
          for (int s = 0; s <= K; ++s) {
            const uint32_t v = row_m1_2(u0 + s - mid - 1, hh);  // 0 in the dead slots
            if (s < K) H[s] = v;
            if (s) F[s - 1] = u0 + s > pad ? __viaddmax_s16x2_relu(v, na2, 0u) : 0u;
          }
        }
        const uint32_t f_row0 = __viaddmax_s16x2_relu(H[0], na2, 0u);
        uint32_t x[2][kWords], tbl[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tbl[h] = s_tbl[(tw[h] >> sh) & 7u];
#pragma unroll
          for (int u = 0; u < kWords; ++u) x[h][u] = __funnelshift_r(win[h][u], win[h][u + 1], sh);
        }
        uint32_t E = 0, HA = na2, key = 0, s4[2] = {0, 0};
        if (P > 1) {
          E = __shfl_up_sync(full, Eout, 1, P);
          if (p == 0) E = 0;
        }
        uint32_t f_in = 0;  // F of the last slot
        auto slot = [&](int s) {
          if (s % 4 == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              s4[h] = prmt(tbl[h], nn, x[h][s / 8] >> (s % 8 ? 16 : 0));
          }
          constexpr uint32_t kSel[4] = {0xC480u, 0xD591u, 0xE6A2u, 0xF7B3u};
          const uint32_t S = prmt(s4[0], s4[1], kSel[s % 4]);
          const uint32_t D = H[s];
          const uint32_t M = __viaddmin_s16x2(D, S, D * mcm);
          if (s) E = __viaddmax_s16x2_relu(E, nb2, HA);
          const uint32_t f = s == K - 1 ? f_in : F[s];
          const uint32_t h2 = __vimax3_s16x2(M, E, f);
          HA = add16x2(h2, na2);
          const uint32_t t2 = __viaddmax_s16x2_relu(h2, nbase2, 0u);
          key = __viaddmax_s16x2(t2 * kmul, (uint32_t)s * 0x00010001u, key);
          if (s) F[s - 1] = __viaddmax_s16x2_relu(f, nb2, HA);
          H[s] = h2;
          return f;
        };
        // F above the first slot goes to the lane before
        uint32_t f_out = __viaddmax_s16x2_relu(slot(0), nb2, HA);
        if (P > 1) {
          if (t < P && i < 0) f_out = f_row0;
          f_in = __shfl_down_sync(full, f_out, 1, P);
          if (p == P - 1) f_in = 0;
        }
#pragma unroll
        for (int s = 1; s < K; ++s) slot(s);
        Eout = __viaddmax_s16x2_relu(E, nb2, HA);
        // F must not leave the band on its left
        if constexpr (kFew) {
#pragma unroll
          for (int n = 0; n < K - 1; n += 2)
            if (kill_s == n) F[n] &= kill;
        } else {
          switch (kill_s) {
#define XT_KILL(n) case n: if (n < K - 1) F[n < K ? n : 0] &= kill; break;
          XT_KILL(0) XT_KILL(2) XT_KILL(4) XT_KILL(6) XT_KILL(8) XT_KILL(10) XT_KILL(12)
          XT_KILL(14) XT_KILL(16) XT_KILL(18) XT_KILL(20) XT_KILL(22) XT_KILL(24) XT_KILL(26)
          XT_KILL(28) XT_KILL(30)
#undef XT_KILL
          default: break;
          }
        }
        // this lane's part of row i's maximum.  The column before the query is
        // not part of the row: where it holds the maximum, the slots after it
        // are looked through again
        // (a lane whose slots all lie at or under the base reports the base:
        // the row's maximum is above it)
        uint32_t m2 = ((key >> kKeyBits) & 0x07FF07FFu) + base2, mu2 = (key & 0x001F001Fu) + u02;
        if (t <= hw + P) {
          const int32_t before = mid - 1 - i - u0;  // slot of column -1
          if (before >= 0 && before < K &&
              ((key & 31u) == (uint32_t)before || ((key >> 16) & 31u) == (uint32_t)before)) {
            uint32_t a0 = 0, a1 = 0;
            if constexpr (kFew) {
#pragma unroll
              for (int s = 1; s < K; ++s) {
                if (s <= before) continue;
                a0 = max(a0, H[s] << 16 | (uint32_t)(u0 + s));
                a1 = max(a1, (H[s] & 0xFFFF0000u) | (uint32_t)(u0 + s));
              }
            } else {
#pragma unroll
              for (int s = 0; s < K; ++s) s_row[s][threadIdx.x] = H[s];
              for (int s = before + 1; s < K; ++s) {
                const uint32_t v = s_row[s][threadIdx.x];
                a0 = max(a0, v << 16 | (uint32_t)(u0 + s));
                a1 = max(a1, (v & 0xFFFF0000u) | (uint32_t)(u0 + s));
              }
            }
            m2 = prmt(a0, a1, 0x7632u);
            mu2 = prmt(a0, a1, 0x5410u);
          }
        }
        {
          uint32_t in = 0, inu = 0;
          if (P > 1) {
            in = __shfl_up_sync(full, M2, 1, P);
            inu = __shfl_up_sync(full, U2, 1, P);
            if (p == 0) in = 0;
          }
          asm("max.s16x2 %0, %1, %2;" : "=r"(M2) : "r"(in), "r"(m2));
          // halves where the lanes before hold more keep their slot (ties: the later slot)
          const uint32_t keep = prmt((M2 ^ m2) + 0x7FFF7FFFu, 0u, 0xBB99u);
          U2 = (inu & keep) | (mu2 & ~keep);
          if (t < P && i < 0) M2 = 0;
        }
        // the rows in order, in the last lane (the others' copies mean nothing)
        const uint32_t was2 = best2;
        asm("max.s16x2 %0, %0, %1;" : "+r"(best2) : "r"(M2));
        const uint32_t up = prmt((best2 ^ was2) + 0x7FFF7FFFu, 0u, 0xBB99u);  // raised halves
        bu2 = (bu2 & ~up) | (U2 & up);
        {
          uint32_t d2;
          asm("max.s16x2 %0, %1, %2;" : "=r"(d2) : "r"(U2 + 0x80008000u - mid2 ^ 0x80008000u),
              "r"(mid2 + 0x80008000u - U2 ^ 0x80008000u));
          asm("max.s16x2 %0, %0, %1;" : "+r"(off2) : "r"(d2 & up));
        }
        if (up & 1u) brow[0] = i;
        if (up >> 31) brow[1] = i;
        // a dead row (a half of 0), a row far below the best, or the last row
        const bool rare = i >= min(row_end[0], row_end[1]) ||
                          (((best2 - M2 + z_off2) | (M2 - 0x00010001u)) & 0x80008000u) != 0;
        // the last query column's cell travels with its row as well
        if (t >= ends_from) {
          uint32_t in = 0;
          if (P > 1) {
            in = __shfl_up_sync(full, G2, 1, P);
            if (p == 0) in = 0;
          }
          G2 = in;
          const int32_t sa = ql[0] - 1 - i + mid - u0, sb = ql[1] - 1 - i + mid - u0;
          const bool oa = i >= 0 && sa >= 0 && sa < K, ob = i >= 0 && sb >= 0 && sb < K;
          if (__any_sync(full, oa || ob)) {
#pragma unroll
            for (int s = 0; s < K; ++s) s_row[s][threadIdx.x] = H[s];
            if (oa) G2 = (G2 & 0xFFFF0000u) | (s_row[sa][threadIdx.x] & 0xFFFFu);
            if (ob) G2 = (G2 & 0xFFFFu) | (s_row[sb][threadIdx.x] & 0xFFFF0000u);
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int32_t ge = h ? hi16(G2) : lo16(G2);
            if (act[h] && ge > 0 && ge > g[h]) {
              g[h] = ge;
              grow[h] = i;
            }
          }
        }
        // a dead row, a z-drop or the last row
        if (rare && p == P - 1 && i >= 0) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!act[h]) continue;
            const int32_t m = half(M2, h), top = half(best2, h);
            bool stop = i >= row_end[h];
            if (NEAR) {
              // a dead row or one far below the best: only the whole band
              // tells whether the extension stops there
              if (m == 0 || (sc.zdrop > 0 && top - m > sc.zdrop)) {
                leave(h);
              } else if (stop) {
                int32_t last = -1;
                if (settled(h, i)) {
                  const NearEnd n = {top, mid - half(bu2, h), g[h], grow[h]};
                  last = near_last_row(n, ql[h], tl[h], h0[h], match, sc);
                }
                if (last >= 0) finish(h, last); else leave(h);
              }
              continue;
            }
            if (m == 0) {
              if (dead_row[h] != i - 1) live_row[h] = i - 1;
              dead_row[h] = i;
              stop |= col_m1(i, h0[h], sc) == 0;
            }
            if (sc.zdrop > 0 && top - m > sc.zdrop) {
              // a dead row's column is its last in-band column
              const int32_t um = m > 0 ? half(U2, h) : min(ql[h] - 1 - i + mid, 2 * hw + pad);
              const int32_t du = abs(um - half(bu2, h));
              stop |= (int64_t)(top - m) - (int64_t)du * beta > sc.zdrop;
            }
            if (stop) finish(h, m > 0 ? i : live_row[h]);
          }
        }
      }
      // Past the query's end: once no cell computed since the last look can
      // raise the best or the end-to-end score, the rows left matter only to
      // the last live row, which the bounds of xt_bounds.cuh give.  The look
      // bounds every cell computed after it, and is used one look later, when
      // the rows computed before it have reached the last lane.
      const int32_t i = t8 + 7 - p;
      if ((t8 + 8) % kCheck == 0 &&
          __any_sync(full, p == P - 1 && ((act[0] && i >= ql[0] - 1) || (act[1] && i >= ql[1] - 1)))) {
        int32_t top[2] = {0, 0};
#pragma unroll
        for (int s = 0; s < K; ++s) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int32_t left = ql[h] - 1 - i + mid - u0 - s;  // columns after this one
            const int32_t v = h ? hi16(H[s]) : lo16(H[s]);
            if (left >= 0 && v > 0) top[h] = max(top[h], v + match * left);
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (P > 1)
#pragma unroll
            for (int o = P / 2; o > 0; o >>= 1) top[h] = max(top[h], __shfl_xor_sync(full, top[h], o, P));
          if (p == P - 1 && act[h] && g[h] > 0 && bound[h] <= g[h]) {
            const NearEnd n = {half(best2, h), mid - half(bu2, h), g[h], grow[h]};
            const int32_t last = near_last_row(n, ql[h], tl[h], h0[h], match, sc);
            if (NEAR && (last < 0 || !settled(h, i)))
              leave(h);
            else if (last >= 0)
              finish(h, last);
          }
          bound[h] = top[h];
        }
      }
      // the rows of the last eight steps against the best before them
      if (NEAR && p == P - 1 && i >= 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // (1') bounds the loss on the rows up to the last hw + 1.  A pair that is a
          // quarter of that ahead of losing it evenly is left at once: long reads with
          // 8% errors fail some way down their thousands of rows anyway (1,000 of them,
          // w = 512, 28.5 -> 17.4 ms with the CTAs for what is left).  A few errors close
          // together are no reason: one pair left of a batch costs the group engine's
          // whole pass (1,000 of 3,800 bases with 2% errors 19.3 ms where one and a half
          // times the even rate from row 255 on was, 8.4 ms so)
          const int32_t rows = ql[h] - hw - 1, seen = i - 7;  // (was_best is of eight rows ago)
          const float lost = h0[h] + match * seen - was_best[h];
          const bool fast = i < rows && lost * rows > (alpha - beta + beta * (hw + 1)) * (seen + 0.25f * rows);
          if (act[h] && (fast || !near_row_ok(i, ql[h], h0[h], match, hw, was_best[h], sc))) leave(h);
          was_best[h] = half(best2, h);
        }
      }
      more = __any_sync(full, p == P - 1 && (act[0] || act[1]));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int u = 0; u + 1 < kWin; ++u) win[h][u] = win[h][u + 1];
        win[h][kWin - 1] = nibbles(qs[h].next(b.q_seq, b.q_seq + b.q_bytes), ql[h] - qpos);
      }
      qpos += 8;
    }
  }
}

// The pairs the NEAR launch of bucket j left move to the front of the bucket's run in
// the queue, in their order (longest first: lanes of a warp then hold pairs of like
// length; in the order they were left 55k streamed pairs, w = 600, took 9.0 ms a call, 7.1
// so).  One block, each thread kPackPer neighbouring places a round; a round's places
// are read before they are written, and none is written before its own round.
// lanes_from > 0: so many pairs or more become the segment of those left to lanes.
constexpr int kPackThreads = 1024;
constexpr int kPackPer = 8;

__global__ void __launch_bounds__(kPackThreads) k_band_pack(Work w, int cls, int j,
                                                            int32_t lanes_from) {
  __shared__ int32_t s_warp[kPackThreads / 32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int32_t begin = w.seg_begin[cls * kNumJ + j], end = w.seg_end[cls * kNumJ + j];
  int32_t out = begin;
  for (int32_t round = begin; round < end; round += kPackThreads * kPackPer) {
    const int32_t first = round + threadIdx.x * kPackPer;
    int32_t pair[kPackPer], mine = 0;
#pragma unroll
    for (int u = 0; u < kPackPer; ++u) {
      const bool left = first + u < end && w.near_tmp[first + u] != 0;
      pair[u] = left ? w.order[first + u] : -1;
      mine += left;
    }
    int32_t inc = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int32_t v = __shfl_up_sync(0xffffffffu, inc, d);
      if (lane >= d) inc += v;
    }
    if (lane == 31) s_warp[wid] = inc;
    __syncthreads();
    int32_t at = out + inc - mine, total = 0;
    for (int u = 0; u < kPackThreads / 32; ++u) {
      if (u < wid) at += s_warp[u];
      total += s_warp[u];
    }
#pragma unroll
    for (int u = 0; u < kPackPer; ++u)
      if (pair[u] >= 0) w.order[at++] = pair[u];
    out += total;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const bool lanes = lanes_from > 0 && out - begin >= lanes_from;
    w.seg_end[cls * kNumJ + j] = lanes ? begin : out;
    if (lanes_from > 0) {
      w.seg_begin[kLanesLeftSeg * kNumJ + j] = begin;
      w.seg_end[kLanesLeftSeg * kNumJ + j] = lanes ? out : begin;
    }
  }
}

// The lane counts and slots compiled: per lane count, fewest slots first.
struct BandShape {
  int P, K;
};
constexpr BandShape kBandShapes[] = {{2, 32},  {4, 32},  {8, 26},  {8, 32},  {16, 14}, {16, 26},
                                     {16, 32}, {32, 8},  {32, 14}, {32, 26}, {32, 32}};

int32_t band_fall(const Score& sc) {
  // the most a row's maximum can fall below the one before it
  int32_t d = sc.alpha;
  d = std::max(d, -(int32_t)(int8_t)((sc.prof[0] >> 8) & 0xFF));
  d = std::max(d, -(int32_t)(int8_t)(sc.nnnn & 0xFF));
  return d;
}

// Whether the engine takes the scoring with P lanes a pair.
bool band_scoring(const Score& sc, int32_t match, int P) {
  if (sc.w < 8 || sc.alpha < 1 || sc.alpha > 127) return false;
  const int32_t fall = band_fall(sc);
  // H - base of a row's maximum, and of the column before the query, within the key
  return base_age(P) * (fall + match) + fall + match + 2 <= (32767 >> kKeyBits) - 1;
}

// A launch with fewer warps than this leaves schedulers idle (four on each of 152 SMs;
// one figure for all parts, so that a pair's engine does not depend on the part).
constexpr int64_t kBandWarps = 608;

}  // namespace

// Lanes per pair: the fewest that hold the band, whose rows cost the least in
// all; while the launch's warps then leave schedulers idle, more lanes with
// fewer slots each, which shorten the time of a row (a row costs a warp about
// 20 cycles a slot and 300 besides).
bool band_shape(const Score& sc, int32_t match, int32_t pairs, int* P, int* K) {
  *P = 0;
  for (const BandShape& s : kBandShapes) {
    if (s.P * s.K < 2 * (int64_t)sc.w + 1 || s.P == *P || !band_scoring(sc, match, s.P)) continue;
    if (*P && (int64_t)pairs * s.P > kBandWarps * 64) break;
    *P = s.P;
    *K = s.K;
  }
  return *P > 0;
}

// The narrow band tried first on the pairs of bucket j where the whole band is
// too wide for the engine: diagonals up to an eighth to a quarter of the
// query's length to each side.  A read with 2% substitutions loses about a tenth
// of its length against a perfect match, and a pair is settled while it loses
// less than the half width.
bool band_near_shape(const Score& sc, int32_t match, int j, int* P, int* K, int* hw) {
  if (j < kBandNearJMin) return false;
  *P = j <= 10 ? 8 : (j == 11 ? 16 : 32);
  *K = 32;
  *hw = *P * *K / 2 - 1;
  return *hw < sc.w && band_scoring(sc, match, *P);
}

int band_grid(int P, int K, int32_t pairs, int num_sms) {
  const int64_t per_cta = 2 * (int64_t)kBandThreads / P;
  const int64_t want = ((int64_t)pairs + per_cta - 1) / per_cta;
  return rounded_grid(want, num_sms, band_blocks(K));
}

cudaError_t launch_band(const Batch* bd, const Score& sc, int32_t match, const Work& w,
                        const Launch& L, int head_id, int num_sms, cudaStream_t stream) {
  int mshift = 0;
  while ((1 << mshift) < match + 1) ++mshift;
  const int32_t fall = band_fall(sc);
#define XT_BL(PP, KK, NN)                                                                      \
  if (L.P == PP && L.R == KK && (L.near_hw > 0) == NN) {                                       \
    k_band<PP, KK, NN><<<L.grid, kBandThreads, 0, stream>>>(                                   \
        bd, sc, w, L.cls, L.j_lo, L.j_hi, head_id, match, 1u << mshift, 1u << kKeyBits, fall,  \
        num_sms, NN ? L.near_hw : sc.w);                                                       \
    if (NN) k_band_pack<<<1, kPackThreads, 0, stream>>>(w, L.cls, L.j_lo, L.lanes_from);                           \
    return cudaGetLastError();                                                                 \
  }
  XT_BL(2, 32, false) XT_BL(4, 32, false) XT_BL(8, 26, false) XT_BL(8, 32, false)
  XT_BL(16, 14, false) XT_BL(16, 26, false) XT_BL(16, 32, false) XT_BL(32, 8, false)
  XT_BL(32, 14, false) XT_BL(32, 26, false) XT_BL(32, 32, false)
  XT_BL(8, 32, true) XT_BL(16, 32, true) XT_BL(32, 32, true)
#undef XT_BL
  return cudaErrorInvalidValue;
}

}  // namespace xt
