// xt_near.cu -- pairs whose query nearly matches its target (see xt_bounds.cuh
// for the bounds): k_diag settles those whose diagonal alone decides, k_near
// those decided by a band of 31 diagonals, and the rest go on to the engines.
#include <algorithm>

#include "xt_kernels.cuh"
#include "xt_lane.cuh"
#include "xt_near.cuh"

namespace xt {
namespace {

// ------------------------------------------------------------------ k_diag
constexpr int kDiagThreads = 256;

// One pair along its diagonal: true when the conditions hold with c = 0,
// where they come to a total loss D (matches not made) below o + e; n and
// *bi receive the ends.  The diagonal of a row that holds no match is worth
// at least 1 throughout, or the pair fails (a dead diagonal may be revived
// from outside).  *hope: it failed while losing no faster than would come to
// k_near's bound at the query's end.
__device__ __forceinline__ bool diag_scan(const Batch& b, const Pair& pr, const Score& sc,
                                          int32_t match, NearEnd* n, int32_t* bi, bool* hope) {
  const int32_t loss_x = match - (int32_t)(int8_t)((sc.prof[0] >> 8) & 0xFF);
  const int32_t loss_n = match - (int32_t)(int8_t)(sc.nnnn & 0xFF);
  const int32_t limit = sc.alpha - 1, bound = sc.alpha + sc.beta * kNearHalf;
  ByteStream qs, ts;
  const uint8_t *qe = b.q_seq + b.q_bytes, *te = b.t_seq + b.t_bytes;
  qs.init(b.q_seq, qe, pr.q);
  ts.init(b.t_seq, te, pr.t);
  int32_t g = pr.h0, best = pr.h0, at = -1, lost = 0, pos = 0;
  for (int32_t c = 0; c < pr.qlen; c += 8) {
    const uint64_t x = qs.next(b.q_seq, qe), y = ts.next(b.t_seq, te);
    const uint64_t any_n = (x | y) & 0xFCFCFCFCFCFCFCFCull;  // a code of 4 or more
    const uint64_t z = (x ^ y) | any_n;
    uint64_t bad = (((z & 0x7F7F7F7F7F7F7F7Full) + 0x7F7F7F7F7F7F7F7Full) | z) & 0x8080808080808080ull;
    if (pr.qlen - c < 8) bad &= (1ull << (8 * (pr.qlen - c))) - 1;
    while (bad) {
      const int p = __ffsll((long long)bad) - 1;  // bit 7 of the byte
      const int32_t idx = c + (p >> 3);
      g += match * (idx - pos);
      if (g > best) { best = g; at = idx - 1; }
      const int32_t loss = ((any_n >> (p & ~7)) & 0xFF) ? loss_n : loss_x;
      g += match - loss;
      lost += loss;
      pos = idx + 1;
      if (lost > limit || g <= 0) {
        *hope = g > 0 && (int64_t)lost * pr.qlen < (int64_t)bound * pos;
        return false;
      }
      bad &= bad - 1;
    }
  }
  g += match * (pr.qlen - pos);
  if (g > best) { best = g; at = pr.qlen - 1; }
  if (sc.zdrop > 0 && lost > sc.zdrop) return false;
  n->best = best;
  n->d_best = 0;
  n->g = g;
  n->row = pr.qlen - 1;
  *bi = at;
  return true;
}

// Settles the pairs it can (class CLS_DONE, results written) and marks the
// others: CLS_NEAR for those k_near may settle, kRest for the rest.  Bounded
// by memory latency: one pair per thread, eight bytes of each sequence a step;
// results leave through shared memory so that a block's stores are whole
// lines.  Of 4M mixed 100-250-base reads (1% substitutions) it settles 69% in
// 0.45 ms, about 2 TB/s of the sequences' diagonals and the metadata.
__global__ void __launch_bounds__(kDiagThreads)
    k_diag(const Batch* __restrict__ bd, Score sc, int32_t match, bool near,
           uint8_t* __restrict__ pclass, int32_t* __restrict__ hopeful) {
  __shared__ int32_t s_out[kDiagThreads * 7];
  __shared__ uint8_t s_done[kDiagThreads];
  const Batch b = *bd;
  const int64_t base = (int64_t)blockIdx.x * kDiagThreads;
  if (base >= b.n) return;
  const int64_t kk = base + threadIdx.x;
  bool done = false, hope = false;
  if (kk < b.n) {
    const int32_t k = (int32_t)kk;
    const int64_t qo = b.q_off[k], to = b.t_off[k];
    Pair pr;
    pr.qlen = b.q_len[k];
    pr.tlen = b.t_len[k];
    pr.h0 = b.h0[k];
    const bool ok = pr.h0 >= 1 && pr.h0 <= XT_MAX_H0 && pr.qlen >= 1 && pr.qlen <= kNearMaxQ &&
                    pr.tlen >= pr.qlen && pr.tlen <= XT_MAX_LEN && qo >= 0 && to >= 0 &&
                    qo <= b.q_bytes - pr.qlen && to <= b.t_bytes - pr.tlen;
    if (ok) {
      pr.q = b.q_seq + qo;
      pr.t = b.t_seq + to;
      NearEnd n;
      int32_t bi = -1, last = -1;
      if (diag_scan(b, pr, sc, match, &n, &bi, &hope))
        last = near_last_row(n, pr.qlen, pr.tlen, pr.h0, match, sc);
      if (last >= 0) {
        done = true;
        int32_t* r = s_out + threadIdx.x * 7;
        r[0] = n.best; r[1] = bi + 1; r[2] = bi + 1; r[3] = n.g; r[4] = pr.qlen; r[5] = 0;
        r[6] = XT_OK;
        if (b.cells) b.cells[k] = band_cells_upto(last, pr.qlen, sc.w);
      }
    }
    // Off the diagonal at least gap_open is lost, and what is left has to carry the
    // deletion run from the end cell to the last row, or the last live row stays
    // unknown but for reads that lack target bases and nothing else: k_near would
    // leave the pair (short reads; 4M mixed ones 4.50 ms a call against 4.79 ms)
    bool reach = false;
    if (ok) {
      const int64_t o = sc.alpha - sc.beta;
      const int64_t rows = min((int64_t)pr.tlen - pr.qlen, (int64_t)sc.w);
      reach = sc.beta * rows <= pr.h0 + (int64_t)match * pr.qlen - 2 * o - 1;
    }
    pclass[k] = done ? (uint8_t)CLS_DONE : (reach && near ? (uint8_t)CLS_NEAR : kRest);
    hope = hope && reach && pr.h0 + match * pr.qlen <= 511;  // (and of the packed class, about)
  }
  s_done[threadIdx.x] = done;
  const int hopes = __syncthreads_count(hope);
  if (threadIdx.x == 0 && near && hopes > 0) atomicAdd(hopeful, hopes);
  int32_t* out = reinterpret_cast<int32_t*>(b.out + base);
#pragma unroll
  for (int u = 0; u < 7; ++u) {
    const int i = u * kDiagThreads + threadIdx.x;
    if (s_done[i / 7]) out[i] = s_out[i];
  }
}

// ------------------------------------------------------------------ k_near
constexpr int kNearThreads = 128;
constexpr int kNearBlocks = 3;  // per SM: up to 168 registers
constexpr int kC = kNearHalf;
constexpr int kSlots = 2 * kC + 1;
constexpr int kKeyBits = 5;
static_assert(kSlots < (1 << kKeyBits) && kSlots <= 32, "slot index fits the row key");
// Two pairs per lane, one in each 16-bit half of every register.  A row's
// kSlots cells sit in registers by diagonal: slot s of row i is column
// i - kC + s, so the diagonal neighbour of the row above has the same slot
// and the one above it the next, and the sweep needs no boundary rows, no
// masks and no memory but the two sequences.  The column before the query and
// the row before the target come out of the same recurrence from the seed's
// slot; columns past the query score kPadScore, which keeps every cell there
// below a cell of the same row inside (alpha from 1 to 127).  Scores: a byte
// permute looks four slots up at once, the target base's score table indexed
// by four query nibbles, and one more per slot puts the two pairs' bytes,
// sign-extended, side by side.
//
// Bounded by the integer ALU pipe: 31 slots of about 10 instructions per row
// of two pairs.  Of the same 4M reads it took the 1.2M left and settled half of
// them in 1.53 ms, 1.20 ms now that k_diag keeps from it the short ones it could
// not settle; the call went from 18.3 to 4.5 ms (1M 150-base reads: 4.6 to 1.15
// ms), as the full band's 201 diagonals are left to 15% of the pairs.
// 31 diagonals are what two pairs' cells, with 16 bits each, leave of 168
// registers; they admit a loss of 21 against a perfect match.
__global__ void __launch_bounds__(kNearThreads, kNearBlocks)
    k_near(const Batch* __restrict__ bd, Score sc, Work w, int32_t match, uint32_t mcm,
           uint32_t kmul, int head_id) {
  __shared__ Batch s_b;
  __shared__ uint32_t s_tbl[8];
  __shared__ uint32_t s_row[kSlots][kNearThreads];
  if (threadIdx.x == 0) {
    s_b = *bd;
#pragma unroll
    for (int c = 0; c < 5; ++c) s_tbl[c] = sc.prof[c];  // S is symmetric: a target base's scores
  }
  __syncthreads();
  const Batch& b = s_b;
  const int lane = threadIdx.x & 31;
  const int32_t begin = w.seg_begin[CLS_NEAR * kNumJ + kNearJMax];
  const int32_t end = w.seg_end[CLS_NEAR * kNumJ + kJMin];
  int32_t* head = w.heads + head_id;
  const int32_t alpha = sc.alpha, beta = sc.beta, gopen = alpha - beta;
  const uint32_t na2 = pack16(-alpha, -alpha), nb2 = pack16(-beta, -beta);
  const uint32_t nn = (sc.nnnn & 0xFFu) | (kPadScore << 8);
  const uint32_t a2 = pack16(match, match);
  const int32_t qbound = gopen + beta * (kC + 1);  // Q
  for (;;) {
    int32_t base = 0;
    if (lane == 0) base = atomicAdd(head, 64);
    base = begin + __shfl_sync(0xffffffffu, base, 0);
    if (base >= end) break;
    int32_t kk[2], ql[2], tl[2], h0[2], rmax[2];
    ByteStream qs[2], ts[2];
    uint32_t act = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int32_t idx = base + 2 * lane + h;
      int32_t k = idx < end ? w.order[idx] : -1;
      if ((uint32_t)k >= (uint32_t)b.n) k = -1;  // a corrupt workspace: no pair
      kk[h] = k;
      ql[h] = k >= 0 ? b.q_len[k] : 1;
      tl[h] = k >= 0 ? b.t_len[k] : 1;
      h0[h] = k >= 0 ? b.h0[k] : 1;
      rmax[h] = k >= 0 ? min(tl[h] - 1, ql[h] - 1 + kC) : -1;
      qs[h].init(b.q_seq, b.q_seq + b.q_bytes, b.q_seq + (k >= 0 ? b.q_off[k] : 0) - kC);
      ts[h].init(b.t_seq, b.t_seq + b.t_bytes, b.t_seq + (k >= 0 ? b.t_off[k] : 0));
      if (k >= 0) act |= 0xFFFFu << (16 * h);
    }
    const int32_t rows = __reduce_max_sync(0xffffffffu, max(rmax[0], rmax[1])) + 1;
    // row -1: slot s is column s - kC - 1
    uint32_t H[kSlots], F[kSlots];  // F: of the row to come
#pragma unroll
    for (int s = 0; s < kSlots; ++s) {
      const int32_t c = s - kC - 1;
      int32_t v[2];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        v[h] = c < -1 ? 0 : (c == -1 ? h0[h] : (c < ql[h] ? max(0, h0[h] - alpha - beta * c) : 0));
      H[s] = pack16(v[0], v[1]);
    }
#pragma unroll
    for (int s = 0; s < kSlots; ++s)
      F[s] = s + 1 < kSlots ? __viaddmax_s16x2_relu(H[s + 1], na2, 0u) : 0u;
    uint32_t best2 = pack16(h0[0], h0[1]), p2 = best2, worst2 = 0, zmax2 = 0;
    const uint32_t pq2 = pack16(h0[0] + match * ql[0], h0[1] + match * ql[1]);
    int32_t brow[2] = {-1, -1}, bslot[2] = {kC, kC}, off[2] = {0, 0}, g[2] = {-1, -1},
            grow[2] = {0, 0};
    // query nibbles: word u holds columns 8u - kC .. 8u - kC + 7
    uint32_t win[2][5];
    int32_t qpos = -kC;
#pragma unroll
    for (int u = 0; u < 5; ++u, qpos += 8)
#pragma unroll
      for (int h = 0; h < 2; ++h) win[h][u] = nibbles(qs[h].next(b.q_seq, b.q_seq + b.q_bytes), ql[h] - qpos);
    for (int32_t i8 = 0; i8 < rows; i8 += 8) {
      uint32_t tw[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) tw[h] = nibbles(ts[h].next(b.t_seq, b.t_seq + b.t_bytes), 8);
      const int32_t i_end = min(i8 + 8, rows);
#pragma unroll 1
      for (int32_t i = i8; i < i_end; ++i) {
        const int sh = 4 * (i - i8);
        uint32_t x[2][4];
        uint32_t tbl[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          tbl[h] = s_tbl[(tw[h] >> sh) & 7u];
#pragma unroll
          for (int u = 0; u < 4; ++u) x[h][u] = __funnelshift_r(win[h][u], win[h][u + 1], sh);
        }
        uint32_t key = 0, E = 0, HA = na2;
        uint32_t s4[2];
#pragma unroll
        for (int s = 0; s < kSlots; ++s) {
          if (s % 4 == 0) {
#pragma unroll
            for (int h = 0; h < 2; ++h)
              s4[h] = prmt(tbl[h], nn, x[h][s / 8] >> (s % 8 ? 16 : 0));
          }
          constexpr uint32_t kSel[4] = {0xC480u, 0xD591u, 0xE6A2u, 0xF7B3u};
          const uint32_t S = prmt(s4[0], s4[1], kSel[s % 4]);
          const uint32_t D = H[s];
          const uint32_t M = __viaddmin_s16x2(D, S, D * mcm);
          E = s ? __viaddmax_s16x2_relu(E, nb2, HA) : 0u;
          const uint32_t f = F[s];
          const uint32_t h2 = __vimax3_s16x2(M, E, f);
          HA = add16x2(h2, na2);
          key = __viaddmax_s16x2(h2 * kmul, (uint32_t)s * 0x00010001u, key);
          if (s) F[s - 1] = __viaddmax_s16x2_relu(f, nb2, HA);
          H[s] = h2;
        }
        // the row maximum; the column before the query (rows 0 .. kC-1) may
        // hold it only below the best, so it matters to the z-drop bound alone
        const uint32_t m2 = (key >> kKeyBits) & 0x07FF07FFu & act;
        const uint32_t was2 = best2;
        asm("max.s16x2 %0, %0, %1;" : "+r"(best2) : "r"(m2));
        const uint32_t up = was2 ^ best2;
        if (up & 0xFFFFu) {
          brow[0] = i;
          bslot[0] = key & 31u;
          off[0] = max(off[0], abs(bslot[0] - kC));
        }
        if (up >> 16) {
          brow[1] = i;
          bslot[1] = (key >> 16) & 31u;
          off[1] = max(off[1], abs(bslot[1] - kC));
        }
        asm("min.s16x2 %0, %1, %2;" : "=r"(p2) : "r"(add16x2(p2, a2)), "r"(pq2));
        // p2 >= best2 and best2 >= mz in each half: no borrow between halves
        asm("max.s16x2 %0, %0, %1;" : "+r"(worst2) : "r"(p2 - best2));
        uint32_t mz = m2;
        if (i < kC) {
          const int32_t c0 = max(0, h0[0] - alpha - beta * i), c1 = max(0, h0[1] - alpha - beta * i);
          if (lo16(m2) <= c0) mz &= 0xFFFF0000u;
          if (hi16(m2) <= c1) mz &= 0x0000FFFFu;
        }
        asm("max.s16x2 %0, %0, %1;" : "+r"(zmax2) : "r"((best2 - mz) & act));
        // rows whose band holds the last query column: its cell, and the end
        const bool ends = ((act & 0xFFFFu) && i >= ql[0] - 1 - kC) ||
                          ((act >> 16) && i >= ql[1] - 1 - kC);
        if (__any_sync(0xffffffffu, ends)) {
#pragma unroll
          for (int s = 0; s < kSlots; ++s) s_row[s][threadIdx.x] = H[s];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int32_t s = ql[h] - 1 - i + kC;
            if (((act >> (16 * h)) & 1u) && s >= 0 && s < kSlots) {
              const uint32_t v = s_row[s][threadIdx.x];
              const int32_t ge = h ? hi16(v) : lo16(v);
              if (ge > 0 && ge > g[h]) {
                g[h] = ge;
                grow[h] = i;
              }
              const int32_t pq = h0[h] + match * ql[h];
              if (i >= rmax[h] ||
                  (s <= kC && g[h] > 0 && pq - gopen - beta * (i + 2 - ql[h]) <= g[h]))
                act &= ~(0xFFFFu << (16 * h));
            }
          }
        }
      }
      // a pair whose bounds are broken stops here
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t lost = h ? hi16(worst2) : lo16(worst2), z = h ? hi16(zmax2) : lo16(zmax2);
        if (lost >= qbound || (sc.zdrop > 0 && z > sc.zdrop)) act &= ~(0xFFFFu << (16 * h));
      }
      if (!__any_sync(0xffffffffu, act != 0)) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int u = 0; u < 4; ++u) win[h][u] = win[h][u + 1];
        win[h][4] = nibbles(qs[h].next(b.q_seq, b.q_seq + b.q_bytes), ql[h] - qpos);
      }
      qpos += 8;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (kk[h] < 0) continue;
      NearEnd n;
      n.best = h ? hi16(best2) : lo16(best2);
      n.d_best = kC - bslot[h];
      n.g = g[h];
      n.row = grow[h];
      const int32_t lost = h ? hi16(worst2) : lo16(worst2), z = h ? hi16(zmax2) : lo16(zmax2);
      int32_t last = -1;
      if (lost < qbound && (sc.zdrop <= 0 || z <= sc.zdrop) && n.g > 0 &&
          h0[h] + match * ql[h] - n.g < qbound)
        last = near_last_row(n, ql[h], tl[h], h0[h], match, sc);
      if (last >= 0) {
        write_result(b, kk[h], n.best, brow[h] - n.d_best + 1, brow[h] + 1, n.g, n.row + 1, off[h],
                     XT_OK, band_cells_upto(last, ql[h], sc.w));
      } else {
        const int nb = bin_of_len(ql[h]), bin = CLS_NEAR * kClassBins + nb;
        const int32_t at = w.cursor[bin] - w.counts[bin] + atomicAdd(&w.near_left[nb], 1);
        w.near_tmp[at] = kk[h];
      }
    }
  }
}

// Pairs left by k_near, from their length's run in near_tmp to one run in the
// queue at the class's place (longest first, as every segment); the class's
// segment table then covers the pairs left.  Every block scans the bins and then
// takes its share of the pairs, finding a pair's bin in the scan: a warp per bin
// left a batch of one length to one warp (1M reads of 150 bases a call, 4%
// substitutions 17.2 -> 7.8 ms, 1% 3.26 -> 1.97 ms).
constexpr int kGatherThreads = kNearBins;  // a thread per bin
constexpr int kGatherBlocks = 152;  // one per SM

__global__ void __launch_bounds__(kGatherThreads) k_near_gather(Work w) {
  __shared__ int32_t s_pre[kNearBins];  // in queue order
  __shared__ int32_t s_src[kNearBins];  // the bin's run in near_tmp, less s_pre
  __shared__ int32_t s_warp[kGatherThreads / 32];
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  // queue position u -> bin kNearBins - 1 - u (longest length first)
  const int nb = kNearBins - 1 - t, bin = CLS_NEAR * kClassBins + nb;
  const int32_t c0 = w.near_left[nb];
  int32_t inc = c0;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int32_t v = __shfl_up_sync(0xffffffffu, inc, d);
    if (lane >= d) inc += v;
  }
  if (lane == 31) s_warp[wid] = inc;
  __syncthreads();
  int32_t before = inc - c0, left = 0;
  for (int u = 0; u < kGatherThreads / 32; ++u) {
    if (u < wid) before += s_warp[u];
    left += s_warp[u];
  }
  s_pre[t] = before;
  s_src[t] = w.cursor[bin] - w.counts[bin] - before;
  __syncthreads();
  const int32_t region = w.seg_begin[CLS_NEAR * kNumJ + kJMax];  // never rewritten below
  for (int32_t i = blockIdx.x * kGatherThreads + t; i < left; i += gridDim.x * kGatherThreads) {
    int u = 0;  // the last bin in queue order that starts at i or before
#pragma unroll
    for (int step = kNearBins / 2; step > 0; step >>= 1)
      if (s_pre[u + step] <= i) u += step;
    w.order[region + i] = w.near_tmp[s_src[u] + i];
  }
  if (blockIdx.x == 0) {
    if (longest_bin(nb)) w.seg_begin[CLS_NEAR * kNumJ + bucket_of_bin(nb)] = region + before;
    if (shortest_bin(nb)) w.seg_end[CLS_NEAR * kNumJ + bucket_of_bin(nb)] = region + before + c0;
  }
}

}  // namespace

cudaError_t launch_diag(const Batch* bd, int32_t n_cap, const Score& sc, int32_t match, bool near,
                        const Work& w, cudaStream_t stream) {
  if (n_cap == 0) return cudaSuccess;
  const int grid = (int)(((int64_t)n_cap + kDiagThreads - 1) / kDiagThreads);
  k_diag<<<grid, kDiagThreads, 0, stream>>>(bd, sc, match, near, w.pclass, w.near_hope);
  return cudaGetLastError();
}

int near_grid(int32_t pairs, int num_sms) {
  const int64_t want = ((int64_t)pairs + 2 * kNearThreads - 1) / (2 * kNearThreads);
  return rounded_grid(want, num_sms, kNearBlocks);
}

cudaError_t launch_near(const Batch* bd, const Score& sc, int32_t match, int grid, const Work& w,
                        int head_id, cudaStream_t stream) {
  if (grid <= 0) return cudaSuccess;
  int mshift = 0;
  while ((1 << mshift) < match + 1) ++mshift;
  k_near<<<grid, kNearThreads, 0, stream>>>(bd, sc, w, match, 1u << mshift, 1u << kKeyBits, head_id);
  k_near_gather<<<kGatherBlocks, kGatherThreads, 0, stream>>>(w);
  return cudaGetLastError();
}

}  // namespace xt
