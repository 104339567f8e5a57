// xt_bwa.cu -- the BWA-MEM-compatible extension (xt_extend_batch_bwa).
//
// The variant (stated in full in include/xt.h) opens gaps from the match value
// M rather than from H and drops the dead cells at both ends of each row.
// Both change how the work parallelises:
//
//  * the insertion chain E of a row depends only on that row's M values,
//    E(i,j) = max(0, max_{k<j} (M(i,k) - o_ins - e_ins*(j-k))), a max-plus
//    prefix scan over the row, and M and F depend only on the row above: a row
//    is data-parallel across its columns;
//  * trimming makes row i+1's columns depend on all of row i (its first and
//    last live cells), so rows must go one after another -- the strip scheme
//    of the default kernels, which keeps several rows in flight, does not
//    apply.
//
// So one pair is extended by a group of G lanes that computes a whole row at
// a time, and only the row's own columns [beg, end): trimming keeps a row far
// narrower than its band (about a quarter of 2w'+1 on short reads), so the
// lanes split the row's width, k = ceil((end - beg) / G) <= K consecutive
// columns each, and the row above lives in shared memory rather than in fixed
// registers.  Per row the group runs an exclusive max-scan for the insertion
// chain, a max-reduction for the row maximum and its column, and a min/max
// reduction for the row's first and last live columns.  G*K is the smallest power of two >= min(qlen,
// 2w'+1), from 64 to 8192 columns; up to 32 lanes a group is a warp segment
// (shuffles), above that a whole CTA (shuffles plus shared memory).  Pairs are
// classified by G*K, and each class runs a persistent kernel whose groups take
// pairs from a counter.
//
// Batches of many short queries run two pairs per lane instead (k_bwa_lane): a
// row then needs no collectives at all.
#include <algorithm>
#include <climits>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "xt.h"
#include "xt_common.cuh"
#include "xt_ctx.cuh"
#include "xt_fork.cuh"
#include "xt_near.cuh"

namespace xt {
namespace {

// Most columns a lane computes in a row (16 or 32): more columns per lane
// means fewer lanes per pair and cheaper per-row collectives, at two
// registers per column.
#ifndef XT_BWA_LANE_COLUMNS
#define XT_BWA_LANE_COLUMNS 32
#endif
constexpr int kBwaK = XT_BWA_LANE_COLUMNS;
static_assert(kBwaK == 16 || kBwaK == 32, "columns per lane: 16 or 32");
constexpr int kBwaGroupClasses = 8;          // G*K = 64 << class columns
// Two pairs per lane: classes by the columns a lane's row buffer has room for; all
// but the last keep a score in a byte.
constexpr int kBwaLaneMinQ = 33;
constexpr int kBwaLaneClasses = 3;
__host__ __device__ constexpr int bwa_lane_cap(int c) { return 64 << c; }
// With fewer pairs of a class its last pairs decide, which a group extends
// sooner (500k / 128k / 64k mixed reads: 7.1 / 2.0 / 1.2 ms on groups alone, 5.2 /
// 1.6 / 1.5 ms with every class on lanes, those up to 64 bases 0.77 and 0.95 ms of
// it; 2M: 28.0 and 18.1 ms).
__host__ __device__ constexpr int32_t bwa_lane_min(int c) { return c == 0 ? 1 << 18 : 1 << 15; }
// The widest lane class holds so little of the SM that rows of few columns run sooner
// on groups of two to four lanes (400k reads of 200 bases, w = 10 / 20 / 40 / 70: 5.06 /
// 6.54 / 9.1 / 11.8 ms on lanes, 3.55 / 5.14 / 9.9 / 16.0 on groups).
constexpr int kBwaLaneMinWidth = 89;
constexpr int kBwaClasses = 16;              // of them 11 in use (their order is the queue's)
// The shortest lane class lies before the narrowest groups, which may take it.
__host__ __device__ constexpr int bwa_lane_id(int c) { return c == 0 ? 0 : kBwaGroupClasses + c; }
__host__ __device__ constexpr int bwa_group_id(int c) { return 1 + c; }
__host__ __device__ constexpr bool bwa_is_lane(int id) { return id == 0 || id > kBwaGroupClasses; }
constexpr int kBwaWarpThreads = 128;         // CTA size of the warp-segment classes
constexpr int32_t kBwaNeg = -(1 << 29);      // below any reachable value
constexpr uint8_t kBwaDone = 0xff;           // pair finished in classify
// Within a class pairs go longest query first, in buckets of query length
// (capped): the groups sharing a warp then extend pairs of like length, whose
// rows are of like width, and the longest pairs do not start last.
constexpr int kBwaLenBuckets = 1024;
constexpr int kBwaScanThreads = 1024;
// A row buffer element's y word: the column's query code above F.
constexpr int kCodeShift = 28;
constexpr uint32_t kFMask = (1u << kCodeShift) - 1u;
static_assert((int64_t)XT_MAX_H0 + (int64_t)XT_MAX_LEN * 127 < (1ll << kCodeShift), "F fits below the code");
static_assert(kBwaLenBuckets * kBwaClasses % kBwaScanThreads == 0, "scan tiling");

static_assert((64 << (kBwaGroupClasses - 1)) == XT_BWA_MAX_WIDTH, "class range must end at the limit");

// Two pairs per lane: the row's key is H * 32 + the chunk of 8 columns.
constexpr int32_t kBwaLaneMaxH = 1023;

struct BwaScore {
  int32_t match, mismatch, nsc;
  int32_t o_ins, e_ins, o_del, e_del;
  int32_t w, zdrop, end_bonus;
};

struct BwaArgs {
  const uint8_t* q_seq;
  const uint8_t* t_seq;
  const int64_t* q_off;
  const int64_t* t_off;
  const int32_t* q_len;
  const int32_t* t_len;
  const int32_t* h0;
  int64_t q_bytes, t_bytes;
  int32_t n;
  xt_result* out;
  int64_t* cells;
  BwaScore sc;
  int mshift;        // 2^mshift > match
  int coarse;        // 2^coarse neighbouring length buckets of a class in one slot
  uint8_t* pclass;   // [n]
  int32_t* order;    // [n] pairs by class, then by query length (longest first)
  int32_t* slots;    // [kBwaClasses * (kBwaLenBuckets >> coarse)] pairs per (class, length), then
                     // positions
  int32_t* counts;   // [kBwaClasses] pairs per class
  int32_t* heads;    // [kBwaClasses] next pair of each class's persistent kernel
};

// Slot of a pair of class c, query length ql and seed score h0: classes in order,
// longer queries first within a class; with two pairs per lane, whose warps sweep
// the columns alive in any of 64 pairs, pairs of like seed scores together.
__device__ __forceinline__ int32_t bwa_slot(int c, int32_t ql, int32_t h0, int coarse) {
  const int32_t key = !bwa_is_lane(c) ? ql : 4 * (ql - 1) + min(h0 >> 4, 3);
  const int32_t b = key < kBwaLenBuckets - 1 ? key : kBwaLenBuckets - 1;
  return (c * kBwaLenBuckets + (kBwaLenBuckets - 1 - b)) >> coarse;
}

// The narrowed band half-width of a pair with query length qlen.
__host__ __device__ inline int32_t bwa_band(const BwaScore& s, int32_t qlen) {
  const int64_t gain = (int64_t)qlen * s.match + s.end_bonus;
  const int64_t wi = gain < s.o_ins ? 1 : (gain - s.o_ins) / s.e_ins + 1;
  const int64_t wd = gain < s.o_del ? 1 : (gain - s.o_del) / s.e_del + 1;
  int64_t w = s.w;
  if (wi < w) w = wi;
  if (wd < w) w = wd;
  return (int32_t)w;
}

__device__ __forceinline__ void put_result(const BwaArgs& a, int32_t k, int32_t score, int32_t qle,
                                           int32_t tle, int32_t gscore, int32_t gtle,
                                           int32_t max_off, int32_t status, int64_t cells) {
  xt_result r;
  r.score = score; r.qle = qle; r.tle = tle; r.gscore = gscore; r.gtle = gtle;
  r.max_off = max_off; r.status = status;
  a.out[k] = r;
  if (a.cells) a.cells[k] = cells;
}

// ---------------------------------------------------------------- classify
// Checks every pair, finishes the degenerate and invalid ones, and counts the
// rest per (class, query length) slot.
__global__ void k_bwa_classify(BwaArgs a) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t ql = a.q_len[k], tl = a.t_len[k], h0 = a.h0[k];
    const int64_t qo = a.q_off[k], to = a.t_off[k];
    bool ok = h0 >= 1 && h0 <= XT_MAX_H0 && ql >= 0 && tl >= 0 && ql <= XT_MAX_LEN &&
              tl <= XT_MAX_LEN && qo >= 0 && to >= 0 && qo <= a.q_bytes - ql &&
              to <= a.t_bytes - tl;
    int32_t width = 0;
    if (ok) {
      const int64_t wb = 2 * (int64_t)bwa_band(a.sc, ql) + 1;
      width = (int32_t)(wb < ql ? wb : ql);
      ok = width <= XT_BWA_MAX_WIDTH;
    }
    uint8_t cls = kBwaDone;
    if (!ok) {
      put_result(a, (int32_t)k, 0, 0, 0, 0, 0, 0, XT_EINVAL, 0);
    } else if (ql == 0) {
      put_result(a, (int32_t)k, h0, 0, 0, h0, 0, 0, XT_OK, 0);
    } else if (tl == 0) {
      put_result(a, (int32_t)k, h0, 0, 0, -1, 0, 0, XT_OK, 0);
    } else {
      int c = 0;
      const int64_t bound = h0 + (int64_t)ql * a.sc.match;
      bool lane = ql >= kBwaLaneMinQ && ql <= bwa_lane_cap(kBwaLaneClasses - 1) &&
                  bound <= kBwaLaneMaxH && ((bound + 1) << a.mshift) <= 32767;
      if (lane) {
        while (bwa_lane_cap(c) < ql) ++c;
        if (bound > 255) c = kBwaLaneClasses - 1;
        lane = c < kBwaLaneClasses - 1 || width >= kBwaLaneMinWidth;
      }
      if (lane) {
        c = bwa_lane_id(c);
      } else {
        for (c = 0; (64 << c) < width;) ++c;
        c = bwa_group_id(c);
      }
      cls = (uint8_t)c;
      atomicAdd(&a.slots[bwa_slot(cls, ql, h0, a.coarse)], 1);
    }
    a.pclass[k] = cls;
  }
}

// One block: slot counts to first positions (exclusive scan in slot order)
// and the pairs per class.
__global__ void __launch_bounds__(kBwaScanThreads) k_bwa_scan(BwaArgs a) {
  constexpr int kPer = kBwaClasses * kBwaLenBuckets / kBwaScanThreads;
  constexpr int kPerClass = kBwaLenBuckets / kPer;  // threads per class (of coarse slots too)
  const int per = kPer >> a.coarse;
  __shared__ int32_t s_warp[kBwaScanThreads / 32];
  __shared__ int32_t s_class[kBwaClasses];
  const int tid = threadIdx.x;
  int32_t v[kPer];
  int32_t sum = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    v[u] = u < per ? a.slots[tid * per + u] : 0;
    sum += v[u];
  }
  if (tid < kBwaClasses) s_class[tid] = 0;
  // inclusive scan of the thread sums
  int32_t inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if ((tid & 31) >= o) inc += t;
  }
  if ((tid & 31) == 31) s_warp[tid >> 5] = inc;
  __syncthreads();
  int32_t before = inc - sum;
  for (int u = 0; u < (tid >> 5); ++u) before += s_warp[u];
  atomicAdd(&s_class[tid / kPerClass], sum);
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    if (u < per) a.slots[tid * per + u] = before;
    before += v[u];
  }
  __syncthreads();
  if (tid < kBwaClasses) a.counts[tid] = s_class[tid];
}

// Each pair takes the next position of its slot.
__global__ void k_bwa_scatter(BwaArgs a) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < a.n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int c = a.pclass[k];
    if (c == kBwaDone) continue;
    const int32_t pos = atomicAdd(&a.slots[bwa_slot(c, a.q_len[k], a.h0[k], a.coarse)], 1);
    if (pos >= 0 && pos < a.n) a.order[pos] = (int32_t)k;
  }
}

// ------------------------------------------------------------ lane groups
// Collectives of the G lanes that extend one pair.
template <int G, bool kSegment = (G <= 32)>
struct Group;

// A warp segment of G lanes (G <= 32).
template <int G>
struct Group<G, true> {
  unsigned mask;
  int lane;
  __device__ __forceinline__ void init() {
    const int wl = threadIdx.x & 31;
    lane = wl & (G - 1);
    mask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (wl & ~(G - 1)));
  }
  __device__ __forceinline__ int index() const { return lane; }
  // orders the group's shared-memory accesses before and after it
  __device__ __forceinline__ void sync() const { __syncwarp(mask); }
  // max over the lanes before this one (kBwaNeg for lane 0)
  __device__ __forceinline__ int32_t excl_max(int32_t v) const {
#pragma unroll
    for (int o = 1; o < G; o <<= 1) {
      const int32_t t = __shfl_up_sync(mask, v, o, G);
      if (lane >= o) v = max(v, t);
    }
    const int32_t r = __shfl_up_sync(mask, v, 1, G);
    return lane == 0 ? kBwaNeg : r;
  }
  // *m = max of v over the group, *at = the largest col among the lanes
  // holding it.  A whole warp uses the warp-reduction instructions; a warp
  // segment, whose neighbours in the warp reduce over other masks at the same
  // time, a shuffle tree (measured faster there).
  __device__ __forceinline__ void max_last(int32_t v, int32_t col, int32_t* m,
                                           int32_t* at) const {
    if constexpr (G == 32) {
      const int32_t x = __reduce_max_sync(mask, v);
      *m = x;
      *at = __reduce_max_sync(mask, v == x ? col : INT32_MIN);
    } else {
      int64_t key = ((int64_t)v << 32) | (uint32_t)col;
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        const int64_t t = __shfl_xor_sync(mask, key, o, G);
        key = t > key ? t : key;
      }
      *m = (int32_t)(key >> 32);
      *at = (int32_t)(key & 0xffffffff);
    }
  }
  // (max of a, min of b) over the group
  __device__ __forceinline__ void all_max_min(int32_t* a, int32_t* b) const {
    if constexpr (G == 32) {
      *a = __reduce_max_sync(mask, *a);
      *b = __reduce_min_sync(mask, *b);
    } else {
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        *a = max(*a, __shfl_xor_sync(mask, *a, o, G));
        *b = min(*b, __shfl_xor_sync(mask, *b, o, G));
      }
    }
  }
  // one lane takes the next pair of the class for the whole group
  __device__ __forceinline__ int32_t claim(int32_t* head) const {
    int32_t p = 0;
    if (lane == 0) p = atomicAdd(head, 1);
    return __shfl_sync(mask, p, 0, G);
  }
};

// A whole CTA of G lanes (G >= 64): shuffles inside warps, shared memory
// across them.  Each collective writes its own shared array once per row and
// ends with one barrier; at least one other barrier separates two uses of the
// same array, so a lane can never overwrite a value another lane still reads.
template <int G>
struct Group<G, false> {
  static constexpr int kW = G / 32;
  struct Shared {
    int32_t scan[kW];
    int64_t key[kW];
    int32_t amax[kW], amin[kW];
    int32_t claim;
  };
  Shared* sh;
  int lane, wl, wid;
  __device__ __forceinline__ void init(Shared* s) {
    sh = s;
    lane = threadIdx.x;
    wl = lane & 31;
    wid = lane >> 5;
  }
  __device__ __forceinline__ int index() const { return lane; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ int32_t excl_max(int32_t v) const {
    int32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int32_t t = __shfl_up_sync(0xffffffffu, inc, o);
      if (wl >= o) inc = max(inc, t);
    }
    if (wl == 31) sh->scan[wid] = inc;
    int32_t ex = __shfl_up_sync(0xffffffffu, inc, 1);
    if (wl == 0) ex = kBwaNeg;
    __syncthreads();
    for (int u = 0; u < wid; ++u) ex = max(ex, sh->scan[u]);
    return ex;
  }
  __device__ __forceinline__ int64_t all_max64(int64_t v) const {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const int64_t t = __shfl_xor_sync(0xffffffffu, v, o);
      v = t > v ? t : v;
    }
    if (wl == 0) sh->key[wid] = v;
    __syncthreads();
    int64_t r = sh->key[0];
    for (int u = 1; u < kW; ++u) r = sh->key[u] > r ? sh->key[u] : r;
    return r;
  }
  // *m = max of v over the group, *at = col of the highest lane holding it
  __device__ __forceinline__ void max_last(int32_t v, int32_t col, int32_t* m,
                                           int32_t* at) const {
    const int64_t key = all_max64(((int64_t)v << 32) | (uint32_t)col);
    *m = (int32_t)(key >> 32);
    *at = (int32_t)(key & 0xffffffff);
  }
  __device__ __forceinline__ void all_max_min(int32_t* a, int32_t* b) const {
    *a = __reduce_max_sync(0xffffffffu, *a);
    *b = __reduce_min_sync(0xffffffffu, *b);
    if (wl == 0) {
      sh->amax[wid] = *a;
      sh->amin[wid] = *b;
    }
    __syncthreads();
    int32_t x = sh->amax[0], y = sh->amin[0];
    for (int u = 1; u < kW; ++u) {
      x = max(x, sh->amax[u]);
      y = min(y, sh->amin[u]);
    }
    *a = x;
    *b = y;
  }
  __device__ __forceinline__ int32_t claim(int32_t* head) const {
    __syncthreads();  // the previous pair's readers of sh->claim are done
    if (lane == 0) sh->claim = atomicAdd(head, 1);
    __syncthreads();
    return sh->claim;
  }
};

// Score row for target code ti (0..4) as biased bytes: byte c of {hi:lo} is
// S(ti, query code c) + 128, c = 0..4; bytes 5..7 are 0.
__device__ __forceinline__ void score_row(uint32_t ti, uint32_t mism4, uint32_t nb, uint32_t mb,
                                          uint32_t* lo, uint32_t* hi) {
  if (ti >= 4u) {
    *lo = nb * 0x01010101u;
  } else {
    const uint32_t sh = 8u * ti;
    *lo = (mism4 & ~(0xffu << sh)) | (mb << sh);
  }
  *hi = nb;
}

// --------------------------------------------------------------- the kernel
// One pair per group of G lanes.  Row i computes only its columns [beg, end):
// lane l takes k consecutive columns from beg + l*k (fewer in the last lanes),
// k = ceil((end - beg) / G) rounded up to odd while <= K.  The row above lives
// in the group's buffer of G*K + 2 elements, one per column j of [beg - 1,
// end]: x = H(i-1, j) and y = query code of column j << 28 | F(i, j), at index
// j - o(i-1) with the origin o(r) = max(-1, r - w' - 1).  The origin moves by
// 0 or 1 column a row, so a row's reads (x of column j-1, y of column j) and
// its writes (column j at index j - o(i)) touch the same window; a barrier of
// the group separates the row's reads from its writes.  Two extra elements per row hold the
// boundary: column beg-1 (x = H of column -1 for the next row: the deletion
// run from the seed, else 0) and column end (y = its query code << 28 | 0).
// F and H stay below 2^28: H <= h0 + qlen * match <= 2^20 + 2^20 * 127.
// A group's row buffer, element e at base[e * S]: the buffers of the S groups
// that share a half-warp are interleaved element by element (S = 16 / G for
// groups of up to 8 lanes, else 1).  With each lane's columns an odd count,
// the G lanes of a group then fall on distinct bank pairs of one residue
// class mod 2S, and the S groups on different classes, so a half-warp's
// 8-byte accesses meet no bank conflict whatever each group's row offsets.
template <int S>
struct RowBuf {
  int2* base;
  __device__ __forceinline__ int2& operator[](int32_t e) const { return base[e * S]; }
  __device__ __forceinline__ RowBuf operator+(int32_t e) const { return RowBuf{base + e * S}; }
};

template <int G, int K, typename Buf>
__device__ __forceinline__ void bwa_pair(const BwaArgs& a, const Group<G>& g, Buf buf,
                                         int32_t k) {
  const BwaScore& sc = a.sc;
  const int32_t qlen = a.q_len[k], tlen = a.t_len[k], h0 = a.h0[k];
  const uint8_t* q = a.q_seq + a.q_off[k];
  const uint8_t* t = a.t_seq + a.t_off[k];
  const int32_t w = bwa_band(sc, qlen);
  const int32_t oe_ins = sc.o_ins + sc.e_ins, oe_del = sc.o_del + sc.e_del;
  const int32_t e_ins = sc.e_ins, e_del = sc.e_del;
  const uint32_t mb = (uint32_t)(sc.match + 128), nb = (uint32_t)(sc.nsc + 128);
  const uint32_t mism4 = (uint32_t)(sc.mismatch + 128) * 0x01010101u;
  const int lane = g.index();

  // row -1 (origin -1): the seed at column -1, the insertion run from it
  // inside the band, no deletion state; each element carries its column's code
  int32_t end = min(qlen, w + 1);
#pragma unroll 4
  for (int32_t idx = lane; idx < end + 2; idx += G) {
    const int32_t j = idx - 1;
    int32_t x = h0;
    if (j >= 0) {
      const int32_t v = h0 - oe_ins - e_ins * j;
      x = (j < qlen && j + 1 <= w && v > 0) ? v : 0;
    }
    const uint32_t c = (j >= 0 && j < qlen) ? clamp_code(q[j]) : 4u;
    buf[idx] = make_int2(x, (int32_t)(c << kCodeShift));
  }
  g.sync();
  int32_t beg = 0;
  int32_t best = h0, bi = -1, bj = -1, max_off = 0, gscore = -1, gtle = 0;
  int64_t cells = 0;
  uint32_t t_next = tlen > 0 ? t[0] : 4u;

  for (int32_t i = 0; i < tlen; ++i) {
    if (beg >= end) break;  // nothing to compute: the row maximum is 0
    const int32_t o_up = max(-1, i - w - 2), o_row = max(-1, i - w - 1);
    uint32_t rp_lo, rp_hi;
    score_row(clamp_code(t_next), mism4, nb, mb, &rp_lo, &rp_hi);
    if (i + 1 < tlen) t_next = t[i + 1];
    // the query code of column end enters with the row's boundary element
    const uint32_t q_end = (lane == G - 1 && end < qlen) ? clamp_code(q[end]) : 4u;
    // columns per lane: ceil((end - beg) / G) <= K (end - beg <= min(qlen, 2w'+1)),
    // rounded up to odd where that stays <= K, so that the lanes of a group
    // read and write distinct shared-memory banks
    const int32_t kq = min(((end - beg + G - 1) / G) | 1, K);
    const int32_t first = beg + lane * kq;
    const int32_t cnt = max(0, min(kq, end - first));

    // pass 1: M, F and H without the insertion carry from earlier lanes;
    // Y is the lane's insertion chain, started from 0
    // The F word of column j goes to the buffer at once: its index in this
    // row's layout holds the y word of column j (origin unchanged) or of
    // column j-1 (origin moved), which this lane has read already.  Only the
    // first column's word waits for the barrier when the origin moved: the
    // lane before reads column first-1's y word in this pass.
    const bool moved = o_row != o_up;
    const Buf wr = buf + (first - o_row);
    int32_t Hp[K];
    int32_t Y = 0, y_first = 0;
    if (cnt > 0) {
      const Buf rd = buf + (first - 1 - o_up);
      int32_t Dn = rd[0].x;
#pragma unroll
      for (int kk = 0; kk < K; ++kk) {
        if (kk >= cnt) break;
        const int2 e = rd[kk + 1];
        const int32_t D = Dn;
        Dn = e.x;
        const uint32_t y = (uint32_t)e.y;
        const int32_t Sb = prmt_s8(rp_lo, rp_hi, (y >> kCodeShift) + 0x5550u);
        const int32_t M = D > 0 ? D + Sb - 128 : 0;
        const int32_t F = (int32_t)(y & kFMask);
        const int32_t Fn = __viaddmax_s32_relu(M, -oe_del, F - e_del);
        const int32_t yn = (int32_t)((y & ~kFMask) | (uint32_t)Fn);
        if (kk > 0 || !moved)
          wr[kk].y = yn;
        else
          y_first = yn;
        Hp[kk] = __vimax3_s32(M, Y, F);
        Y = __viaddmax_s32_relu(M, -oe_ins, Y - e_ins);
      }
    }
    // insertion carry into this lane: max over earlier lanes l' of their
    // carry Y_l' decayed over the (l - 1 - l') * k columns in between
    const int32_t decay = e_ins * kq;
    const int32_t ex = g.excl_max(Y + decay * lane);
    int32_t E = lane == 0 ? 0 : max(0, ex - decay * (lane - 1));
    g.sync();  // every read of the row above is done
    // pass 2: H, the lane's maximum (largest column on ties), dead columns
    int32_t Hl = -1, kl = 0;
    uint32_t dead = 0;
    if (cnt > 0) {
      if (moved) wr[0].y = y_first;
#pragma unroll
      for (int kk = 0; kk < K; ++kk) {
        if (kk >= cnt) break;
        const int32_t H = max(Hp[kk], E);
        E -= e_ins;
        const bool ge = H >= Hl;
        Hl = ge ? H : Hl;
        kl = ge ? kk : kl;
        dead |= H == 0 ? 1u << kk : 0u;
        wr[kk].x = H;
      }
    }
    const int32_t hb = (beg == 0 && i + 1 <= w) ? max(0, h0 - oe_del - e_del * i) : 0;
    if (lane == 0) buf[beg - 1 - o_row] = make_int2(hb, (int32_t)(4u << kCodeShift));
    if (lane == G - 1) buf[end - o_row] = make_int2(0, (int32_t)(q_end << kCodeShift));
    int32_t m, mj;
    g.max_last(Hl, first + kl, &m, &mj);
    g.sync();  // the row is stored
    // end-to-end score when the row reaches the last query column
    if (end == qlen) {
      const int32_t gv = buf[qlen - 1 - o_row].x;
      if (gv >= gscore) {
        gscore = gv;
        gtle = i + 1;
      }
    }
    if (m == 0) break;
    cells += end - beg;
    if (m > best) {
      best = m;
      bi = i;
      bj = mj;
      max_off = max(max_off, abs(mj - i));
    } else if (sc.zdrop > 0) {
      const int64_t di = i - bi, dj = mj - bj;
      const int64_t drop = di > dj ? (int64_t)best - m - (di - dj) * e_del
                                   : (int64_t)best - m - (dj - di) * e_ins;
      if (drop > sc.zdrop) break;
    }
    // the first and the last live column of the row (the row maximum is > 0,
    // so some lane holds one); the dead cells at both ends are dropped
    const uint32_t live = (cnt >= 32 ? 0xffffffffu : (1u << cnt) - 1u) & ~dead;
    int32_t ll = live ? first + 31 - __clz(live) : -1;
    int32_t fl = live ? first + __ffs(live) - 1 : INT_MAX;
    g.all_max_min(&ll, &fl);
    // next row: the columns the live cells reach in one step, within the band
    beg = max(fl, i + 1 - w);
    end = min(min(ll + 2, i + w + 2), qlen);
  }
  if (lane == 0) put_result(a, k, best, bj + 1, bi + 1, gscore, gtle, max_off, XT_OK, cells);
  g.sync();  // the buffer is free for the group's next pair
}

// -------------------------------------------------------- two pairs per lane
// A lane sweeps the rows of its two pairs, one in each 16-bit half of every
// register, in chunks of 8 columns from the first beg to the last end of the
// two; columns outside a pair's own [beg, end) are masked to dead, and chunks
// inside every pair's range of the warp skip the masks.  The row above is in
// shared memory (lane-interleaved: the lanes' chunks differ without bank
// conflicts): H and F of both pairs in one word, a byte each, or in two where a
// score passes 255.  Besides a column's cell update the row keeps its maximum
// with the chunk that holds it and the set of live chunks; the columns are then
// looked up in those chunks.  A warp's pairs have like lengths (the class is
// ordered by length), and a row lasts as long as the widest of them.
//
// Columns before beg need no mask while beg is the row above's first live column:
// all before it are dead there, and a dead neighbourhood gives dead cells.
// Column end of a row, if the query has it, is stored dead (the next row may
// compute it), column -1
// the boundary while the row computes column 0.
//
// Bounded by latency and issue: shared memory holds 10 warps of 128 columns
// per SM (ALU pipe 72% busy) and 3 of 256 (31%), so the classes run side by side.
// Of 500k mixed reads the 185k of 65-128 bases take 1.62 ms and the 78k longer ones
// 2.59 ms, against 3.10 and 3.27 ms on groups.
constexpr int kBwaChunk = 8;

template <bool BYTES>
struct BwaCells;
template <>
struct BwaCells<true> {
  using T = uint32_t;  // H of both pairs, then F
  static __device__ __forceinline__ void get(T v, uint32_t* h, uint32_t* f) {
    *h = prmt(v, 0u, 0x4140u);
    *f = prmt(v, 0u, 0x4342u);
  }
  static __device__ __forceinline__ T put(uint32_t h, uint32_t f) { return prmt(h, f, 0x6420u); }
};
template <>
struct BwaCells<false> {
  using T = uint2;
  static __device__ __forceinline__ void get(T v, uint32_t* h, uint32_t* f) {
    *h = v.x;
    *f = v.y;
  }
  static __device__ __forceinline__ T put(uint32_t h, uint32_t f) { return make_uint2(h, f); }
};

template <int CAP, bool BYTES>
__global__ void __launch_bounds__(32) k_bwa_lane(BwaArgs a, int32_t off, int32_t count, int cls) {
  static_assert(CAP % kBwaChunk == 0 && CAP / kBwaChunk <= 32, "chunk index fits the key");
  using Cells = BwaCells<BYTES>;
  using T = typename Cells::T;
  constexpr int C = kBwaChunk;
  extern __shared__ __align__(16) unsigned char s_lane[];
  T* const col0 = reinterpret_cast<T*>(s_lane) + 32 + threadIdx.x;  // columns -1 .. CAP + 7
  uint32_t* const qn0 =
      reinterpret_cast<uint32_t*>(reinterpret_cast<T*>(s_lane) + 32 * (CAP + C + 1)) + threadIdx.x;
  const int lane = threadIdx.x;
  const BwaScore& sc = a.sc;
  const int32_t oe_ins = sc.o_ins + sc.e_ins, oe_del = sc.o_del + sc.e_del;
  const uint32_t nai = pack16(-oe_ins, -oe_ins), nbi = pack16(-sc.e_ins, -sc.e_ins);
  const uint32_t nad = pack16(-oe_del, -oe_del), nbd = pack16(-sc.e_del, -sc.e_del);
  const uint32_t mcm = 1u << a.mshift;
  const uint32_t nsc = (uint32_t)(uint8_t)sc.nsc, nn = nsc | (kPadScore << 8);
  const uint32_t mism4 = (uint32_t)(uint8_t)sc.mismatch * 0x01010101u, mb = (uint32_t)(uint8_t)sc.match;
  const uint8_t *q_hi = a.q_seq + a.q_bytes, *t_hi = a.t_seq + a.t_bytes;
  const unsigned full = 0xffffffffu;
  for (;;) {
    int32_t base = 0;
    if (lane == 0) base = atomicAdd(&a.heads[cls], 64);
    base = __shfl_sync(full, base, 0);
    if (base >= count) break;
    int32_t kk[2], ql[2], tl[2], h0[2], w[2], beg[2], end[2];
    bool live[2];
    ByteStream ts[2];
    {
      ByteStream qs[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int32_t p = base + 2 * lane + h, idx = off + p;
        int32_t k = p < count && idx >= 0 && idx < a.n ? a.order[idx] : -1;
        if ((uint32_t)k >= (uint32_t)a.n || a.q_len[k] > CAP) k = -1;  // a corrupt workspace: no pair
        kk[h] = k;
        live[h] = k >= 0;
        ql[h] = k >= 0 ? a.q_len[k] : 1;
        tl[h] = k >= 0 ? a.t_len[k] : 0;
        h0[h] = k >= 0 ? a.h0[k] : 1;
        w[h] = bwa_band(sc, ql[h]);
        beg[h] = 0;
        end[h] = min(ql[h], w[h] + 1);
        qs[h].init(a.q_seq, q_hi, a.q_seq + (k >= 0 ? a.q_off[k] : 0));
        ts[h].init(a.t_seq, t_hi, a.t_seq + (k >= 0 ? a.t_off[k] : 0));
      }
      // row -1: the seed before the query, the insertion run from it in the band
      col0[-32] = Cells::put(pack16(h0[0], h0[1]), 0u);
      const int32_t chunks = __reduce_max_sync(full, max(ql[0], ql[1])) / C + 1;
      for (int32_t c = 0; c < chunks; ++c) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          qn0[(2 * c + h) * 32] = nibbles(qs[h].next(a.q_seq, q_hi), ql[h] - C * c);
        for (int32_t j = C * c; j < C * c + C; ++j) {
          int32_t x[2];
#pragma unroll
          for (int h = 0; h < 2; ++h)
            x[h] = j < ql[h] && j + 1 <= w[h] ? max(h0[h] - oe_ins - sc.e_ins * j, 0) : 0;
          col0[j * 32] = Cells::put(pack16(x[0], x[1]), 0u);
        }
      }
    }
    int32_t best[2] = {h0[0], h0[1]}, bi[2] = {-1, -1}, bj[2] = {-1, -1}, max_off[2] = {0, 0};
    int32_t gscore[2] = {-1, -1}, gtle[2] = {0, 0}, cells[2] = {0, 0};
    bool edge[2] = {true, true};   // column -1 may hold the boundary
    bool cut[2] = {false, false};  // the band has cut live columns off before beg
    uint32_t tw[2] = {0, 0};
    for (int32_t i = 0;; ++i) {
      if ((i & 7) == 0)
#pragma unroll
        for (int h = 0; h < 2; ++h) tw[h] = nibbles(ts[h].next(a.t_seq, t_hi), 8);
      bool row[2];
      int32_t b0 = CAP - 1, e0 = -1;
      uint32_t tbl[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        row[h] = live[h] && i < tl[h] && beg[h] < end[h];
        if (row[h]) {
          b0 = min(b0, beg[h]);
          e0 = max(e0, min(end[h], ql[h] - 1));
        }
        const uint32_t tc = tw[h] & 7u, sh = 8u * tc;
        tbl[h] = tc >= 4u ? nsc * 0x01010101u : (mism4 & ~(0xFFu << sh)) | mb << sh;
        tw[h] >>= 4;
      }
      const int32_t c0 = b0 / C;
      const int32_t n_ch = e0 >= 0 ? e0 / C - c0 + 1 : 0;
      const int32_t most = __reduce_max_sync(full, n_ch);
      if (most == 0) break;
      const uint32_t rows2 = (row[0] ? 0xFFFFu : 0u) | (row[1] ? 0xFFFF0000u : 0u);
      uint32_t D, Y = 0, key = 0, live_c[2] = {0, 0}, unused;
      Cells::get(col0[(c0 * C - 1) * 32], &D, &unused);
      for (int32_t cc = 0; cc < most; ++cc) {
        const bool mine = cc < n_ch;
        const int32_t c = mine ? c0 + cc : 0, j0 = c * C;
        T* const p = col0 + j0 * 32;
        uint32_t in[2], Hu[C], Fu[C], s4[2] = {0, 0}, m8 = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          in[h] = row[h] ? bit_range(cut[h] ? beg[h] - j0 : 0, end[h] - 1 - j0, C) : 0u;
        }
        const uint32_t qa = qn0[2 * c * 32], qb = qn0[(2 * c + 1) * 32];
#pragma unroll
        for (int u = 0; u < C; ++u) Cells::get(p[u * 32], &Hu[u], &Fu[u]);
        const bool inside = (!row[0] || in[0] == 0xFFu) && (!row[1] || in[1] == 0xFFu);
        auto column = [&](int u, uint32_t bm) {
          if (u % 4 == 0) {
            s4[0] = prmt(tbl[0], nn, qa >> (u ? 16 : 0));
            s4[1] = prmt(tbl[1], nn, qb >> (u ? 16 : 0));
          }
          constexpr uint32_t kSel[4] = {0xC480u, 0xD591u, 0xE6A2u, 0xF7B3u};
          const uint32_t S = prmt(s4[0], s4[1], kSel[u % 4]);
          const uint32_t M = __viaddmin_s16x2(D, S, D * mcm), F = Fu[u];
          D = Hu[u];
          const uint32_t H = __vimax3_s16x2(M, Y, F) & bm;
          const uint32_t Fn = __viaddmax_s16x2_relu(F, nbd, add16x2(M, nad)) & bm;
          Y = __viaddmax_s16x2_relu(Y, nbi, add16x2(M, nai)) & bm;
          if (mine) p[u * 32] = Cells::put(H, Fn);
          asm("max.s16x2 %0, %0, %1;" : "+r"(m8) : "r"(H));
        };
        if (__all_sync(full, inside || !mine)) {
#pragma unroll
          for (int u = 0; u < C; ++u) column(u, 0xFFFFFFFFu);
        } else {
          const uint32_t in2 = in[0] | in[1] << 16;
#pragma unroll
          for (int u = 0; u < C; ++u) column(u, prmt(in2 << (15 - u), 0u, 0xBB99u));
        }
        m8 = mine ? m8 & rows2 : 0u;
        asm("max.s16x2 %0, %0, %1;" : "+r"(key) : "r"(m8 * 32u + (uint32_t)cc * 0x00010001u));
        if (m8 & 0xFFFFu) live_c[0] |= 1u << cc;
        if (m8 >> 16) live_c[1] |= 1u << cc;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!row[h]) continue;
        auto h_at = [&](int32_t j) -> int32_t {
          uint32_t hh, ff;
          Cells::get(col0[j * 32], &hh, &ff);
          return h ? hi16(hh) : lo16(hh);
        };
        if (end[h] == ql[h]) {
          const int32_t gv = h_at(ql[h] - 1);
          if (gv >= gscore[h]) {
            gscore[h] = gv;
            gtle[h] = i + 1;
          }
        }
        const int32_t kv = h ? hi16(key) : lo16(key), m = kv >> 5;
        if (m == 0) {
          live[h] = false;
          continue;
        }
        cells[h] += end[h] - beg[h];
        const int32_t fc = (c0 + __ffs(live_c[h]) - 1) * C, lc = (c0 + 31 - __clz(live_c[h])) * C;
        int32_t fl = 0, ll = 0;
#pragma unroll
        for (int u = 0; u < C; ++u) {
          if (h_at(fc + C - 1 - u) > 0) fl = C - 1 - u;
          if (h_at(lc + u) > 0) ll = u;
        }
        if (m > best[h] || (sc.zdrop > 0 && best[h] - m > sc.zdrop)) {
          const int32_t mc = (c0 + (kv & 31)) * C;
          int32_t mj = 0;
#pragma unroll
          for (int u = 0; u < C; ++u)
            if (h_at(mc + u) == m) mj = mc + u;
          if (m > best[h]) {
            best[h] = m;
            bi[h] = i;
            bj[h] = mj;
            max_off[h] = max(max_off[h], abs(mj - i));
          } else {
            const int32_t di = i - bi[h], dj = mj - bj[h];
            const int32_t drop =
                best[h] - m - (di > dj ? (di - dj) * sc.e_del : (dj - di) * sc.e_ins);
            if (drop > sc.zdrop) live[h] = false;
          }
        }
        beg[h] = fc + fl;
        if (beg[h] < i + 1 - w[h]) {
          beg[h] = i + 1 - w[h];
          cut[h] = true;
        }
        if (edge[h]) {  // the boundary's H for the next row's column 0
          edge[h] = beg[h] == 0;
          const int32_t hb =
              edge[h] && i + 1 <= w[h] ? max(0, h0[h] - oe_del - sc.e_del * i) : 0;
          uint32_t hh, ff;
          Cells::get(col0[-32], &hh, &ff);
          hh = h ? (hh & 0xFFFFu) | (uint32_t)hb << 16 : (hh & 0xFFFF0000u) | (uint32_t)hb;
          col0[-32] = Cells::put(hh, 0u);
        }
        end[h] = min(min(lc + ll + 2, i + w[h] + 2), ql[h]);
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (kk[h] >= 0)
        put_result(a, kk[h], best[h], bj[h] + 1, bi[h] + 1, gscore[h], gtle[h], max_off[h], XT_OK,
                   cells[h]);
  }
}

// Columns per lane K and lanes per pair G of a class (capacity 64 << class).
template <int C>
struct BwaClass {
  static constexpr int K = kBwaK;
  static constexpr int G = (64 << C) / K;
  static constexpr bool kSeg = G <= 32;
  static constexpr int kPairsPerBlock = kSeg ? kBwaWarpThreads / G : 1;
  static constexpr int kBufElems = G * K + 2;  // per pair
  static constexpr int kThreads = kSeg ? kBwaWarpThreads : G;
  static constexpr size_t kSmem = (size_t)kPairsPerBlock * kBufElems * sizeof(int2);
};

// Six CTAs per SM for the warp-segment classes (at most 80 registers, no
// spills; 6 x 33 KB of row buffers): more warps to cover shared-memory and
// dependency latency.
template <int C>
__global__ void __launch_bounds__(kBwaWarpThreads, 6) k_bwa_seg(BwaArgs a, int32_t off,
                                                                int32_t count, int cls) {
  using Cl = BwaClass<C>;
  constexpr int G = Cl::G;
  __shared__ int2 s_buf[Cl::kPairsPerBlock * Cl::kBufElems];
  Group<G> g;
  g.init();
  // the S groups of a half-warp interleave their buffers (see RowBuf)
  constexpr int S = G <= 8 ? 16 / G : 1;
  static_assert(Cl::kPairsPerBlock % S == 0, "groups of a block fill whole interleaved sets");
  const int gi = threadIdx.x / G;
  const RowBuf<S> buf{s_buf + (gi / S) * S * Cl::kBufElems + gi % S};
  for (;;) {
    const int32_t p = g.claim(&a.heads[cls]);
    if (p >= count) break;
    const int32_t idx = off + p;
    if (idx < 0 || idx >= a.n) break;  // defensive: order index out of range
    const int32_t k = a.order[idx];
    if (k < 0 || k >= a.n) continue;
    bwa_pair<G, Cl::K>(a, g, buf, k);
  }
}

// One pair per CTA; the row buffer in dynamic shared memory.
template <int C>
__global__ void __launch_bounds__(BwaClass<C>::G, 512 / BwaClass<C>::G)
    k_bwa_cta(BwaArgs a, int32_t off, int32_t count) {
  using Cl = BwaClass<C>;
  constexpr int G = Cl::G;
  __shared__ typename Group<G, false>::Shared s;
  extern __shared__ int2 d_buf[];
  Group<G> g;
  g.init(&s);
  for (;;) {
    const int32_t p = g.claim(&a.heads[bwa_group_id(C)]);
    if (p >= count) break;
    const int32_t idx = off + p;
    if (idx < 0 || idx >= a.n) break;
    const int32_t k = a.order[idx];
    if (k < 0 || k >= a.n) continue;
    bwa_pair<G, Cl::K>(a, g, RowBuf<1>{d_buf}, k);
  }
}

template <int C>
cudaError_t launch_class(xt_ctx* ctx, const BwaArgs& a, int32_t off, int32_t count, int cls,
                         cudaStream_t stream) {
  using Cl = BwaClass<C>;
  int& resident = ctx->bwa_blocks[bwa_group_id(C)];
  const size_t dyn = Cl::kSeg ? 0 : Cl::kSmem;
  if (resident == 0) {
    cudaError_t e;
    if constexpr (Cl::kSeg) {
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_bwa_seg<C>, Cl::kThreads, 0);
    } else {
      e = cudaFuncSetAttribute(k_bwa_cta<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)dyn);
      if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k_bwa_cta<C>, Cl::kThreads,
                                                          dyn);
    }
    if (e != cudaSuccess) return e;
    if (resident < 1) resident = 1;
  }
  const int64_t want = ((int64_t)count + Cl::kPairsPerBlock - 1) / Cl::kPairsPerBlock;
  const int grid = (int)std::min<int64_t>(want, (int64_t)resident * ctx->num_sms);
  if constexpr (Cl::kSeg)
    k_bwa_seg<C><<<grid, Cl::kThreads, 0, stream>>>(a, off, count, cls);
  else
    k_bwa_cta<C><<<grid, Cl::kThreads, dyn, stream>>>(a, off, count);
  return cudaGetLastError();
}

template <int C>
cudaError_t launch_lane_class(xt_ctx* ctx, const BwaArgs& a, int32_t off, int32_t count,
                              cudaStream_t stream) {
  constexpr int kCap = bwa_lane_cap(C);
  constexpr bool kBytes = C < kBwaLaneClasses - 1;
  constexpr size_t kSmem = 32 * ((size_t)(kCap + kBwaChunk + 1) * sizeof(typename BwaCells<kBytes>::T) +
                                 (size_t)(kCap / kBwaChunk + 1) * 2 * sizeof(uint32_t));
  auto kern = k_bwa_lane<kCap, kBytes>;
  int& resident = ctx->bwa_blocks[bwa_lane_id(C)];
  if (resident == 0) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, kern, 32, kSmem);
    if (e != cudaSuccess) return e;
    if (resident < 1) resident = 1;
  }
  const int64_t want = ((int64_t)count + 63) / 64;
  const int grid = (int)std::min<int64_t>(want, (int64_t)resident * ctx->num_sms);
  kern<<<grid, 32, kSmem, stream>>>(a, off, count, bwa_lane_id(C));
  return cudaGetLastError();
}

cudaError_t launch_bwa_class(xt_ctx* ctx, const BwaArgs& a, int cls, int32_t off, int32_t count,
                             cudaStream_t stream) {
  switch (cls) {
    case bwa_lane_id(0): return launch_lane_class<0>(ctx, a, off, count, stream);
    case bwa_group_id(0): return launch_class<0>(ctx, a, off, count, cls, stream);
    case bwa_group_id(1): return launch_class<1>(ctx, a, off, count, cls, stream);
    case bwa_group_id(2): return launch_class<2>(ctx, a, off, count, cls, stream);
    case bwa_group_id(3): return launch_class<3>(ctx, a, off, count, cls, stream);
    case bwa_group_id(4): return launch_class<4>(ctx, a, off, count, cls, stream);
    case bwa_group_id(5): return launch_class<5>(ctx, a, off, count, cls, stream);
    case bwa_group_id(6): return launch_class<6>(ctx, a, off, count, cls, stream);
    case bwa_group_id(7): return launch_class<7>(ctx, a, off, count, cls, stream);
    case bwa_lane_id(1):
      return count >= bwa_lane_min(1) ? launch_lane_class<1>(ctx, a, off, count, stream)
                                      : launch_class<1>(ctx, a, off, count, cls, stream);
    case bwa_lane_id(2):
      return count >= bwa_lane_min(2) ? launch_lane_class<2>(ctx, a, off, count, stream)
                                      : launch_class<2>(ctx, a, off, count, cls, stream);
    default: return cudaErrorInvalidValue;
  }
}

bool bwa_scoring_ok(const xt_bwa_scoring* s) {
  if (!s) return false;
  if (s->match < 1 || s->match > 127) return false;
  if (s->mismatch > 0 || s->mismatch < -127) return false;
  if (s->n_score > 0 || s->n_score < -127) return false;
  if (s->o_del < 0 || s->o_del > 1023 || s->o_ins < 0 || s->o_ins > 1023) return false;
  if (s->e_del < 1 || s->e_del > 1023 || s->e_ins < 1 || s->e_ins > 1023) return false;
  if (s->w < 0) return false;
  if (s->end_bonus < 0 || s->end_bonus > (1 << 20)) return false;
  return true;
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace
}  // namespace xt

using namespace xt;

extern "C" xt_status xt_bwa_scoring_check(const xt_bwa_scoring* sc) {
  return bwa_scoring_ok(sc) ? XT_OK : XT_EINVAL;
}

extern "C" xt_status xt_extend_batch_bwa(xt_ctx* ctx, const uint8_t* q_seq, int64_t q_bytes,
                                         const int64_t* q_off, const int32_t* q_len,
                                         const uint8_t* t_seq, int64_t t_bytes,
                                         const int64_t* t_off, const int32_t* t_len,
                                         const int32_t* h0, int32_t n_pairs,
                                         const xt_bwa_scoring* scr, xt_result* out,
                                         int64_t* cells_out, void* stream) {
  if (!ctx) return XT_EINVAL;
  std::lock_guard<std::mutex> lk(ctx->mu);
  if (n_pairs < 0) return ctx_fail(ctx, XT_EINVAL, "n_pairs < 0");
  if (!bwa_scoring_ok(scr)) return ctx_fail(ctx, XT_EINVAL, "scoring record out of range");
  if (q_bytes < 0 || t_bytes < 0) return ctx_fail(ctx, XT_EINVAL, "negative buffer size");
  if (n_pairs > 0 && (!q_off || !q_len || !t_off || !t_len || !h0 || !out))
    return ctx_fail(ctx, XT_EINVAL, "null array");
  if ((q_bytes > 0 && !q_seq) || (t_bytes > 0 && !t_seq))
    return ctx_fail(ctx, XT_EINVAL, "null sequence buffer");
  if (ctx->pending.active) return ctx_fail(ctx, XT_EBUSY, "a begun call has not been finished");
  if (n_pairs == 0) return XT_OK;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e != cudaSuccess) return ctx_cuda_fail(ctx, e, "cudaSetDevice");
  xt_status s = ctx_codes(ctx, &q_seq, &q_bytes, &t_seq, &t_bytes, st);
  if (s != XT_OK) return s;
  // workspace: class bytes, order, counters
  const size_t n = (size_t)n_pairs;
  const size_t o_cls = 0;
  const size_t o_order = align256(o_cls + n);
  const size_t o_slots = align256(o_order + 4 * n);
  // (half as many slots where a budget does not hold them all: lengths in pairs)
  BwaArgs a;
  a.coarse = 0;
  size_t n_ctr = 0;
  for (int coarse = 0; coarse < 2; ++coarse) {
    const std::string last_error = ctx->last_error;
    a.coarse = coarse;
    n_ctr = (size_t)kBwaClasses * (kBwaLenBuckets >> coarse) + 2 * kBwaClasses;
    s = ctx_alloc(ctx, &ctx->bwa_ws, &ctx->bwa_ws_bytes, align256(o_slots + 4 * n_ctr));
    if (s == XT_OK) {
      ctx->last_error = last_error;
      break;
    }
  }
  if (s != XT_OK) return s;
  char* ws = static_cast<char*>(ctx->bwa_ws);
  a.q_seq = q_seq; a.t_seq = t_seq; a.q_off = q_off; a.t_off = t_off; a.q_len = q_len;
  a.t_len = t_len; a.h0 = h0; a.q_bytes = q_bytes; a.t_bytes = t_bytes; a.n = n_pairs;
  a.out = out; a.cells = cells_out;
  a.sc.match = scr->match; a.sc.mismatch = scr->mismatch; a.sc.nsc = scr->n_score;
  a.sc.o_ins = scr->o_ins; a.sc.e_ins = scr->e_ins; a.sc.o_del = scr->o_del;
  a.sc.e_del = scr->e_del;
  // a band wider than any pair changes nothing; clamp so index arithmetic stays in int32
  a.sc.w = scr->w > 2 * XT_MAX_LEN ? 2 * XT_MAX_LEN : scr->w;
  a.sc.zdrop = scr->zdrop; a.sc.end_bonus = scr->end_bonus;
  a.mshift = 0;
  while ((1 << a.mshift) < scr->match + 1) ++a.mshift;
  a.pclass = reinterpret_cast<uint8_t*>(ws + o_cls);
  a.order = reinterpret_cast<int32_t*>(ws + o_order);
  a.slots = reinterpret_cast<int32_t*>(ws + o_slots);
  a.counts = a.slots + kBwaClasses * (kBwaLenBuckets >> a.coarse);
  a.heads = a.counts + kBwaClasses;
  const int threads = 256;
  const int grid = (int)std::min<int64_t>(((int64_t)n_pairs + threads - 1) / threads,
                                          (int64_t)ctx->num_sms * 8);
  e = cudaMemsetAsync(a.slots, 0, 4 * n_ctr, st);
  if (e == cudaSuccess) {
    k_bwa_classify<<<grid, threads, 0, st>>>(a);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) {
    k_bwa_scan<<<1, kBwaScanThreads, 0, st>>>(a);
    e = cudaGetLastError();
  }
  // the class sizes come back to size the launches
  int32_t* cnt_host = ctx->seg_host + kSegHostBwaCounts;
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(cnt_host, a.counts, 4 * kBwaClasses, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaEventRecord(ctx->seg_ev, st);
  if (e == cudaSuccess) e = cudaEventSynchronize(ctx->seg_ev);
  if (e != cudaSuccess) return ctx_cuda_fail(ctx, e, "BWA classify");
  int32_t off[kBwaClasses];
  int32_t total = 0;
  int32_t cnt[kBwaClasses];
  for (int c = 0; c < kBwaClasses; ++c) {
    cnt[c] = cnt_host[c];
    off[c] = total;
    total += cnt[c];
  }
  if (total == 0) return XT_OK;
  k_bwa_scatter<<<grid, threads, 0, st>>>(a);
  e = cudaGetLastError();
  // The classes run side by side on the context's streams, the widest groups and
  // the longest queries first: they hold the longest rows, and what limits one
  // class (shared memory, issue, its last pairs) leaves room for another.
  if (cnt[bwa_lane_id(0)] < bwa_lane_min(0)) {  // its pairs go first in the narrowest groups' launch
    cnt[bwa_group_id(0)] += cnt[bwa_lane_id(0)];
    off[bwa_group_id(0)] = off[bwa_lane_id(0)];
    cnt[bwa_lane_id(0)] = 0;
  }
  int used = 0;
  for (int c = 0; c < kBwaClasses; ++c) used += cnt[c] > 0;
  const int nb = std::min(ctx->branches, used);
  Fork fork(st, ctx->aux, ctx->fork_ev, ctx->join_ev, e == cudaSuccess ? nb : 0);
  if (e == cudaSuccess) e = fork.error();
  int rr = 0;
  auto launch = [&](int c) {
    if (cnt[c] > 0 && e == cudaSuccess)
      e = launch_bwa_class(ctx, a, c, off[c], cnt[c], fork.branch(rr++));
  };
  for (int c = kBwaGroupClasses - 1; c >= 2; --c) launch(bwa_group_id(c));
  for (int c = kBwaLaneClasses - 1; c >= 1; --c) launch(bwa_lane_id(c));
  for (int id : {bwa_group_id(1), bwa_lane_id(0), bwa_group_id(0)}) launch(id);
  const cudaError_t joined = fork.join();
  if (e == cudaSuccess) e = joined;
  if (e != cudaSuccess) return ctx_cuda_fail(ctx, e, "BWA extension");
  ctx->calls++;
  return XT_OK;
}
