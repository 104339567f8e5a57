// xt_kernels.cuh -- kernel declarations and launch-plan types shared by the
// host API and the kernel translation units.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "xt_common.cuh"

namespace xt {

// Pair classes after classify.
//   PACKED: two strips in the 16-bit halves of each register (one-lane engine)
//   NARROW: 32-bit, row key H*65536 + j (h0 + match*min(qlen,tlen) <= 32767)
//   WIDE:   32-bit with an explicit (max, column) pair per row
//   HUGE:   band ring too large for shared memory (global slab per group)
//   NEAR:   PACKED pairs that k_near tries on a narrow band first
//   BAND:   NARROW pairs whose scores fit 16 bits under the anchoring
//           multiplier, where the band engine holds the band or a narrower one
enum PairClass : uint8_t {
  CLS_PACKED = 0, CLS_NARROW = 1, CLS_WIDE = 2, CLS_HUGE = 3, CLS_NEAR = 4, CLS_BAND = 5,
  CLS_DONE = 6
};
constexpr int kNumClasses = 6;           // classes that need a DP kernel
// The segments of BAND pairs left to lanes: the buckets of CLS_NEAR it has no pairs in.
constexpr int kLanesLeftSeg = CLS_NEAR;
constexpr uint8_t kRest = 0xFF;          // seen by k_diag, class still to be found
constexpr bool packed_class(int cls) { return cls == CLS_PACKED || cls == CLS_NEAR; }
// per-bucket flags (Work::jflags)
constexpr uint8_t kJHuge = 1;            // bucket's pairs go to the HUGE class
constexpr uint8_t kJPacked = 2;          // bucket runs the one-lane engine: packed pairs allowed
constexpr uint8_t kJHugeWide = 4;        // the bucket's WIDE pairs (group engine only) are HUGE
constexpr uint8_t kJTag4 = 8;            // packed row keys of the bucket carry 4-bit step tags
constexpr uint8_t kJBand = 16;           // bucket's NARROW pairs may go to the BAND class
// Step-tag bits of the packed row keys (H * 2^bits + step in 16 bits) in
// bucket j: 6 (H <= 511) up to queries of 510 bases, 4 (H <= 2047, folded
// every 16 steps) beyond, where a pair's score bound grows past 511.
constexpr int kTag4J = 10;
constexpr int packed_tag_bits(int j) { return j >= kTag4J ? 4 : 6; }
// Calls of at least this many pairs pack those buckets' pairs (kJTag4): only
// then are there enough of them to run one lane per pair; in smaller calls
// they go to lane groups, which run them in 32-bit anyway (c5-mix calls:
// 800k pairs 16.43 -> 16.00 ms, 4M 68.1 -> 58.8 ms; 400k 9.76 -> 11.90 ms had
// they been packed: a second group launch waited for the first).
constexpr int32_t kTag4MinPairs = 1 << 19;
constexpr int kJMin = 5;                 // length buckets j: qlen + 2 <= 2^j
constexpr int kJMax = 21;
constexpr int kNumJ = kJMax + 1;
// Bins the queue is ordered by, within a class: one per exact query length in
// the buckets up to kExactJ, kLongSub of equal width in each longer one (bins
// of 1.6% of the length; a one-block scan reads them all in every call).
constexpr int kExactJ = 9;
constexpr int kLongSub = 64;
constexpr int kExactBins = 1 << kExactJ;
constexpr int kClassBins = kExactBins + kLongSub * (kJMax - kExactJ);
// buckets (queries of 511 bases and longer) the band engine tries on a narrow
// band where the whole band is too wide for it
constexpr int kBandNearJMin = 10;
constexpr int kNumBuckets = kNumClasses * kClassBins;
// Calls of fewer pairs skip the near passes: their time is launches and one
// pair's latency, which the passes add to (1,000 pairs of 100 bases 147 ->
// 223 us; 5,000 of 64 bases 180 -> 164 us).
constexpr int32_t kNearMinPairs = 4096;
// k_near's narrow band: diagonals |i - j| <= kNearHalf; queries it takes, and
// the calls' scoring it holds for (see xt_bounds.cuh)
constexpr int kNearHalf = 15;
constexpr int kNearJMax = 9;
constexpr int kNearMaxQ = (1 << kNearJMax) - 2;
static_assert(kNearJMax <= kExactJ, "one bin per length");
static_assert(kNearJMax < kBandNearJMin, "kLanesLeftSeg's buckets are free");
constexpr int kNearBins = 1 << kNearJMax;
constexpr int kQueueThreads = 128;       // threads per CTA of the queue kernels
// Queue-kernel launches per call (heads), at most one a bucket and class: WIDE pairs
// in every bucket, PACKED and NARROW ones up to 65,535 bases, NEAR ones up to
// kNearMaxQ, BAND ones up to 65,535 bases (where a narrow band comes first, at 511
// and longer, up to three launches each), HUGE ones and the near pass one each.
constexpr int kShortJMax = 17;           // bucket of 65,535-base queries
constexpr int kBandLaunches = 3;
constexpr int kMaxLaunches = 80;
static_assert((kJMax - kJMin + 1) + 2 * (kShortJMax - kJMin + 1) + (kNearJMax - kJMin + 1) +
                      (kShortJMax - kJMin + 1 > kBandLaunches * (kShortJMax - kBandNearJMin + 1)
                           ? kShortJMax - kJMin + 1
                           : kBandLaunches * (kShortJMax - kBandNearJMin + 1)) + 2 <= kMaxLaunches,
              "a head for every launch");

// Device workspace of one call (carved from the context's pool).
struct Work {
  uint8_t* pclass;      // [n]
  int32_t* order;       // [n] pairs grouped by (class, bucket desc, sub desc)
  int32_t* counts;      // [kNumBuckets]
  int32_t* cursor;      // [kNumBuckets]
  int32_t* seg_begin;   // [kNumClasses * kNumJ]
  int32_t* seg_end;     // [kNumClasses * kNumJ]
  int32_t* near_hope;   // [1] NEAR pairs whose diagonal promises that k_near settles them
  int32_t* heads;       // [kMaxLaunches]
  int32_t* near_left;   // [kNearBins] pairs k_near left, per exact length
  int32_t* near_tmp;    // [n] those pairs, each length's run where its queue run was; or 1 at
                        // the places in the queue of the pairs a narrow band left
};

constexpr int kLaneThreads = 128;        // threads per CTA of the one-lane kernels
constexpr int kLaneStageJMax = 9;        // one-lane kernels stage queries up to 2^9 - 2 bases

// One persistent launch: pairs of class cls, buckets [j_lo, j_hi].  Every
// field has a default, so a launch built field by field never carries stack
// contents into the dispatch.
struct Launch {
  int cls = 0, j_lo = 0, j_hi = 0;
  bool lane = false;         // one-lane engine (k_lane) instead of the group engine (k_queue)
  bool band = false;         // band engine (k_band): P lanes of R slots
  int near_hw = 0;           // > 0: on a narrower band of this half width
  int cls2 = -1;             // one-lane engine: then this class's pairs of the same buckets
  bool after_prev = false;   // takes the pairs the launch before it left, on its stream
  // a narrow band launch: from so many pairs left on they go to lanes (0: never), which
  // only the device knows; and the one-lane launch that takes them then
  int32_t lanes_from = 0;
  bool lanes_left = false;
  int P = 1, R = 8;          // lanes per pair, rows per lane-strip (per half when packed)
  int rs_log2 = 0;           // ring entries per group = 1 << rs_log2
  bool global_ring = false;  // ring in a global slab per group instead of shared memory
  int64_t slab = 0;          // entries per global slab (power of two)
  int grid = 0;              // CTAs
  int mparam = 0;            // one-lane engine: match + 1 (32-bit) or shift k (packed)
  size_t pool_off = 0;       // global ring: byte offset of the launch's slabs in the pool
};

// Host-side launchers (defined in xt_kernels.cu); all enqueue on `stream`.
// Per-bucket flags (kJHuge | kJPacked), passed to classify by value.
struct JFlags {
  uint8_t f[kNumJ];
};
// Kernels read the batch arguments from a device copy (bd) so that one
// captured graph serves every call; n_cap sizes the per-pair grids (>= n).
// after_diag: launch_diag ran before on the same stream (w.pclass holds its marks).
cudaError_t launch_classify(const Batch* bd, int32_t n_cap, const Score& sc, int32_t match,
                            const JFlags& jf, bool after_diag, const Work& w, cudaStream_t stream);
// Settle the pairs whose diagonal alone decides; mark the others for classify
// (near: CLS_NEAR where k_near may settle them).
cudaError_t launch_diag(const Batch* bd, int32_t n_cap, const Score& sc, int32_t match, bool near,
                        const Work& w, cudaStream_t stream);
// The NEAR class on its narrow band; its segment table and queue region then
// hold the pairs left, longest first.
int near_grid(int32_t pairs, int num_sms);
// Grids of these passes and of the band engine are rounded up, so that calls of like
// size share a graph, to four sizes an octave: CTAs without a pair end at once, but
// many of them cost the launches beside them room (55k streamed pairs 1,068 -> 1,084 us
// with 128 CTAs of k_near for 82).
// Nor does the rounding pass a whole number of CTAs per SM: the spare ones would take
// the place of others (5,000 tables of 180 bases, 286 CTAs of k_band in 304 / 320: 267,
// 320 us).
inline int rounded_grid(int64_t want, int num_sms, int per_sm) {
  if (want < 1) return 0;
  int64_t step = 1;
  while (8 * step < want) step *= 2;
  const int64_t grid = (want + step - 1) / step * step;
  const int64_t whole = (want + num_sms - 1) / num_sms * num_sms;
  const int64_t most = (int64_t)num_sms * per_sm;
  return (int)(grid < whole ? (grid < most ? grid : most) : (whole < most ? whole : most));
}
cudaError_t launch_near(const Batch* bd, const Score& sc, int32_t match, int grid, const Work& w,
                        int head_id, cudaStream_t stream);
cudaError_t launch_order(const Batch* bd, int32_t n_cap, const Work& w, cudaStream_t stream);
cudaError_t launch_queue(const Batch* bd, const Score& sc, const Work& w, const Launch& L,
                         int head_id, int2* gring, cudaStream_t stream);
cudaError_t launch_plain(const Batch* bd, int32_t n_cap, const Score& sc, const Work& w,
                         int rs_log2, cudaStream_t stream);
cudaError_t launch_lane(const Batch* bd, const Score& sc, const Work& w, const Launch& L,
                        int head_id, void* gring, cudaStream_t stream);
// The band engine's lanes per pair and slots per lane for a scoring and a
// launch of so many pairs; false where it does not hold the band or the
// scoring's row keys.
bool band_shape(const Score& sc, int32_t match, int32_t pairs, int* P, int* K);
// The narrow band (half width hw) for bucket j's pairs of a wider band.
bool band_near_shape(const Score& sc, int32_t match, int j, int* P, int* K, int* hw);
int band_grid(int P, int K, int32_t pairs, int num_sms);
cudaError_t launch_band(const Batch* bd, const Score& sc, int32_t match, const Work& w,
                        const Launch& L, int head_id, int num_sms, cudaStream_t stream);
// ASCII letters to base codes (A/C/G/T either case -> 0..3, else 4), n bytes.
cudaError_t launch_ascii_codes(const uint8_t* in, uint8_t* out, int64_t n, int num_sms,
                               cudaStream_t stream);
// 4-bit codes, two per byte, to one code per byte: bytes [b0, b1) of `in`
// become bytes [2 b0, 2 b1) of `out`.
cudaError_t launch_unpack4(const uint8_t* in, uint8_t* out, int64_t b0, int64_t b1, int num_sms,
                           cudaStream_t stream);
// Both-direction extension of seeds: device workspace (carved by the host).
struct SeedWork {
  int32_t *lq_len, *lt_len;   // left (reversed prefix) lengths, -1: invalid seed
  int64_t *lq_off, *lt_off;   // their offsets in rev_q / rev_t
  int32_t *rq_len, *rt_len;   // right (suffix) lengths, -1: invalid seed
  int64_t *rq_off, *rt_off;   // their offsets in the caller's buffers
  int32_t* rh0;               // right side's seed score
  int64_t *block_q, *block_t; // per-block sums of the left lengths
  int64_t* totals;            // [2]: bytes of rev_q and rev_t
  uint8_t *rev_q, *rev_t;     // reversed prefixes
};
// Prep, lengths, and the scan up to the totals (sw.totals, read by the host).
cudaError_t launch_seed_front(int32_t n, const int32_t* q_len, const int32_t* t_len,
                              const int64_t* q_off, const int64_t* t_off, int64_t q_bytes,
                              int64_t t_bytes, const int32_t* q_beg, const int32_t* t_beg,
                              const int32_t* seed_len, const SeedWork& sw, cudaStream_t stream);
// Offsets of the reversed prefixes and the reversed copies (sw.rev_q/rev_t set).
cudaError_t launch_seed_reverse(int32_t n, const uint8_t* q_seq, const int64_t* q_off,
                                const uint8_t* t_seq, const int64_t* t_off, const SeedWork& sw,
                                cudaStream_t stream);
// Right side's seed scores from the left results.
cudaError_t launch_seed_right_h0(int32_t n, const int32_t* h0, const xt_result* left,
                                 const SeedWork& sw, cudaStream_t stream);
// Shared memory a queue launch needs per CTA (bytes).
size_t queue_smem_bytes(int P, int rs_log2);
// Ring bytes per lane of a one-lane launch (per CTA in shared memory: x kLaneThreads).
size_t lane_ring_bytes(int cls, int rs_log2);
// Query staging bytes per CTA of a one-lane launch whose longest bucket is j_hi (0: none).
size_t lane_stage_bytes(int j_hi);
// Ring-feed slot bytes per CTA of a one-lane launch (global rings of 32-bit pairs).
size_t lane_pipe_bytes(int cls, bool global_ring);
int max_smem_per_block_optin(int device);

__device__ __forceinline__ int ceil_log2(uint32_t x) {  // x >= 1
  return x <= 1 ? 0 : 32 - __clz(x - 1);
}

// Length bucket j of a query: qlen + 2 <= 2^j, at least kJMin.
__device__ __forceinline__ int bucket_of(int32_t ql) {
  const int j = ceil_log2((uint32_t)ql + 2u);
  return j < kJMin ? kJMin : j;
}

// Bin of a query length: bucket j <= kExactJ is the bins 2^(j-1) .. 2^j - 1
// (kJMin: from 0), one per length; the buckets after it kLongSub bins each.
__device__ __forceinline__ int bin_of_len(int32_t ql) {
  if (ql + 2 <= kExactBins) return ql + 1;
  const int j = bucket_of(ql);
  const int sub = (ql + 1 - (1 << (j - 1))) >> (j - 7);  // 2^(j-1) lengths, 64 bins
  return kExactBins + (j - kExactJ - 1) * kLongSub + (sub < kLongSub ? sub : kLongSub - 1);
}
static_assert(kLongSub == 64, "bin_of_len's shift");

// Bucket of a bin, and whether the bin is its bucket's longest or shortest.
__device__ __forceinline__ int bucket_of_bin(int bin) {
  if (bin >= kExactBins) return kExactJ + 1 + (bin - kExactBins) / kLongSub;
  const int j = 32 - __clz(bin);
  return j < kJMin ? kJMin : j;
}
__device__ __forceinline__ bool longest_bin(int bin) {
  return bin >= kExactBins ? bin % kLongSub == kLongSub - 1
                           : bin == (1 << bucket_of_bin(bin)) - 1;
}
__device__ __forceinline__ bool shortest_bin(int bin) {
  if (bin >= kExactBins) return bin % kLongSub == 0;
  return bin == 0 || (bin >= 1 << kJMin && (bin & (bin - 1)) == 0);
}

}  // namespace xt
