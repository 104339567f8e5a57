// xt_near.cuh -- reading sequences for the kernels that hold a band in
// registers: words of eight bases, base codes as nibbles.
#pragma once
#include <cstdint>

#include "xt_common.cuh"
#include "xt_bounds.cuh"
#include "xt_lane.cuh"

namespace xt {

// Bases of one sequence, eight per step, read as aligned 8-byte words of the
// caller's buffer [lo, hi); a word that is not wholly inside it is put
// together from its bytes that are.
struct ByteStream {
  const uint8_t* at;  // the aligned word after cur
  uint64_t cur;
  int sh;
  __device__ __forceinline__ static uint64_t word(const uint8_t* lo, const uint8_t* hi,
                                                  const uint8_t* p) {
    if (p >= lo && p + 8 <= hi) return __ldg(reinterpret_cast<const unsigned long long*>(p));
    uint64_t v = 0;
    if (p + 8 > lo && p < hi)
      for (int k = 0; k < 8; ++k)
        if (p + k >= lo && p + k < hi) v |= (uint64_t)__ldg(p + k) << (8 * k);
    return v;
  }
  __device__ __forceinline__ void init(const uint8_t* lo, const uint8_t* hi, const uint8_t* p) {
    const uint8_t* a = reinterpret_cast<const uint8_t*>(reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)7);
    sh = (int)(reinterpret_cast<uintptr_t>(p) & 7) * 8;
    cur = word(lo, hi, a);
    at = a + 8;
  }
  // the next eight bytes (those outside the buffer 0)
  __device__ __forceinline__ uint64_t next(const uint8_t* lo, const uint8_t* hi) {
    const uint64_t n = word(lo, hi, at);
    at += 8;
    const uint64_t v = sh ? (cur >> sh) | (n << (64 - sh)) : cur;
    cur = n;
    return v;
  }
};

constexpr uint32_t kPadCode = 5u;  // columns past the query: score kPadScore
constexpr uint32_t kPadScore = 0x80u;

// Eight base codes (bytes) as nibbles, codes above 4 as 4, those at positions
// left.. as kPadCode.
__device__ __forceinline__ uint32_t nibbles(uint64_t v, int32_t left) {
  uint32_t lo = (uint32_t)v, hi = (uint32_t)(v >> 32);
  if (((lo + 0x7B7B7B7Bu) | lo | (hi + 0x7B7B7B7Bu) | hi) & 0x80808080u) {  // some byte above 4
    lo = __vminu4(lo, 0x04040404u);
    hi = __vminu4(hi, 0x04040404u);
  }
  uint32_t w = prmt(lo | (lo >> 4), hi | (hi >> 4), 0x6420u);
  if (left < 8) {
    const uint32_t keep = left <= 0 ? 0u : (1u << (4 * left)) - 1u;
    w = (w & keep) | (0x11111111u * kPadCode & ~keep);
  }
  return w;
}

}  // namespace xt
