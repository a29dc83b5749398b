// echo_slowdown_int.h -- rint(fl(d * factor)) in integers, for durations below 2^31 and
// factors in [1, 2): the values and both roundings (to 53 bits, then to an integer, ties to
// even each time) of the fp64 expression, bit for bit.  No CUDA dependency of its own, so
// the same function is compiled for the host and tested there.
//
// What it is for: the part does 527 G fp64 operations/s, and the expression needs three (a
// conversion, a product, a conversion back), so 190 G slowed durations/s at most; this takes
// about 20 integer instructions, which run beside everything else at 10 times that rate.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define ECHO_SD_HD __host__ __device__ __forceinline__
#else
#define ECHO_SD_HD inline
#endif

namespace echo {

// whether slowed_int applies: 0 <= d < 2^31, factor (its bits) in [1, 2)
ECHO_SD_HD bool slowed_int_ok(int64_t d, uint64_t factor_bits) {
  return (uint64_t)d < (1ull << 31) && (factor_bits >> 52) == 1023;
}

// factor = m / 2^52 with the 53-bit integer m, so x = d * factor = d * m / 2^52 exactly:
// integer part i (at most 32 bits), fraction f / 2^52.  fl(x) keeps 53 bits, so of the
// fraction it drops as many as i has beyond its first: rounding moves f by at most
// t = 2^(bits of i - 2).  Hence fl(x) lies on the half exactly when f is within t of it
// (both ends included: their ties go to the half, whose last kept bit is 0), below it when
// f is smaller and above it when f is larger; and rint of that is i, i + 1, or on the half
// the even one of them.
ECHO_SD_HD int64_t slowed_int(int64_t d, uint64_t factor_bits) {
  const uint64_t m = (factor_bits & ((1ull << 52) - 1)) | (1ull << 52);
  const uint64_t lo = (uint64_t)(uint32_t)d * (uint32_t)m;
  const uint64_t hi = (uint64_t)(uint32_t)d * (uint32_t)(m >> 32) + (lo >> 32);  // x * 2^20, rounded down
  const uint32_t i = (uint32_t)(hi >> 20);
  const uint64_t f = ((hi & 0xFFFFFu) << 32) | (uint32_t)lo;
#if defined(__CUDA_ARCH__)
  const int bits = 32 - __clz((int)i);
#else
  const int bits = i ? 32 - __builtin_clz(i) : 0;
#endif
  const uint64_t half = 1ull << 51, t = (1ull << bits) >> 2;  // (0 for i < 2: nothing is dropped)
  const bool up = f > half + t || (f >= half - t && (i & 1));
  return (int64_t)((uint64_t)i + up);
}

}  // namespace echo
