// quot_range.cuh -- the integer parts of the FP64 quotient (sslbm_internal.cuh, force_quot): which
// divisors take the float-seeded reciprocal, and the change of format.  Unsigned arithmetic, which
// wraps: a divisor of -0 or a small negative one has the most negative high words there are.
#pragma once
#ifdef __CUDACC__
#define SSLBM_HD __host__ __device__ __forceinline__
#else
#define SSLBM_HD inline
#endif

namespace sslbm {

// The high word of a double in [2^-99, 2^99): sign clear, exponent in range (NaN, infinities, zeros and
// negative values fail it).
SSLBM_HD bool quot_in_range(int hi) {
  return (unsigned)hi - ((1023u - 99u) << 20) < (198u << 20);
}
// High and low word of the double with the value of the float whose bits are rb (normal, positive).
SSLBM_HD int quot_hi(int rb) { return (int)(((unsigned)rb >> 3) + ((1023u - 127u) << 20)); }
SSLBM_HD int quot_lo(int rb) { return (int)((unsigned)rb << 29); }

}  // namespace sslbm
