// Order of float64 numbers on the integer pipe: minima by their bits instead of by float64 comparisons
// (each of which holds a quarter of an SM for 64 cycles a warp).  Plain C++, host and device.
#pragma once

#ifdef __CUDACC__
#define IPM_HD __host__ __device__ __forceinline__
#else
#define IPM_HD inline
#endif

namespace ipmk {

constexpr long long kInfBits = 0x7ff0000000000000ll;   // INFINITY's bits

// A key whose order as a signed integer is the numbers' order (-0 just below +0): the bits of a number
// with its sign bit clear, the others reversed below them.  NaN of either sign gives INFINITY's key,
// so that a minimum passes it over as fmin does.
IPM_HD long long min_key(long long bits) {
  if ((bits & 0x7fffffffffffffffll) > kInfBits) return kInfBits;
  return bits ^ ((bits >> 63) & 0x7fffffffffffffffll);
}

// The bits of the number a key stands for.
IPM_HD long long min_key_bits(long long key) { return key ^ ((key >> 63) & 0x7fffffffffffffffll); }

}  // namespace ipmk
