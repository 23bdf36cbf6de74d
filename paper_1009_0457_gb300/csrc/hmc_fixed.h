// Integer helpers of the FP64 MPM step's fixed-point sums (k_mpm64.cu), for the host too.
#pragma once

#ifdef __CUDACC__
#define HMC_HD __host__ __device__ __forceinline__
#else
#define HMC_HD inline
#endif

namespace hmc {

// x / 2^n to the nearest, halves away from zero, |x| < 2^63 (the remainder is taken bit by bit: adding
// half a unit first would leave 63 bits)
HMC_HD long long rshift(long long x, int n) {
    if (n <= 0) return x;
    if (n > 63) return 0;
    const long long y = x + (x >> 63);
    return (y >> n) + (y >> (n - 1) & 1);
}

// whether a sum of up to eight integers, whose high words / 8 sum to t, stays below 2^63 in magnitude
HMC_HD bool fits63(int t) { return (unsigned)(t + (1 << 28) - 1) <= (1u << 29) - 9u; }

}  // namespace hmc
