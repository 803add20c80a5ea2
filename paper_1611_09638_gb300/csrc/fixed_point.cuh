// fixed_point.cuh -- 64-bit fixed-point forms of the FP64 fields.  GB300
// issues two FP64 operations a clock and SM against 64 or more integer ones,
// so stencils of phi and dphi that need more than FP32 run on integers: a
// value is scaled by a power of two 2^Q and rounded; sums and differences of
// such values are exact, also modulo 2^64 where the result is known to fit.
#pragma once

#include <cuda_runtime.h>

namespace recon {

// x 2^Q rounded to nearest (|x| 2^Q < 2^62), from the bits of x.
__device__ __forceinline__ long long to_fixed(double x, int Q) {
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    // |x| = m 2^(e - 1075); m 2^10 shifted right by t = 10 - (e - 1075 + Q)
    const unsigned long long m = e ? (((unsigned long long)b << 10) & 0x3ffffffffffffc00ull) | (1ull << 62) : 0ull;
    const int r = 1085 - Q - e, t = min(max(r, 0), 63);
    const unsigned long long v = r > 63 ? 0ull : (m + ((1ull << t) >> 1)) >> t;
    const long long s = b >> 63;
    return ((long long)v ^ s) - s;
}

// x 2^Q rounded to nearest modulo 2^64, for any finite x.
__device__ __forceinline__ unsigned long long to_fixed_mod(double x, int Q) {
    const long long b = __double_as_longlong(x);
    const int e = (int)(b >> 52) & 0x7ff;
    const unsigned long long m = e ? (((unsigned long long)b << 10) & 0x3ffffffffffffc00ull) | (1ull << 62) : 0ull;
    const int r = 1085 - Q - e, t = min(max(r, 0), 63);
    unsigned long long v = r > 63 ? 0ull : (m + ((1ull << t) >> 1)) >> t;
    // (r < -63 leaves nothing below 2^64: m is a multiple of 2^10)
    if (__builtin_expect(r < 0, 0)) v <<= min(-r, 63);
    const unsigned long long s = (unsigned long long)(b >> 63);
    return (v ^ s) - s;
}

// v 2^n modulo 2^64 for n >= 0, v 2^n rounded for n < 0.
__device__ __forceinline__ long long shift_fixed(long long v, int n) {
    if (n >= 0) return n > 63 ? 0ll : (long long)((unsigned long long)v << n);
    const int r = min(-n, 63);
    return (v >> r) + ((v >> (r - 1)) & 1);
}

// The upper half of v, times unit: an absolute error below one unit besides
// the rounding.
__device__ __forceinline__ float upper_float(long long v, float unit) { return (float)(int)(v >> 32) * unit; }

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }  // -126 <= e <= 127

}  // namespace recon
