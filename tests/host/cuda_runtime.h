// Stands in for the CUDA header where a test compiles device helpers for the
// host: the qualifiers and the few intrinsics they use.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cstdlib>

#define __device__
#define __forceinline__ inline

using std::abs;
using std::max;
using std::min;

inline long long __double_as_longlong(double x) {
    long long v;
    memcpy(&v, &x, sizeof v);
    return v;
}
inline int __float_as_int(float x) {
    int v;
    memcpy(&v, &x, sizeof v);
    return v;
}
inline float __int_as_float(int x) {
    float v;
    memcpy(&v, &x, sizeof v);
    return v;
}
inline float __fdividef(float a, float b) { return a / b; }
inline int __float2int_rn(float x) { return (int)lrintf(x); }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
