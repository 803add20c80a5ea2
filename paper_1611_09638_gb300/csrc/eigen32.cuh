// eigen32.cuh -- the smallest eigenvalue of a node's triad in FP32 with a bound
// on its error, for the screens of FP64 results (it also compiles for the host).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace recon {

constexpr float kU = 5.96046448e-8f;  // 2^-24

// lambda0 of I + h from the closed form, and el >= its error, where every entry
// of I + h is within eps and at most big in magnitude.  Weyl's theorem bounds
// what the entries' errors do (3 eps).  The trace-free part is formed from
// differences of the diagonal, so that its rounding and its trace scale with pp
// and not with the 1 on the diagonal: near a double eigenvalue the angle moves
// by the square root of what r is off, and 2^-8 pp covers that for the some
// 2^-18 r can be off.  (With xx - q instead, q rounded at the size of 1, the
// error reached twice this el at |h| of 1e-3.)  The largest seen here is 0.17 el.
__device__ __forceinline__ float lambda32(float hxx, float hyy, float hzz, float hxy, float hxz, float hyz,
                                          float big, float eps, float& el) {
    constexpr float third = 1.f / 3.f;
    const float q = ((1.f + hxx) + (1.f + hyy) + (1.f + hzz)) * third;
    const float xy = hxx - hyy, xz = hxx - hzz, yz = hyy - hzz;
    const float b1 = (xy + xz) * third, b2 = (yz - xy) * third, b3 = -(xz + yz) * third;
    const float p2 = b1 * b1 + b2 * b2 + b3 * b3 + 2.f * (hxy * hxy + hxz * hxz + hyz * hyz);
    const float pp = sqrtf(p2 * (1.f / 6.f)), ip = 1.f / fmaxf(pp, 1e-30f);
    const float r = 0.5f * ip * ip * ip * (b1 * (b2 * b3 - hyz * hyz) - hxy * (hxy * b3 - hyz * hxz) +
                                          hxz * (hxy * hyz - b2 * hxz));
    el = 3.f * eps + 0.00390625f * pp + 16.f * kU * big;
    return q + 2.f * pp * cosf(acosf(fminf(1.f, fmaxf(-1.f, r))) * third + 2.0943951f);
}

}  // namespace recon
