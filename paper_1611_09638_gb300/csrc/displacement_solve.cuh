// displacement_solve.cuh -- the node's system of the tracer displacement,
// e U = alpha G in 64-bit fixed point (displacement.cu).  Integer and FP32 work
// only, so that it also compiles for the host.
#pragma once

#include "fixed_point.cuh"

namespace recon {

constexpr int kDispBits = 53;  // fraction bits of a displacement, in cells

using U64 = unsigned long long;

// phi's scale: 2^kPhiBits, modulo 2^64.
constexpr int kPhiBits = 54;

// The scales of a step: dphi 2^Qd and alpha = 2^-kexp.  ok = false where the
// fixed-point form does not apply: alpha is no power of two in [2^-40, 1] (a
// replayed one), some second difference of phi may not be known from its value
// modulo 2^10 cells (wide), or dphi is not finite (sum_dphi) or beyond 2^90.
// max_g: the largest central difference of dphi.  It, and not dphi's own size,
// sets Qd, since only differences of dphi are used.
struct DispScales {
    int Qd, kexp;
    bool ok;
};
__device__ __forceinline__ DispScales disp_scales(double alpha, double max_g, double sum_dphi, bool wide) {
    DispScales s;
    const long long a = __double_as_longlong(alpha), g = __double_as_longlong(max_g);
    const int e = (int)(g >> 52) & 0x7ff, es = (int)(__double_as_longlong(sum_dphi) >> 52) & 0x7ff;
    s.kexp = 1023 - (int)(a >> 52);
    s.Qd = min(120, 1083 - e);  // max_g < 2^(e - 1022), twice that below 2^62
    s.ok = (a & 0xfffffffffffffll) == 0 && a > 0 && s.kexp >= 0 && s.kexp <= 40 && !wide && es < 0x7ff &&
           g >= 0 && e <= 1022 + 90;
    return s;
}

// A column's sums over the planes it is fed: the second differences of phi and
// twice the gradient of dphi at the node one plane back, both modulo 2^64.
struct DispColumn {
    U64 ca, cb, ja, jb, ka, kb, da, db;      // planes p - 2, p - 1: own value, differences in j and k, own dphi
    U64 syb, szb, yzb, gyb, gzb;             // plane p - 1's second differences and gradient
    // f, w: the node's phi and dphi in the plane, rows of `row` values apart;
    // h (xx, yy, zz and four times xy, xz, yz) and g are those of the node before
    __device__ __forceinline__ void feed(const U64* f, const U64* w, int row, long long (&h)[6], long long (&g)[3]) {
        const U64 c = f[0], jp = f[row], jm = f[-row], kp = f[1], km = f[-1], dc = w[0];
        const U64 jd = jp - jm, kd = kp - km;
        h[0] = (long long)(c + ca - 2 * cb), h[1] = (long long)syb, h[2] = (long long)szb;
        h[3] = (long long)(jd - ja), h[4] = (long long)(kd - ka), h[5] = (long long)yzb;
        g[0] = (long long)(dc - da), g[1] = (long long)gyb, g[2] = (long long)gzb;
        syb = jp + jm - 2 * c, szb = kp + km - 2 * c;
        yzb = (f[row + 1] - f[row - 1]) - (f[-row + 1] - f[-row - 1]);
        gyb = w[row] - w[-row], gzb = w[1] - w[-1];
        ca = cb, cb = c, ja = jb, jb = jd, ka = kb, kb = kd, da = db, db = dc;
    }
};

// e U = alpha G from the integer sums: h = second differences (xx, yy, zz) at
// scale 2^kPhiBits and four times the mixed ones (xy, xz, yz), g = twice the
// gradient of dphi at scale 2^Qd.  Returns whether U (scale 2^kDispBits) is within its
// last place or so.
__device__ __forceinline__ bool solve_fixed(const DispScales& sc, const long long (&h)[6],
                                            const long long (&g)[3], long long (&out)[3]) {
    // FP32: e, its inverse X and the right-hand side
    int top = 0;  // every sum below 64 at its scale, or the node is not for integers
#pragma unroll
    for (int q = 0; q < 6; ++q) top = max(top, abs((int)(h[q] >> 32)));
    if (top >= 1 << (kPhiBits - 26)) return false;
    constexpr int low = kPhiBits - 24;  // sums as 32-bit integers at scale 2^24
    const float ue = pow2f(-24);
    const float xx = 1.f + (float)(int)(h[0] >> low) * ue, yy = 1.f + (float)(int)(h[1] >> low) * ue,
                zz = 1.f + (float)(int)(h[2] >> low) * ue;
    const float xy = (float)(int)(h[3] >> low) * (0.25f * ue), xz = (float)(int)(h[4] >> low) * (0.25f * ue),
                yz = (float)(int)(h[5] >> low) * (0.25f * ue);
    float Xxx = yy * zz - yz * yz, Xyy = xx * zz - xz * xz, Xzz = xx * yy - xy * xy;
    float Xxy = xz * yz - xy * zz, Xxz = xy * yz - yy * xz, Xyz = xy * xz - xx * yz;
    const float rdet = __fdividef(1.f, xx * Xxx + xy * Xxy + xz * Xxz);
    Xxx *= rdet, Xyy *= rdet, Xzz *= rdet, Xxy *= rdet, Xxz *= rdet, Xyz *= rdet;
    const float emax = fmaxf(fmaxf(fabsf(xx), fabsf(yy)), fmaxf(fabsf(zz), fmaxf(fabsf(xy), fmaxf(fabsf(xz), fabsf(yz)))));
    float ug = pow2f(max(31 - sc.Qd - sc.kexp, -126));
    float g0 = upper_float(g[0], ug), g1 = upper_float(g[1], ug), g2 = upper_float(g[2], ug);
    float gm = fmaxf(fabsf(g0), fmaxf(fabsf(g1), fabsf(g2)));
    if (gm < 1048576.f * ug) {
        // far below the field's largest gradient, which set the scale: brought to
        // 62 bits first, or the first piece would have too few of them
        const U64 any = (U64)(g[0] ^ (g[0] >> 63)) | (U64)(g[1] ^ (g[1] >> 63)) | (U64)(g[2] ^ (g[2] >> 63));
        const int sh = max(__clzll((long long)any) - 2, 0);
        ug = pow2f(max(31 - sc.Qd - sc.kexp - sh, -126));
        g0 = upper_float((long long)((U64)g[0] << sh), ug), g1 = upper_float((long long)((U64)g[1] << sh), ug),
        g2 = upper_float((long long)((U64)g[2] << sh), ug);
        gm = fmaxf(fabsf(g0), fmaxf(fabsf(g1), fabsf(g2)));
    }
    // integers: e at scale 2^54
    const U64 Exx = (U64)h[0] + (1ull << kPhiBits), Eyy = (U64)h[1] + (1ull << kPhiBits),
              Ezz = (U64)h[2] + (1ull << kPhiBits);
    auto mixed = [&](long long v) { return (U64)((v + 2) >> 2); };
    const U64 Exy = mixed(h[3]), Exz = mixed(h[4]), Eyz = mixed(h[5]);
    float u0, u1, u2, um;  // a piece and its largest magnitude
    auto piece = [&](float r0, float r1, float r2) {
        u0 = Xxx * r0 + Xxy * r1 + Xxz * r2;
        u1 = Xxy * r0 + Xyy * r1 + Xyz * r2;
        u2 = Xxz * r0 + Xyz * r1 + Xzz * r2;
        um = fmaxf(fabsf(u0), fmaxf(fabsf(u1), fabsf(u2)));
    };
    piece(g0, g1, g2);
    // The residual of a piece must fit 62 bits: the error of X is about
    // 2^-22 |e|^2 / det; where that is more, smaller pieces.
    const float crit = emax * emax * emax * fabsf(rdet) * __fdividef(gm, fmaxf(um, 1e-30f));
    if (!(um < 32.f && crit < 3e5f)) return false;
    const int bits = 17 - max(((__float_as_int(crit) >> 23) & 255) - 127 - 9, 0);
    // U = D 2^-s in pieces of at most bits + 1 bits, the last at 2^-57
    auto scale_of = [&] { return min(bits - (((__float_as_int(um) >> 23) & 255) - 127), 57); };
    int s = scale_of();
    long long a0 = __float2int_rn(u0 * pow2f(s)), a1 = __float2int_rn(u1 * pow2f(s)), a2 = __float2int_rn(u2 * pow2f(s));
    U64 D0 = a0, D1 = a1, D2 = a2;
    float last = um, err = um;
    constexpr float done = 7e-18f;  // 2^-57 cells
    if (err >= done) {
        const int n = 53 + s - sc.Qd - sc.kexp;
        U64 R0 = shift_fixed(g[0], n), R1 = shift_fixed(g[1], n), R2 = shift_fixed(g[2], n);
#pragma unroll 1
        for (int it = 0; it < 7; ++it) {
            // residual alpha G - e U at scale 2^(54 + s)
            R0 -= Exx * (U64)a0 + Exy * (U64)a1 + Exz * (U64)a2;
            R1 -= Exy * (U64)a0 + Eyy * (U64)a1 + Eyz * (U64)a2;
            R2 -= Exz * (U64)a0 + Eyz * (U64)a1 + Ezz * (U64)a2;
            const float ur = pow2f(-22 - s);
            const U64 half = 1ull << 31;
            piece(upper_float(R0 + half, ur), upper_float(R1 + half, ur), upper_float(R2 + half, ur));
            // (22 bits at most: what the upper halves show of the residual)
            const int ns = min(max(scale_of(), s), s + 22), m = ns - s;
            s = ns;
            const float sc2 = pow2f(s);
            a0 = __float2int_rn(u0 * sc2), a1 = __float2int_rn(u1 * sc2), a2 = __float2int_rn(u2 * sc2);
            D0 = (D0 << m) + a0, D1 = (D1 << m) + a1, D2 = (D2 << m) + a2;
            // what remains: the piece's rounding, X's error as the last two
            // pieces show it, or the residual's rounding (half a unit of each
            // upper half, through X)
            err = fmaxf(pow2f(-1 - s), um * __fdividef(um, last));
            if (err < done) {
                err = fmaxf(fmaxf(fmaxf(fabsf(Xxx), fabsf(Xyy)), fmaxf(fabsf(Xzz), fabsf(Xxy))), fmaxf(fabsf(Xxz), fabsf(Xyz))) *
                      (1.5f * ur);
                if (err < done) break;
            }
            if (!(um < 0.25f * last)) return false;
            last = fmaxf(um, ur);  // (a residual of no unit: its rounding may show next)
            R0 <<= m, R1 <<= m, R2 <<= m;
        }
    }
    // 2^-53 cells; the pieces end at 2^-57 (at 2^-56 with err at its bound)
    const int n = s - kDispBits;
    auto place = [&](U64 v) { return n > 0 ? ((long long)(v + (1ull << (n - 1)))) >> n : (long long)(v << -n); };
    out[0] = place(D0), out[1] = place(D1), out[2] = place(D2);
    return err < done;
}

}  // namespace recon
