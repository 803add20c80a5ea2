// mg_stencil.cuh -- the per-node arithmetic of the FP32 multigrid levels that
// run one kernel per phase (App. A's 7-point operator with face coefficients
// (a + a_nbr)/2 and spacing factors h_a^-2), and the layout of the coarsest
// level's inverse.
#pragma once

#include "recon_internal.cuh"

namespace recon {

// Seven-point operator pieces at a node: diagonal D and off-diagonal sum O,
// so that (L u)_c = O - D u_c.
struct Stencil7 {
    float diag, off;
};

// From the node's coefficient ac and its neighbours' coefficients a* and
// values u* (x: i, y: j, z: k; p: +1, m: -1).
__device__ inline Stencil7 stencil7v(float hx, float hy, float hz, float ac, float axp, float axm, float ayp, float aym, float azp,
                                        float azm, float uxp, float uxm, float uyp, float uym, float uzp, float uzm) {
    const float h = 0.5f;
    float apx = h * (ac + axp) * hx, amx = h * (ac + axm) * hx;
    float apy = h * (ac + ayp) * hy, amy = h * (ac + aym) * hy;
    float apz = h * (ac + azp) * hz, amz = h * (ac + azm) * hz;
    Stencil7 s;
    s.diag = (apx + amx) + (apy + amy) + (apz + amz);
    s.off = (apx * uxp + amx * uxm) + (apy * uyp + amy * uym) + (apz * uzp + amz * uzm);
    return s;
}

// At node c = (i, j, k) of a periodic level stored as one array.
__device__ inline Stencil7 stencil7(const Dims& d, float hx, float hy, float hz, int i, int j, int k, int c,
                                       const float* __restrict__ u, const float* __restrict__ a) {
    const int xp = cell_index(d, i + 1, j, k), xm = cell_index(d, i - 1, j, k);
    const int yp = cell_index(d, i, j + 1, k), ym = cell_index(d, i, j - 1, k);
    const int zp = cell_index(d, i, j, k + 1), zm = cell_index(d, i, j, k - 1);
    return stencil7v(hx, hy, hz, a[c], a[xp], a[xm], a[yp], a[ym], a[zp], a[zm], u[xp], u[xm], u[yp],
                        u[ym], u[zp], u[zm]);
}

// The same pieces from face sums G (face coefficient x 2) of the six faces.
__device__ inline Stencil7 stencil7g(float hx, float hy, float hz, float gpx, float gmx, float gpy, float gmy, float gpz, float gmz,
                                        float uxp, float uxm, float uyp, float uym, float uzp, float uzm) {
    const float h = 0.5f;
    float apx = h * gpx * hx, amx = h * gmx * hx;
    float apy = h * gpy * hy, amy = h * gmy * hy;
    float apz = h * gpz * hz, amz = h * gmz * hz;
    Stencil7 s;
    s.diag = (apx + amx) + (apy + amy) + (apz + amz);
    s.off = (apx * uxp + amx * uxm) + (apy * uyp + amy * uym) + (apz * uzp + amz * uzm);
    return s;
}

// At node c = (i, j, k) of a level: from its nodal coefficient a, or (face)
// from its face sums g (x faces, then y, then z, each d.cells long).
__device__ inline Stencil7 stencil7_any(const Dims& d, float hx, float hy, float hz, int i, int j, int k, int c,
                                           const float* __restrict__ u, const float* __restrict__ a, int face) {
    if (!face) return stencil7(d, hx, hy, hz, i, j, k, c, u, a);
    const int xp = cell_index(d, i + 1, j, k), xm = cell_index(d, i - 1, j, k);
    const int yp = cell_index(d, i, j + 1, k), ym = cell_index(d, i, j - 1, k);
    const int zp = cell_index(d, i, j, k + 1), zm = cell_index(d, i, j, k - 1);
    const float* gx = a;
    const float* gy = a + d.cells;
    const float* gz = a + 2 * (size_t)d.cells;
    return stencil7g(hx, hy, hz, gx[c], gx[xm], gy[c], gy[ym], gz[c], gz[zm], u[xp], u[xm], u[yp], u[ym],
                        u[zp], u[zm]);
}

// The coarsest (4^3) level is solved with the matrix that takes f to the
// mean-free solution of L u = f - mean(f) (kNc x kNc doubles, by rows).
constexpr int kNc = 64;

}  // namespace recon
