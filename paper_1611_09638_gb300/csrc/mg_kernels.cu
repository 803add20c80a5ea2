// mg_kernels.cu -- variable-coefficient multigrid kernels for the linearised
// elliptic equation of App. A (Eq. elliptic with x ~ xi):
//     L u = sum_a h_a^-2 [A+ (u+ - u) - A- (u - u-)],  A+- = (a + a+-) / 2,
// red-black Gauss-Seidel smoothing (red = (i+j+k) even first), residual,
// full-weighting restriction, trilinear prolongation, and a dense solve of the
// 4^3 coarsest level with the mean constraint, for the FP32 levels (mixed mode)
// and the FP64 ones.
#include "mg_stencil.cuh"
#include "recon_internal.cuh"
#include "reduce.cuh"

namespace recon {

namespace {

constexpr int kThreads = 256;

inline int nblocks(long long work) { return (int)((work + kThreads - 1) / kThreads); }

// One colour of a red-black Gauss-Seidel sweep; thread t owns the t-th node
// of that colour (nodes of a colour alternate along the fastest axis).
__global__ void k_rbgs_colour(Dims d, float hx, float hy, float hz, int colour, float* __restrict__ u,
                              const float* __restrict__ f, const float* __restrict__ a, int face) {
    const int half = d.cells >> 1;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= half) return;
    const int hs2 = d.s2 - 1;
    const int kk = t & ((1 << hs2) - 1);
    const int j = (t >> hs2) & (d.n1 - 1);
    const int i = t >> (d.s1 + hs2);
    const int k = 2 * kk + ((i + j + colour) & 1);
    const int c = cell_index(d, i, j, k);
    Stencil7 s = stencil7_any(d, hx, hy, hz, i, j, k, c, u, a, face);
    u[c] = (s.off - f[c]) / s.diag;
}

// One colour of a red-black sweep of an FP64 level from its stored face
// coefficients A = h^-2 (a_c + a_n) / 2 (F: +x, +y, +z face of each node) and
// the inverse of the node's diagonal D = sum of its six A:
// u_c = (sum_n A_n u_n - f_c) / D_c in 8 FP64 instructions per node, since
// FP64 issue (2 lanes a clock and SM), not memory, bounds this sweep on GB300:
// 18.3 us a colour of 128^3 against 13.6 us of issue.  Forming the faces and
// dividing in each sweep took some 45 instructions, 14 us a colour of 64^3.
// zero: u is 0 on entry and is not read (the red colour of a first sweep; the
// black one reads red values only, so u need not be cleared).
__global__ void k_rbgs_colour64(Dims d, int colour, int zero, double* __restrict__ u,
                                const double* __restrict__ f, const double* __restrict__ F,
                                const double* __restrict__ inv_d) {
    const int half = d.cells >> 1;
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= half) return;
    const int hs2 = d.s2 - 1;
    const int kk = t & ((1 << hs2) - 1);
    const int j = (t >> hs2) & (d.n1 - 1);
    const int i = t >> (d.s1 + hs2);
    const int k = 2 * kk + ((i + j + colour) & 1);
    const int c = cell_index(d, i, j, k);
    if (zero) {
        u[c] = -f[c] * inv_d[c];
        return;
    }
    const int n0 = cell_index(d, i + 1, j, k), n1 = cell_index(d, i - 1, j, k);
    const int n2 = cell_index(d, i, j + 1, k), n3 = cell_index(d, i, j - 1, k);
    const int n4 = cell_index(d, i, j, k + 1), n5 = cell_index(d, i, j, k - 1);
    const size_t n = (size_t)d.cells;
    double o = F[c] * u[n0];
    o = fma(F[n1], u[n1], o);
    o = fma(F[n + c], u[n2], o);
    o = fma(F[n + n3], u[n3], o);
    o = fma(F[2 * n + c], u[n4], o);
    o = fma(F[2 * n + n5], u[n5], o);
    u[c] = (o - f[c]) * inv_d[c];
}

// r = f - L u of an FP64 level, from the same coefficients, for the
// restriction: 7 FMAs a node.  Restricting a stored residual instead of
// evaluating it at the 27 fine nodes of every coarse node (each evaluation
// with its faces) takes this step at 128^3 from 280 to 45 us.
__global__ void k_residual64(Dims d, const double* __restrict__ u, const double* __restrict__ f,
                             const double* __restrict__ F, const double* __restrict__ D,
                             double* __restrict__ r) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const size_t n = (size_t)d.cells;
    const int n1 = cell_index(d, i - 1, j, k), n3 = cell_index(d, i, j - 1, k), n5 = cell_index(d, i, j, k - 1);
    double v = fma(D[c], u[c], f[c]);
    v = fma(-F[c], u[cell_index(d, i + 1, j, k)], v);
    v = fma(-F[n1], u[n1], v);
    v = fma(-F[n + c], u[cell_index(d, i, j + 1, k)], v);
    v = fma(-F[n + n3], u[n3], v);
    v = fma(-F[2 * n + c], u[cell_index(d, i, j, k + 1)], v);
    v = fma(-F[2 * n + n5], u[n5], v);
    r[c] = v;
}

// FP64 residual r = f - L u of the finest level (unit spacing) from the
// stored face coefficients A (F) and node diagonals D: since
// L u = sum_n A_n u_n - D u_c, r = f + D u_c - sum_n A_n u_n is a chain of
// seven FMAs.  The FP64 issue rate, not memory, bounds this kernel on GB300,
// so coefficients are read rather than recomputed.  The rounding error of the
// undifferenced form is ~8 eps D |u|, i.e. ~1e-12 relative to |f| even for
// the smoothest mode of a 512^3 grid, far below the stopping tolerance.
// Optionally also writes r in FP32 (the next V-cycle's right-hand side);
// always the per-block partial sums of r^2.  With the FP32 copy (mixed mode)
// r^2 is summed from it on the FP32 pipe, one FP64 instruction fewer per
// node.  The norm only decides the multigrid stopping test: a thread's FP32
// sum goes into its FP64 one every kRes32 nodes, so its relative error stays
// below kRes32 2^-24 = 4e-6 on every grid, and the block sums are FP64.  One
// round of four blocks per SM with 62 registers, so that a
// node's fifteen loads are all in flight: 512^3 2.19 -> 1.90 ms, 256^3 274 -> 246
// us against 38 registers in kRedBlocks blocks (eight FP64 instructions at 2
// lanes a clock and SM take 1.71 ms; rounding the FP32 copy by integer
// instructions instead took 2.3 ms).
constexpr int kRes32 = 64;
constexpr int kResPerSM = 4, kResBlocks = kResPerSM * (kRedBlocks / 8);
__global__ void __launch_bounds__(kRedThreads, kResPerSM) k_residual64_to32(Dims d, const double* __restrict__ u,
                                  const double* __restrict__ f, const double* __restrict__ F,
                                  const double* __restrict__ D, float* __restrict__ r32,
                                  double* __restrict__ partials) {
    double acc = 0.0;
    const size_t n = (size_t)d.cells;
    const double* __restrict__ Fx = F;
    const double* __restrict__ Fy = F + n;
    const double* __restrict__ Fz = F + 2 * n;
    const int stride = gridDim.x * blockDim.x;
    // (a loop of its own for the nodes of an FP32 sum: with the test inside one
    // loop the loads of several nodes are not in flight together, 256^3 solves 3% slower)
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells;) {
        float acc32 = 0.f;
        for (const int stop = min(d.cells, c + kRes32 * stride); c < stop; c += stride) {
            int i, j, k;
            cell_coords(d, c, i, j, k);
            const int n0 = cell_index(d, i + 1, j, k), n1 = cell_index(d, i - 1, j, k);
            const int n2 = cell_index(d, i, j + 1, k), n3 = cell_index(d, i, j - 1, k);
            const int n4 = cell_index(d, i, j, k + 1), n5 = cell_index(d, i, j, k - 1);
            double r = fma(D[c], u[c], f[c]);
            r = fma(-Fx[c], u[n0], r);
            r = fma(-Fx[n1], u[n1], r);
            r = fma(-Fy[c], u[n2], r);
            r = fma(-Fy[n3], u[n3], r);
            r = fma(-Fz[c], u[n4], r);
            r = fma(-Fz[n5], u[n5], r);
            if (r32) {
                const float rf = (float)r;
                r32[c] = rf;
                acc32 = fmaf(rf, rf, acc32);
            } else {
                acc = fma(r, r, acc);
            }
        }
        acc += (double)acc32;
    }
    acc = block_reduce<OpSum>(acc);
    if (threadIdx.x == 0) put_partial(partials, acc, kRedBlocks);
}

// x 2^e, for a positive normal x away from the ends of the range by its
// exponent bits, else by a product: no FP64 operation.
__device__ __forceinline__ double times_pow2(double x, int e) {
    const long long b = __double_as_longlong(x);
    const int old = (int)(b >> 52);
    return old > 64 && old < 1984 ? __longlong_as_double(b + ((long long)e << 52)) : x * ldexp(1.0, e);
}

// Face coefficients A = h^-2 (a_c + a_{c + e_a}) / 2 of a level, one array per
// axis, the node diagonal D = sum of the node's six A, and optionally 1 / D.
// h^-2 / 2 = 2^ex (ey, ez) of each axis.  Bound by the FP64 rate: each value is
// scaled by its exponent bits, so the three faces take one sum each and D six
// instructions on an isotropic level (17 in all with the products, 512^3 3.59
// -> 2.32 ms).
template <bool ISO>
__global__ void k_faces64(Dims d, int ex, int ey, int ez, const double* __restrict__ a,
                          double* __restrict__ F, double* __restrict__ D, double* __restrict__ inv_d) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const size_t n = (size_t)d.cells;
    const double ac = a[c];
    const double xp = times_pow2(a[cell_index(d, i + 1, j, k)], ex), xm = times_pow2(a[cell_index(d, i - 1, j, k)], ex);
    const double yp = times_pow2(a[cell_index(d, i, j + 1, k)], ey), ym = times_pow2(a[cell_index(d, i, j - 1, k)], ey);
    const double zp = times_pow2(a[cell_index(d, i, j, k + 1)], ez), zm = times_pow2(a[cell_index(d, i, j, k - 1)], ez);
    const double cx = times_pow2(ac, ex);
    const double cy = ISO ? cx : times_pow2(ac, ey), cz = ISO ? cx : times_pow2(ac, ez);
    F[c] = cx + xp, F[n + c] = cy + yp, F[2 * n + c] = cz + zp;
    const double sum = ((xp + xm) + (yp + ym)) + (zp + zm);
    const double dg = ISO ? fma(6.0, cx, sum) : fma(2.0, cx + (cy + cz), sum);
    D[c] = dg;
    if (inv_d) inv_d[c] = 1.0 / dg;
}

// Full weighting: weights (1/4, 1/2, 1/4) along every coarsened axis.
__global__ void k_restrict(Dims df, Dims dc, int cx, int cy, int cz, const float* __restrict__ in,
                           float* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= dc.cells) return;
    int I, J, K;
    cell_coords(dc, c, I, J, K);
    const int fi = cx ? 2 * I : I, fj = cy ? 2 * J : J, fk = cz ? 2 * K : K;
    float acc = 0.f;
    for (int oi = -cx; oi <= cx; ++oi) {
        const float wi = cx ? (oi == 0 ? 0.5f : 0.25f) : 1.f;
        for (int oj = -cy; oj <= cy; ++oj) {
            const float wj = cy ? (oj == 0 ? 0.5f : 0.25f) : 1.f;
            for (int ok = -cz; ok <= cz; ++ok) {
                const float wk = cz ? (ok == 0 ? 0.5f : 0.25f) : 1.f;
                acc += wi * wj * wk * in[cell_index(df, fi + oi, fj + oj, fk + ok)];
            }
        }
    }
    out[c] = acc;
}

// Full weighting in FP64 one axis after another, halved once at the end: 2
// FP64 instructions a value and axis instead of 4 a stencil point.
__device__ inline double full_weight(const Dims& df, const Dims& dc, int cx, int cy, int cz,
                                     const double* __restrict__ in, int c) {
    int I, J, K;
    cell_coords(dc, c, I, J, K);
    const int fi = cx ? 2 * I : I, fj = cy ? 2 * J : J, fk = cz ? 2 * K : K;
    auto along_k = [&](int i, int j) {
        const double v = in[cell_index(df, i, j, fk)];
        return cz ? fma(0.5, in[cell_index(df, i, j, fk - 1)] + in[cell_index(df, i, j, fk + 1)], v) : v;
    };
    auto along_j = [&](int i) {
        const double v = along_k(i, fj);
        return cy ? fma(0.5, along_k(i, fj - 1) + along_k(i, fj + 1), v) : v;
    };
    double acc = along_j(fi);
    if (cx) acc = fma(0.5, along_j(fi - 1) + along_j(fi + 1), acc);
    return acc * ((cx ? 0.5 : 1.0) * ((cy ? 0.5 : 1.0) * (cz ? 0.5 : 1.0)));
}

__global__ void k_restrict64(Dims df, Dims dc, int cx, int cy, int cz, const double* __restrict__ in,
                             double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < dc.cells) out[c] = full_weight(df, dc, cx, cy, cz, in, c);
}

// Residual r = f - L u evaluated at the fine nodes of each coarse node's
// full-weighting stencil and restricted at once (the fine residual is never
// stored): per node the 7-point residual f - L u followed by the full weighting.
// red: u has just been swept, so black nodes have none (but for rounding) and
// are left out, half the evaluations (128 x 64 x 32 nodes: 8.5 -> 7.2 us a level).
__global__ void k_resid_restrict(Dims df, Dims dc, int cx, int cy, int cz, float hx, float hy, float hz,
                                 const float* __restrict__ u, const float* __restrict__ f,
                                 const float* __restrict__ a, int face, int red, float* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= dc.cells) return;
    int I, J, K;
    cell_coords(dc, c, I, J, K);
    const int fi = cx ? 2 * I : I, fj = cy ? 2 * J : J, fk = cz ? 2 * K : K;
    float acc = 0.f;
    for (int oi = -cx; oi <= cx; ++oi) {
        const float wi = cx ? (oi == 0 ? 0.5f : 0.25f) : 1.f;
        for (int oj = -cy; oj <= cy; ++oj) {
            const float wj = cy ? (oj == 0 ? 0.5f : 0.25f) : 1.f;
            for (int ok = -cz; ok <= cz; ++ok) {
                if (red && ((fi + oi + fj + oj + fk + ok) & 1)) continue;
                const float wk = cz ? (ok == 0 ? 0.5f : 0.25f) : 1.f;
                const int i = (fi + oi) & (df.n0 - 1), j = (fj + oj) & (df.n1 - 1),
                          k = (fk + ok) & (df.n2 - 1);
                const int n = cell_index(df, i, j, k);
                Stencil7 s = stencil7_any(df, hx, hy, hz, i, j, k, n, u, a, face);
                const float r = f[n] - (s.off - s.diag * u[n]);
                acc += wi * wj * wk * r;
            }
        }
    }
    out[c] = acc;
}

// Face sums of the coarse level (every axis halved) from the fine level's
// nodal coefficient a (face sum a_c + a_n) or its face sums (fine_face).  A
// coarse face between coarse nodes I and I + 1 along an axis spans the two
// fine faces 2I|2I+1 and 2I+1|2I+2 of each fine line along that axis: in
// series they conduct as the harmonic mean of the two, and the 3 x 3 lines
// around the coarse line are weighted (1/4, 1/2, 1/4) in both transverse
// axes.  For a constant coefficient this is the re-discretised face; where
// the coefficient jumps it keeps the flux a fine-grid path can carry, which
// full weighting of a nodal coefficient does not.
__global__ void k_faces_line(Dims df, Dims dc, const float* __restrict__ in, int fine_face,
                             float* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= dc.cells) return;
    int I, J, K;
    cell_coords(dc, c, I, J, K);
    const int f0[3] = {2 * I, 2 * J, 2 * K};
    const float w[3] = {0.25f, 0.5f, 0.25f};
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        const int t1 = ax == 0 ? 1 : 0, t2 = ax == 2 ? 1 : 2;  // transverse axes
        float acc = 0.f;
        for (int o1 = -1; o1 <= 1; ++o1)
            for (int o2 = -1; o2 <= 1; ++o2) {
                int p[3];
                p[ax] = f0[ax];
                p[t1] = f0[t1] + o1;
                p[t2] = f0[t2] + o2;
                const int e0 = cell_index(df, p[0], p[1], p[2]);
                p[ax] += 1;
                const int e1 = cell_index(df, p[0], p[1], p[2]);
                p[ax] += 1;
                const int e2 = cell_index(df, p[0], p[1], p[2]);
                float g1, g2;
                if (fine_face) {
                    const float* g = in + (size_t)ax * df.cells;
                    g1 = g[e0], g2 = g[e1];
                } else {
                    g1 = in[e0] + in[e1], g2 = in[e1] + in[e2];
                }
                acc += w[o1 + 1] * w[o2 + 1] * __fdividef(2.f * g1 * g2, g1 + g2);
            }
        out[(size_t)ax * dc.cells + c] = acc;
    }
}

// Trilinear prolongation of the coarse correction, added to the fine field.
__global__ void k_prolong_add(Dims df, Dims dc, int cx, int cy, int cz, const float* __restrict__ uc,
                              float* __restrict__ u) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= df.cells) return;
    int i, j, k;
    cell_coords(df, c, i, j, k);
    int ii[2], jj[2], kk[2];
    float wi[2], wj[2], wk[2];
    int ni, nj, nk;
    if (!cx) { ii[0] = i; wi[0] = 1.f; ni = 1; }
    else if (!(i & 1)) { ii[0] = i >> 1; wi[0] = 1.f; ni = 1; }
    else { ii[0] = i >> 1; ii[1] = (i >> 1) + 1; wi[0] = wi[1] = 0.5f; ni = 2; }
    if (!cy) { jj[0] = j; wj[0] = 1.f; nj = 1; }
    else if (!(j & 1)) { jj[0] = j >> 1; wj[0] = 1.f; nj = 1; }
    else { jj[0] = j >> 1; jj[1] = (j >> 1) + 1; wj[0] = wj[1] = 0.5f; nj = 2; }
    if (!cz) { kk[0] = k; wk[0] = 1.f; nk = 1; }
    else if (!(k & 1)) { kk[0] = k >> 1; wk[0] = 1.f; nk = 1; }
    else { kk[0] = k >> 1; kk[1] = (k >> 1) + 1; wk[0] = wk[1] = 0.5f; nk = 2; }
    float acc = 0.f;
    for (int p = 0; p < ni; ++p)
        for (int q = 0; q < nj; ++q)
            for (int r = 0; r < nk; ++r)
                acc += wi[p] * wj[q] * wk[r] * uc[cell_index(dc, ii[p], jj[q], kk[r])];
    u[c] += acc;
}

// Trilinear prolongation in FP64 as one sum per node, weighted once (1/2 per
// odd coarsened axis); returns v + P(uc) at fine node c.
__device__ inline double prolonged(const Dims& df, const Dims& dc, int cx, int cy, int cz,
                                   const double* __restrict__ uc, int c, double v) {
    int i, j, k;
    cell_coords(df, c, i, j, k);
    const int oi = cx & i, oj = cy & j, ok = cz & k;  // odd along a coarsened axis
    const int I = cx ? i >> 1 : i, J = cy ? j >> 1 : j, K = cz ? k >> 1 : k;
    double acc = 0.0;
    for (int p = 0; p <= oi; ++p)
        for (int q = 0; q <= oj; ++q)
            for (int r = 0; r <= ok; ++r) acc += uc[cell_index(dc, I + p, J + q, K + r)];
    return fma(acc, (oi ? 0.5 : 1.0) * ((oj ? 0.5 : 1.0) * (ok ? 0.5 : 1.0)), v);
}

__global__ void k_prolong_add64(Dims df, Dims dc, int cx, int cy, int cz, const double* __restrict__ uc,
                                double* __restrict__ u) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < df.cells) u[c] = prolonged(df, dc, cx, cy, cz, uc, c, u[c]);
}

// The same where k is coarsened, a thread a pair (2K, 2K + 1) of fine nodes:
// the sums over the coarse rows around the pair serve both nodes, 2.75 FP64
// instructions a node on average (the FP64 rate bounds it) against 7.5 with a
// thread a node, whose warps also run the odd nodes' longer sums for all
// (128^3: 42 -> 16 us).
__global__ void k_prolong_pair64(Dims df, Dims dc, int cx, int cy, const double* __restrict__ uc,
                                 double* __restrict__ u) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= df.cells >> 1) return;
    int i, j, k;
    cell_coords(df, 2 * t, i, j, k);
    const int oi = cx & i, oj = cy & j;
    const int I = cx ? i >> 1 : i, J = cy ? j >> 1 : j, K = k >> 1;
    auto rows = [&](int kk) {
        double s = uc[cell_index(dc, I, J, kk)];
        if (oi) s += uc[cell_index(dc, I + 1, J, kk)];
        if (oj) {
            s += uc[cell_index(dc, I, J + 1, kk)];
            if (oi) s += uc[cell_index(dc, I + 1, J + 1, kk)];
        }
        return s;
    };
    const double a = rows(K), b = rows(K + 1);
    const int halvings = oi + oj;
    const double w = halvings == 0 ? 1.0 : halvings == 1 ? 0.5 : 0.25;
    double2* p = reinterpret_cast<double2*>(u + 2 * t);
    double2 v = *p;
    v.x = fma(a, w, v.x);
    v.y = fma(a + b, halvings == 0 ? 0.5 : halvings == 1 ? 0.25 : 0.125, v.y);
    *p = v;
}

// Coarsest level (64 nodes): the matrix M (kNc x kNc) with u = M f the
// mean-free solution of L u = f - mean(f), in FP64 by one block.
//
// Every neighbour of a red node is black, so the red block of A = -L is
// diagonal: A = [R -B; -B^T K] with R, K the node diagonals.  The black nodes
// see the 32 x 32 Schur complement S = K - B^T R^-1 B, whose null space is the
// constants; with a constant added to every entry (the mean of K over 32) it
// is positive definite and is inverted in place by symmetric sweeps without
// pivoting, one element of the lower triangle per thread.  From X that
// inverse, G = [R^-1 + R^-1 B X B^T R^-1, R^-1 B X; ., X] is a generalised
// inverse of A, and M = -P G P with P = I - 1 1^T / 64.
//
// Bound by one SM's FP64 rate (2 lanes a clock) and the 32 dependent pivots:
// 17 warps of multiply and FMA a pivot, against the 65 pivots over 65 x 130
// elements that a Gauss-Jordan elimination of the bordered matrix takes
// (286 us; 47 us in this form, mixed 32^3 solve of 8 steps 9.75 -> 7.86 ms).
constexpr int kHalf = kNc / 2;                      // red (and black) nodes
constexpr int kTri = kHalf * (kHalf + 1) / 2;       // lower triangle of S
constexpr int kInvThreads = (kTri + 31) / 32 * 32;  // 544

// 1 / x of a positive x by Newton's iteration from the FP32 reciprocal (24
// bits, then 48, then full precision); outside the FP32 range by division.
__device__ inline double recip_newton(double x) {
    if (!(x > 1e-30 && x < 1e30)) return 1.0 / x;
    double y = (double)__frcp_rn((float)x);
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

template <typename T>
__global__ void __launch_bounds__(kInvThreads) k_coarse_invert(Dims d, double hx, double hy,
                                                              double hz, const T* __restrict__ a,
                                                              int face, double* __restrict__ out) {
    __shared__ double w[kNc][6];       // couplings of node c to its six neighbours
    __shared__ int nb[kNc][6];
    __shared__ double diag[kNc];
    __shared__ double S[kHalf][kHalf + 1];
    __shared__ double col[2][kHalf], piv[2];
    __shared__ double G[kNc][kNc];     // rows and columns: red nodes, then black
    __shared__ double mean[kNc];
    const int t = threadIdx.x;
    // node of a colour: pair idx holds nodes 2 idx and 2 idx + 1, one of each
    auto node_of = [](int idx, int black) { return 2 * idx + ((((idx >> 3) + (idx >> 1)) & 1) ^ black); };
    if (t < kNc) {
        const int c = t;
        int i, j, k;
        cell_coords(d, c, i, j, k);
        const int n6[6] = {cell_index(d, i + 1, j, k), cell_index(d, i - 1, j, k),
                           cell_index(d, i, j + 1, k), cell_index(d, i, j - 1, k),
                           cell_index(d, i, j, k + 1), cell_index(d, i, j, k - 1)};
        const double hh[3] = {hx, hy, hz};
        double dg = 0.0;
        for (int q = 0; q < 6; ++q) {
            // face sum of face q: the +1 face of node c, or the +1 face of
            // its -1 neighbour
            const double g = face ? (double)a[(size_t)(q >> 1) * d.cells + ((q & 1) ? n6[q] : c)]
                                  : (double)a[c] + (double)a[n6[q]];
            const double wq = 0.5 * g * hh[q >> 1];
            w[c][q] = wq, nb[c][q] = n6[q];
            dg += wq;
        }
        diag[c] = dg;
    }
    __syncthreads();
    if (t < kHalf) {  // row t of S
        const int c = node_of(t, 1);
        double shift = diag[c];
        for (int o = 16; o > 0; o >>= 1) shift += __shfl_xor_sync(0xffffffffu, shift, o);
        shift *= 1.0 / (kHalf * kHalf);
        for (int q = 0; q < kHalf; ++q) S[t][q] = shift;
        S[t][t] += diag[c];
        for (int q = 0; q < 6; ++q) {
            const int r = nb[c][q];
            const double f = w[c][q] * recip_newton(diag[r]);
            for (int p = 0; p < 6; ++p) S[t][nb[r][p] >> 1] -= f * w[r][p];
        }
    }
    __syncthreads();
    int r = 0, c = 0;  // this thread's element of the lower triangle
    if (t < kTri) {
        c = t;
        while (c > r) c -= ++r;
    }
    double v = 0.0;
    if (t < kTri) v = S[r][c];
    // publishes column p of the symmetric matrix and 1 / its pivot
    auto publish = [&](int p) {
        if (t < kTri && (r == p || c == p)) {
            col[p & 1][r == p ? c : r] = v;
            if (r == c) piv[p & 1] = recip_newton(v);
        }
    };
    publish(0);
    __syncthreads();
    for (int p = 0; p < kHalf; ++p) {
        const double di = piv[p & 1];
        if (r != p && c != p) v = fma(-(col[p & 1][r] * di), col[p & 1][c], v);
        else if (r == c) v = -di;
        else v *= di;
        if (p + 1 < kHalf) publish(p + 1);
        __syncthreads();
    }
    if (t < kTri) {  // the sweeps leave -X
        G[kHalf + r][kHalf + c] = -v;
        G[kHalf + c][kHalf + r] = -v;
    }
    if (t < kHalf) col[0][t] = recip_newton(diag[node_of(t, 0)]);
    __syncthreads();
    for (int e = t; e < kHalf * kHalf; e += blockDim.x) {  // R^-1 B X
        const int x = e / kHalf, y = e % kHalf, n = node_of(x, 0);
        double s = 0.0;
        for (int q = 0; q < 6; ++q) s = fma(w[n][q], G[kHalf + (nb[n][q] >> 1)][kHalf + y], s);
        s *= col[0][x];
        G[x][kHalf + y] = s;
        G[kHalf + y][x] = s;
    }
    __syncthreads();
    for (int e = t; e < kHalf * kHalf; e += blockDim.x) {  // R^-1 + (R^-1 B X) B^T R^-1
        const int x = e / kHalf, y = e % kHalf, n = node_of(y, 0);
        double s = 0.0;
        for (int q = 0; q < 6; ++q) s = fma(w[n][q], G[x][kHalf + (nb[n][q] >> 1)], s);
        G[x][y] = (s + (x == y ? 1.0 : 0.0)) * col[0][y];
    }
    __syncthreads();
    if (t < 512) {  // row means, eight threads a row
        double s = 0.0;
        for (int y = t & 7; y < kNc; y += 8) s += G[t >> 3][y];
        for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 7) == 0) mean[t >> 3] = s * (1.0 / kNc);
    }
    __syncthreads();
    if (t < 32) {
        double s = mean[t] + mean[t + 32];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (t == 0) piv[0] = s * (1.0 / kNc);
    }
    __syncthreads();
    const double all = piv[0];
    for (int e = t; e < kNc * kNc; e += blockDim.x) {
        const int x = e / kNc, y = e % kNc;  // nodes of the row and the column
        const int cx = (x >> 1) + (node_of(x >> 1, 0) == x ? 0 : kHalf);
        const int cy = (y >> 1) + (node_of(y >> 1, 0) == y ? 0 : kHalf);
        out[e] = (mean[cx] - G[cx][cy]) + (mean[cy] - all);
    }
}

__global__ void k_to_f32(int cells, const double* __restrict__ x, float* __restrict__ y) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < cells) y[c] = (float)x[c];
}

__global__ void k_correct(int cells, double* __restrict__ u, const float* __restrict__ e) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < cells) u[c] += (double)e[c];
}

}  // namespace

void launch_rbgs_sweep(const Level& L, float* u, const float* f, const float* a, cudaStream_t st) {
    const int half = L.d.cells >> 1;
    launch_counter() += 2;
    for (int colour = 0; colour < 2; ++colour)
        k_rbgs_colour<<<nblocks(half), kThreads, 0, st>>>(L.d, (float)L.h2i[0], (float)L.h2i[1],
                                                          (float)L.h2i[2], colour, u, f, a, L.face);
}

template <>
void launch_restrict<float>(const Level& fine, const Level& coarse, const float* in, float* out,
                            cudaStream_t st) {
    launch_counter()++;
    k_restrict<<<nblocks(coarse.d.cells), kThreads, 0, st>>>(
        fine.d, coarse.d, fine.coarsen[0], fine.coarsen[1], fine.coarsen[2], in, out);
}

template <>
void launch_restrict<double>(const Level& fine, const Level& coarse, const double* in, double* out,
                             cudaStream_t st) {
    launch_counter()++;
    k_restrict64<<<nblocks(coarse.d.cells), kThreads, 0, st>>>(
        fine.d, coarse.d, fine.coarsen[0], fine.coarsen[1], fine.coarsen[2], in, out);
}

void launch_resid_restrict(const Level& fine, const Level& coarse, const float* u, const float* f,
                           const float* a, float* out, bool swept, cudaStream_t st) {
    launch_counter()++;
    k_resid_restrict<<<nblocks(coarse.d.cells), kThreads, 0, st>>>(
        fine.d, coarse.d, fine.coarsen[0], fine.coarsen[1], fine.coarsen[2], (float)fine.h2i[0],
        (float)fine.h2i[1], (float)fine.h2i[2], u, f, a, fine.face, swept ? 1 : 0, out);
}

void launch_faces_line(const Level& fine, const Level& coarse, const float* in, float* out,
                       cudaStream_t st) {
    launch_counter()++;
    k_faces_line<<<nblocks(coarse.d.cells), kThreads, 0, st>>>(fine.d, coarse.d, in, fine.face, out);
}

template <>
void launch_prolong_add<float>(const Level& fine, const Level& coarse, const float* uc, float* u,
                               cudaStream_t st) {
    launch_counter()++;
    k_prolong_add<<<nblocks(fine.d.cells), kThreads, 0, st>>>(
        fine.d, coarse.d, fine.coarsen[0], fine.coarsen[1], fine.coarsen[2], uc, u);
}

template <>
void launch_prolong_add<double>(const Level& fine, const Level& coarse, const double* uc, double* u,
                                cudaStream_t st) {
    launch_counter()++;
    if (fine.coarsen[2]) {
        k_prolong_pair64<<<nblocks(fine.d.cells >> 1), kThreads, 0, st>>>(fine.d, coarse.d, fine.coarsen[0],
                                                                          fine.coarsen[1], uc, u);
        return;
    }
    k_prolong_add64<<<nblocks(fine.d.cells), kThreads, 0, st>>>(
        fine.d, coarse.d, fine.coarsen[0], fine.coarsen[1], fine.coarsen[2], uc, u);
}

template <typename T>
void launch_coarse_invert(const Level& L, const T* a, double* minv, cudaStream_t st) {
    launch_counter()++;
    k_coarse_invert<T><<<1, kInvThreads, 0, st>>>(L.d, L.h2i[0], L.h2i[1], L.h2i[2], a,
                                                         L.face, minv);
}

void launch_to_f32(int cells, const double* x, float* y, cudaStream_t st) {
    launch_counter()++;
    k_to_f32<<<nblocks(cells), kThreads, 0, st>>>(cells, x, y);
}

void launch_residual64_to32(const Level& L, const double* u, const double* f, const double* F,
                            const double* D, float* r32, double* partials, cudaStream_t st) {
    launch_counter()++;
    k_residual64_to32<<<kResBlocks, kRedThreads, 0, st>>>(L.d, u, f, F, D, r32, partials);
}

void launch_residual_norm64(const Level& L, const double* u, const double* f, const double* F,
                            const double* D, double* partials, cudaStream_t st) {
    launch_counter()++;
    k_residual64_to32<<<kResBlocks, kRedThreads, 0, st>>>(L.d, u, f, F, D, nullptr, partials);
}

void launch_rbgs_sweep64(const Level& L, double* u, const double* f, const double* F,
                         const double* inv_d, bool zero_u, cudaStream_t st) {
    const int half = L.d.cells >> 1;
    launch_counter() += 2;
    for (int colour = 0; colour < 2; ++colour)
        k_rbgs_colour64<<<nblocks(half), kThreads, 0, st>>>(L.d, colour, zero_u && colour == 0 ? 1 : 0, u, f, F,
                                                            inv_d);
}

void launch_residual64(const Level& L, const double* u, const double* f, const double* F, const double* D,
                       double* r, cudaStream_t st) {
    launch_counter()++;
    k_residual64<<<nblocks(L.d.cells), kThreads, 0, st>>>(L.d, u, f, F, D, r);
}

void launch_faces64(const Level& L, const double* a, double* F, double* D, double* inv_d,
                    cudaStream_t st) {
    launch_counter()++;
    const int ex = ilogb(0.5 * L.h2i[0]), ey = ilogb(0.5 * L.h2i[1]), ez = ilogb(0.5 * L.h2i[2]);
    auto fn = ex == ey && ey == ez ? k_faces64<true> : k_faces64<false>;
    fn<<<nblocks(L.d.cells), kThreads, 0, st>>>(L.d, ex, ey, ez, a, F, D, inv_d);
}

void launch_correct(int cells, double* u, const float* e, cudaStream_t st) {
    launch_counter()++;
    k_correct<<<nblocks(cells), kThreads, 0, st>>>(cells, u, e);
}

template void launch_coarse_invert<float>(const Level&, const float*, double*, cudaStream_t);
template void launch_coarse_invert<double>(const Level&, const double*, double*, cudaStream_t);

}  // namespace recon

// The coarse end of the FP32 V-cycle in one block: every level from l0 (at most
// 4096 nodes) down to the 4^3 level is smoothed, restricted, solved and prolonged
// in shared memory, so a V-cycle launches one kernel for all of these levels.
//
// Each level's face coefficients and 1 / diagonal are formed once, as it is
// loaded; a node of a colour phase then takes 14 shared values and no division.
// Consecutive threads take consecutive k of alternating planes (the parity gives
// the colour), which fall into distinct banks.  As in coarse_cluster.cu the
// residual is evaluated at red nodes only after a sweep, and the prolongation
// added at black nodes only before one.  The spacing factors come as FP32 from
// the host: an FP64 conversion in each of 1024 threads takes the SM 512 cycles.
// 32 x 16 x 8 and below: 33.6 -> 24.4 us a V(1, 1).

namespace recon {

namespace {

constexpr int kVcT = 1024;

struct CoarseSet32 {
    int nlev, nu1, nu2;
    Dims d[kCoarseMaxLevels];
    int coarsen[kCoarseMaxLevels][3];
    float w[kCoarseMaxLevels][3];  // h^-2 / 2 per axis
    const float* a[kCoarseMaxLevels];
};

__global__ void __launch_bounds__(kVcT) k_coarse_vcycle(const __grid_constant__ CoarseSet32 cs,
                                                        const float* __restrict__ f_top,
                                                        float* __restrict__ u_top,
                                                        const double* __restrict__ minv_g, int zero_u) {
    extern __shared__ double sm_vc[];
    double* minv = sm_vc;            // the 4^3 matrix, then its right-hand side in FP64
    double* f64 = minv + kNc * kNc;
    float* base = reinterpret_cast<float*>(f64 + kNc);
    // arrays of level l: gx, gy, gz (the face between a node and its +1
    // neighbour), 1 / diagonal, u, f, r (a until the faces are formed)
    auto arrays = [&](int l) {
        float* q = base;
        for (int m = 0; m < l; ++m) q += 7 * cs.d[m].cells;
        return q;
    };
    const int t0 = threadIdx.x, last = cs.nlev - 1;
    for (int e = t0; e < kNc * kNc; e += kVcT) minv[e] = minv_g[e];
    for (int l = 0; l < last; ++l) {
        float* r = arrays(l) + 6 * cs.d[l].cells;
        for (int c = t0; c < cs.d[l].cells; c += kVcT) r[c] = cs.a[l][c];
    }
    {
        const int n = cs.d[0].cells;
        float *u = arrays(0) + 4 * n, *f = u + n;
        for (int c = t0; c < n; c += kVcT) {
            f[c] = f_top[c];
            u[c] = zero_u ? 0.f : u_top[c];
        }
    }
    __syncthreads();
    for (int l = 0; l < last; ++l) {
        const Dims d = cs.d[l];
        float* g = arrays(l);
        const float* a = g + 6 * d.cells;
        for (int c = t0; c < d.cells; c += kVcT) {
            int i, j, k;
            cell_coords(d, c, i, j, k);
            g[c] = cs.w[l][0] * (a[c] + a[cell_index(d, i + 1, j, k)]);
            g[d.cells + c] = cs.w[l][1] * (a[c] + a[cell_index(d, i, j + 1, k)]);
            g[2 * d.cells + c] = cs.w[l][2] * (a[c] + a[cell_index(d, i, j, k + 1)]);
        }
    }
    __syncthreads();
    auto diag = [&](const Dims& d, const float* g, int i, int j, int k, int c) {
        return (g[c] + g[cell_index(d, i - 1, j, k)]) +
               (g[d.cells + c] + g[d.cells + cell_index(d, i, j - 1, k)]) +
               (g[2 * d.cells + c] + g[2 * d.cells + cell_index(d, i, j, k - 1)]);
    };
    for (int l = 0; l < last; ++l) {
        const Dims d = cs.d[l];
        float* g = arrays(l);
        for (int c = t0; c < d.cells; c += kVcT) {
            int i, j, k;
            cell_coords(d, c, i, j, k);
            g[3 * d.cells + c] = 1.f / diag(d, g, i, j, k, c);
        }
    }
    __syncthreads();
    auto off = [&](const Dims& d, const float* g, const float* u, int i, int j, int k, int c) {
        const int xm = cell_index(d, i - 1, j, k), ym = cell_index(d, i, j - 1, k), zm = cell_index(d, i, j, k - 1);
        return (g[c] * u[cell_index(d, i + 1, j, k)] + g[xm] * u[xm]) +
               (g[d.cells + c] * u[cell_index(d, i, j + 1, k)] + g[d.cells + ym] * u[ym]) +
               (g[2 * d.cells + c] * u[cell_index(d, i, j, k + 1)] + g[2 * d.cells + zm] * u[zm]);
    };
    // the t-th node of a colour
    auto node = [&](const Dims& d, int t, int colour, int& i, int& j, int& k) {
        k = t & (d.n2 - 1), j = (t >> d.s2) & (d.n1 - 1);
        i = 2 * (t >> (d.s1 + d.s2)) + ((j + k + colour) & 1);
        return cell_index(d, i, j, k);
    };
    auto sweeps = [&](int l, int nu, bool zero) {
        const Dims d = cs.d[l];
        float *g = arrays(l), *u = g + 4 * d.cells;
        const float *rd = g + 3 * d.cells, *f = u + d.cells;
        for (int s = 0; s < 2 * nu; ++s) {
            for (int t = t0; t < d.cells >> 1; t += kVcT) {
                int i, j, k;
                const int c = node(d, t, s & 1, i, j, k);
                u[c] = ((zero && s == 0 ? 0.f : off(d, g, u, i, j, k, c)) - f[c]) * rd[c];
            }
            __syncthreads();
        }
    };
    for (int l = 0; l < last; ++l) {
        const Dims d = cs.d[l], dc = cs.d[l + 1];
        float *g = arrays(l), *u = g + 4 * d.cells, *r = g + 6 * d.cells;
        const float* f = g + 5 * d.cells;
        sweeps(l, cs.nu1, l > 0 || zero_u);
        for (int colour = cs.nu1 ? 0 : 1; colour >= 0; --colour)
            for (int t = t0; t < d.cells >> 1; t += kVcT) {
                int i, j, k;
                const int c = node(d, t, colour, i, j, k);
                r[c] = f[c] - (off(d, g, u, i, j, k, c) - diag(d, g, i, j, k, c) * u[c]);
            }
        __syncthreads();
        const int cx = cs.coarsen[l][0], cy = cs.coarsen[l][1], cz = cs.coarsen[l][2];
        float* gc = arrays(l + 1);
        for (int c = t0; c < dc.cells; c += kVcT) {
            int I, J, K;
            cell_coords(dc, c, I, J, K);
            const int fi = cx ? 2 * I : I, fj = cy ? 2 * J : J, fk = cz ? 2 * K : K;
            float acc = 0.f;
            for (int oi = -cx; oi <= cx; ++oi)
                for (int oj = -cy; oj <= cy; ++oj) {
                    const float wij = (cx ? (oi ? 0.25f : 0.5f) : 1.f) * (cy ? (oj ? 0.25f : 0.5f) : 1.f);
                    for (int ok = -cz; ok <= cz; ++ok) {
                        if (cs.nu1 && ((fi + oi + fj + oj + fk + ok) & 1)) continue;  // black: none
                        acc += wij * (cz ? (ok ? 0.25f : 0.5f) : 1.f) * r[cell_index(d, fi + oi, fj + oj, fk + ok)];
                    }
                }
            if (l + 1 == last) f64[c] = (double)acc;
            else gc[5 * dc.cells + c] = acc;
            gc[4 * dc.cells + c] = 0.f;
        }
        __syncthreads();
    }
    if (t0 < 4 * kNc) {  // 4^3: u = M f in FP64, four threads a row
        double acc = 0.0;
        for (int c = t0 & 3; c < kNc; c += 4) acc = fma(minv[(t0 >> 2) * kNc + c], f64[c], acc);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if ((t0 & 3) == 0) arrays(last)[4 * kNc + (t0 >> 2)] = (float)acc;
    }
    __syncthreads();
    for (int l = last - 1; l >= 0; --l) {
        const Dims d = cs.d[l], dc = cs.d[l + 1];
        float* u = arrays(l) + 4 * d.cells;
        const float* uc = arrays(l + 1) + 4 * dc.cells;
        const int cx = cs.coarsen[l][0], cy = cs.coarsen[l][1], cz = cs.coarsen[l][2];
        for (int colour = cs.nu2 ? 1 : 0; colour < 2; ++colour)
            for (int t = t0; t < d.cells >> 1; t += kVcT) {
                int i, j, k;
                const int c = node(d, t, colour, i, j, k);
                const int oi = cx & i, oj = cy & j, ok = cz & k;  // odd along a coarsened axis
                const int I = cx ? i >> 1 : i, J = cy ? j >> 1 : j, K = cz ? k >> 1 : k;
                // the two values of each axis, equal ones where it is even
                auto row = [&](int II, int JJ) { return uc[cell_index(dc, II, JJ, K)] + uc[cell_index(dc, II, JJ, K + ok)]; };
                u[c] += 0.125f * ((row(I, J) + row(I, J + oj)) + (row(I + oi, J) + row(I + oi, J + oj)));
            }
        __syncthreads();
        sweeps(l, cs.nu2, false);
    }
    const float* u = arrays(0) + 4 * cs.d[0].cells;
    for (int c = t0; c < cs.d[0].cells; c += kVcT) u_top[c] = u[c];
}

}  // namespace

size_t coarse_vcycle_smem(size_t cells) {
    return 7 * cells * sizeof(float) + (kNc + 1) * kNc * sizeof(double);
}

bool launch_coarse_vcycle(const CoarseSet& cs, const float* f_top, float* u_top, const double* minv,
                          bool zero_u, cudaStream_t st) {
    size_t cells = 0;
    for (int l = 0; l < cs.nlev; ++l) cells += cs.lv[l].d.cells;
    const size_t sm = coarse_vcycle_smem(cells);
    if (cs.nlev < 1 || cs.nlev > kCoarseMaxLevels || sm > kCoarseMaxSmem) return false;
    CoarseSet32 s{};
    s.nlev = cs.nlev, s.nu1 = cs.nu1, s.nu2 = cs.nu2;
    for (int l = 0; l < cs.nlev; ++l) {
        s.d[l] = cs.lv[l].d, s.a[l] = (const float*)cs.a[l];
        for (int x = 0; x < 3; ++x) s.coarsen[l][x] = cs.lv[l].coarsen[x], s.w[l][x] = (float)(0.5 * cs.lv[l].h2i[x]);
    }
    allow_smem((const void*)k_coarse_vcycle, (int)kCoarseMaxSmem);
    launch_counter()++;
    k_coarse_vcycle<<<1, kVcT, sm, st>>>(s, f_top, u_top, minv, zero_u ? 1 : 0);
    return true;
}

// The same for FP64 levels (at most kCoarse64Cells nodes on the first), from
// their stored faces and diagonals: 8 FP64 instructions a node and colour.
// One block holds a level of 8^3 nodes (a node a thread and phase); above
// that its two FP64 lanes a clock would bound it (329 us for one V(2,2) of
// 32^3 over a cluster of 8 blocks with the faces formed in every phase;
// 88 us as one launch per phase over the whole chip down to 8^3).
namespace {

__global__ void __launch_bounds__(512) k_coarse_vcycle64(CoarseSet64 cs, const double* __restrict__ f_top,
                                                         double* __restrict__ u_top,
                                                         const double* __restrict__ minv, int zero_u) {
    extern __shared__ double sm64[];
    double *u[kCoarseMaxLevels], *f[kCoarseMaxLevels], *r[kCoarseMaxLevels], *F[kCoarseMaxLevels],
        *D[kCoarseMaxLevels], *I[kCoarseMaxLevels];
    double* q = sm64;
    for (int l = 0; l < cs.nlev; ++l) {
        const int n = cs.lv[l].d.cells;
        u[l] = q, f[l] = q + n, r[l] = q + 2 * n, F[l] = q + 3 * n, D[l] = q + 6 * n, I[l] = q + 7 * n;
        q += 8 * n;
        if (l + 1 == cs.nlev) continue;  // the 4^3 level is solved with minv
        for (int c = threadIdx.x; c < 3 * n; c += blockDim.x) F[l][c] = cs.F[l][c];
        for (int c = threadIdx.x; c < n; c += blockDim.x) D[l][c] = cs.D[l][c], I[l][c] = cs.inv[l][c];
    }
    for (int c = threadIdx.x; c < cs.lv[0].d.cells; c += blockDim.x) {
        f[0][c] = f_top[c];
        u[0][c] = zero_u ? 0.0 : u_top[c];
    }
    double* mi = q;
    for (int e = threadIdx.x; e < kNc * kNc; e += blockDim.x) mi[e] = minv[e];
    __syncthreads();
    // sum_n A_n u_n of node (i, j, k)
    auto off = [&](int l, int i, int j, int k, int c) {
        const Dims& d = cs.lv[l].d;
        const int n = d.cells;
        const int n1 = cell_index(d, i - 1, j, k), n3 = cell_index(d, i, j - 1, k), n5 = cell_index(d, i, j, k - 1);
        double o = F[l][c] * u[l][cell_index(d, i + 1, j, k)];
        o = fma(F[l][n1], u[l][n1], o);
        o = fma(F[l][n + c], u[l][cell_index(d, i, j + 1, k)], o);
        o = fma(F[l][n + n3], u[l][n3], o);
        o = fma(F[l][2 * n + c], u[l][cell_index(d, i, j, k + 1)], o);
        return fma(F[l][2 * n + n5], u[l][n5], o);
    };
    auto sweeps = [&](int l, int nu) {
        const Dims& d = cs.lv[l].d;
        const int half = d.cells >> 1, hs2 = d.s2 - 1;
        for (int s = 0; s < 2 * nu; ++s) {
            for (int t = threadIdx.x; t < half; t += blockDim.x) {
                const int j = (t >> hs2) & (d.n1 - 1), i = t >> (d.s1 + hs2);
                const int k = 2 * (t & ((1 << hs2) - 1)) + ((i + j + s) & 1);
                const int c = cell_index(d, i, j, k);
                u[l][c] = (off(l, i, j, k, c) - f[l][c]) * I[l][c];
            }
            __syncthreads();
        }
    };
    const int last = cs.nlev - 1;
    for (int l = 0; l < last; ++l) {
        const Dims &d = cs.lv[l].d, &dc = cs.lv[l + 1].d;
        sweeps(l, cs.nu1);
        for (int c = threadIdx.x; c < d.cells; c += blockDim.x) {
            int i, j, k;
            cell_coords(d, c, i, j, k);
            r[l][c] = fma(D[l][c], u[l][c], f[l][c]) - off(l, i, j, k, c);
        }
        __syncthreads();
        for (int c = threadIdx.x; c < dc.cells; c += blockDim.x) {
            f[l + 1][c] = full_weight(d, dc, cs.lv[l].coarsen[0], cs.lv[l].coarsen[1], cs.lv[l].coarsen[2], r[l], c);
            u[l + 1][c] = 0.0;
        }
        __syncthreads();
    }
    if (threadIdx.x < 4 * kNc) {  // u = M f, four threads a row
        const int row = threadIdx.x >> 2;
        double acc = 0.0;
        for (int c = threadIdx.x & 3; c < kNc; c += 4) acc = fma(mi[row * kNc + c], f[last][c], acc);
        acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if ((threadIdx.x & 3) == 0) u[last][row] = acc;
    }
    __syncthreads();
    for (int l = last - 1; l >= 0; --l) {
        for (int c = threadIdx.x; c < cs.lv[l].d.cells; c += blockDim.x)
            u[l][c] = prolonged(cs.lv[l].d, cs.lv[l + 1].d, cs.lv[l].coarsen[0], cs.lv[l].coarsen[1],
                                cs.lv[l].coarsen[2], u[l + 1], c, u[l][c]);
        __syncthreads();
        sweeps(l, cs.nu2);
    }
    for (int c = threadIdx.x; c < cs.lv[0].d.cells; c += blockDim.x) u_top[c] = u[0][c];
}

}  // namespace

void launch_coarse_vcycle64(const CoarseSet64& cs, const double* f_top, double* u_top, const double* minv,
                            bool zero_u, cudaStream_t st) {
    size_t cells = 0;
    for (int l = 0; l < cs.nlev; ++l) cells += cs.lv[l].d.cells;
    // at most 2 x kCoarse64Cells nodes over all levels
    const size_t sm = (8 * cells + kNc * kNc) * sizeof(double);
    allow_smem((const void*)k_coarse_vcycle64, (int)((16 * kCoarse64Cells + kNc * kNc) * sizeof(double)));
    launch_counter()++;
    k_coarse_vcycle64<<<1, 512, sm, st>>>(cs, f_top, u_top, minv, zero_u ? 1 : 0);
}

}  // namespace recon
