// screened.cu -- the passes of a step that decide something at every node from
// the triad e = I + Hess phi: the limited source (App. A Eq. elliptic), the
// step limiter and the closing statistics; and the outputs det e, lambda0 and
// delta_r.  Source and limiter need FP64 only near a threshold (the compression limit
// xi_m, the volume limit v_m, the eigenvalue floor): everywhere else FP32
// values with a bound on their error settle the question, and the result is
// the FP64 one.
//
// Both stream planes of an 8 x 32 (or 16 x 16) tile along i: a plane's FP32 values (with a
// one-node ring) go through shared memory once, and a thread keeps its
// column's sums of the last two planes in registers.  A node that FP32 does not
// settle is put on its warp's list, and a full list of 32 runs the FP64 form
// with every lane at work (at about one node in a hundred, a third of all
// warps would otherwise run it for a lane or two).  The lists follow the nodes' order, so sums
// do not depend on timing.  The grid is one round of resident blocks over the
// planes of all tiles.
//
// 512^3: the source 11.9 -> 1.08 ms (it formed and stored e in FP64), the
// limiter 5.35 -> 1.13 ms.  With three blocks of 80 registers an SM the issue
// slots are 58% and 62% busy (256^3, first step) and the FP64 pipe 60% in the
// source, whose 1 - m and sum are FP64 at every node; DRAM is far from its rate.
#include "checked.cuh"
#include "eigen32.cuh"
#include "geometry.cuh"
#include "recon_internal.cuh"
#include "reduce.cuh"

namespace recon {

namespace {

// A tile of 256 nodes of the (j, k) plane, GK of them along k (32, or 16 on
// grids whose last axis is no multiple of 32), and with its one-node ring.
constexpr int GT = 256;
template <int GK>
struct Tile {
    static constexpr int J = GT / GK, PK = GK + 2, N = (J + 2) * PK;
    // the thread's node in a plane's buffer, which holds the ring around it
    // (RC_OFF: checked against the extent in the RECON_CHECKED build)
    __device__ static int own() {
        return PK + 1 + RC_OFF((int)(threadIdx.x / GK) * PK + (int)(threadIdx.x % GK), N - 2 * PK - 2, 401);
    }
};
constexpr int GPERSM = 3, GBLOCKS = GPERSM * (kRedBlocks / 8);

// lambda_min(M) > floor by Sylvester's criterion on M - floor I.
__device__ inline bool pd_above(Sym3 M, double floor) {
    M.xx -= floor, M.yy -= floor, M.zz -= floor;
    return M.xx > 0.0 && (M.xx * M.yy - M.xy * M.xy) > 0.0 && det3(M) > 0.0;
}

struct Hess32 {
    float xx, yy, zz, xy, xz, yz, vmax;  // vmax: the largest |value| read
};

// One FP32 field's sums of a column: fed plane after plane, it gives the
// Hessian at the node one plane back.  An entry combines at most four stencil
// values of magnitude <= vmax; the FP32 copies and at most four operations
// each round by 2^-24 relative, so 32 u vmax bounds its error with room.
template <int GPK>
struct Column32 {
    float ca, cb, ja, jb, ka, kb, va, vb, syb, szb, yzb, gyb, gzb, gx;
    // f: the node in the plane (its ring around it); gives the Hessian and
    // twice the gradient (gx, gyo, gzo) of the node on the plane before
    __device__ __forceinline__ Hess32 feed(const float* f, float& gyo, float& gzo) {
        const float c = f[0], jp = f[GPK], jm = f[-GPK], kp = f[1], km = f[-1];
        const float pp = f[GPK + 1], pm = f[GPK - 1], mp = f[-GPK + 1], mm = f[-GPK - 1];
        const float jd = jp - jm, kd = kp - km;
        const float v = fmaxf(fmaxf(fmaxf(fabsf(c), fabsf(jp)), fmaxf(fabsf(jm), fabsf(kp))),
                              fmaxf(fmaxf(fabsf(km), fabsf(pp)), fmaxf(fmaxf(fabsf(pm), fabsf(mp)), fabsf(mm))));
        Hess32 h;
        h.xx = (c - 2.f * cb) + ca, h.yy = syb, h.zz = szb;
        h.xy = 0.25f * (jd - ja), h.xz = 0.25f * (kd - ka), h.yz = yzb;
        h.vmax = fmaxf(v, fmaxf(va, vb));
        gx = c - ca, gyo = gyb, gzo = gzb;
        syb = (jp - 2.f * c) + jm, szb = (kp - 2.f * c) + km, yzb = 0.25f * ((pp - pm) - (mp - mm));
        gyb = jd, gzb = kd;
        ca = cb, cb = c, ja = jb, jb = jd, ka = kb, kb = kd, va = vb, vb = v;
        return h;
    }
};

// Sylvester's test of N = M - floor I in FP32 with a bound on its error:
// returns +1 when N is certainly positive definite, -1 when it certainly is
// not, 0 when FP32 cannot tell.  eps bounds the error of every entry of M;
// the minors' bounds add the propagated entry errors and the FP32 roundings
// of their own evaluation (u = 2^-24).
__device__ __forceinline__ int sylvester32(float xx, float yy, float zz, float xy, float xz, float yz,
                                           float floor, float eps) {
    xx -= floor, yy -= floor, zz -= floor;
    const float big = fmaxf(fmaxf(fabsf(xx), fabsf(yy)), fmaxf(fabsf(zz),
                            fmaxf(fabsf(xy), fmaxf(fabsf(xz), fabsf(yz)))));
    const float en = eps + 2.0f * kU * (big + floor);  // entries of N
    const float m1 = xx;
    const float m2 = xx * yy - xy * xy;
    const float m3 = xx * (yy * zz - yz * yz) - xy * (xy * zz - yz * xz) + xz * (xy * yz - yy * xz);
    const float e1 = en;
    const float e2 = 4.0f * en * big + en * en + 8.0f * kU * big * big;
    const float e3 = 9.0f * en * big * big + 3.0f * en * en * big + en * en * en + 72.0f * kU * big * big * big;
    if (m1 < -e1 || m2 < -e2 || m3 < -e3) return -1;
    if (m1 > e1 && m2 > e2 && m3 > e3) return 1;
    return 0;
}

// The nodes of the tile's planes in a fixed order: calls plane(p, buffer) for
// every plane from the one before a piece to the one after it, with the
// piece's first plane and column origin, from NF fields staged in shared
// memory.
template <int GK, int NF, typename Begin, typename Plane>
__device__ __forceinline__ void stream_planes(const Dims& d, const float* const (&field)[NF],
                                              float (&buf)[2][NF][Tile<GK>::N], Begin&& begin, Plane&& plane) {
    constexpr int GJ = Tile<GK>::J, GPK = Tile<GK>::PK, GN = Tile<GK>::N;
    static_assert(GN <= 2 * GT, "two values a thread and field");
    const int t = threadIdx.x;
    const int tiles_k = d.n2 / GK;
    const long long planes = (long long)tiles_k * (d.n1 / GJ) * d.n0;
    long long at = planes * blockIdx.x / gridDim.x;
    const long long end = planes * (blockIdx.x + 1) / gridDim.x;
    const int e1 = t + GT;
    const bool two = e1 < GN;
    while (at < end) {
        const int col = (int)(at / d.n0), i0 = (int)(at % d.n0);
        const int i1 = (int)min((long long)d.n0, i0 + (end - at));
        at += i1 - i0;
        const int k0 = (col % tiles_k) * GK, j0 = (col / tiles_k) * GJ;
        const int c0 = cell_index(d, 0, j0 - 1 + t / GPK, k0 - 1 + t % GPK);
        const int c1 = two ? cell_index(d, 0, j0 - 1 + e1 / GPK, k0 - 1 + e1 % GPK) : 0;
        const int np = d.n1 * d.n2;
        float v0[NF], v1[NF];
        auto load = [&](int i) {
            const int b = (i & (d.n0 - 1)) * np;
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                v0[q] = field[q][RC_OFF(b + c0, d.cells, 402)];
                v1[q] = two ? field[q][RC_OFF(b + c1, d.cells, 403)] : 0.f;
            }
        };
        begin();
        load(i0 - 1);
        for (int p = i0 - 1; p <= i1; ++p) {
            const int w = (p - i0 + 1) & 1;
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                buf[w][q][t] = v0[q];
                if (two) buf[w][q][e1] = v1[q];
            }
            if (p < i1) load(p + 1);
            __syncthreads();  // (the other buffer is read until the next one)
            plane(p, p > i0, j0, k0, w);
        }
        __syncthreads();
    }
}

// A warp's list of nodes for the FP64 form.
struct WarpList {
    int* slot;  // 64 entries in shared memory
    int n;
    // adds node c of the lanes with `on`, in lane order
    __device__ __forceinline__ void add(bool on, int c) {
        const unsigned b = __ballot_sync(0xffffffffu, on);
        if (on) slot[RC_OFF(n + __popc(b & ((1u << (threadIdx.x & 31)) - 1)), 64, 404)] = c;
        n += __popc(b);
        __syncwarp();
    }
    // takes up to 32 nodes off the end; -1 in lanes without one
    __device__ __forceinline__ int take() {
        const int lane = threadIdx.x & 31, have = min(n, 32);
        const int c = lane < have ? slot[RC_OFF(n - have + lane, 64, 405)] : -1;
        n -= have;
        __syncwarp();
        return c;
    }
};

// Source of App. A Eq. (elliptic) before smoothing, t = Sigma + C + E with
// Sigma = 1 - m, C(lambda0) the compression limiter of the triad
// e = I + Hess phi and E = -2 H(sqrt_g - v_m) |Sigma| the expansion limiter, at
// one node in FP64.  lambda0 only matters where it is below xi_m (for the soft
// and step readings C vanishes above it).  *wide: set to 1 where a second difference
// of phi, or four times a mixed one, reaches 448 (or is not finite), by the upper
// words, without FP64 work; the displacements of the step know them modulo 1024 only.
__device__ __noinline__ double source64(const Dims& d, const SourceParams& sp, const double* __restrict__ phi,
                                        const double* __restrict__ m, int c, int* wide) {
    int i, j, k;
    cell_coords(d, c, i, j, k);
    Sym3 e = hessian(d, phi, i, j, k);
    auto upper = [](double x) { return __double2hiint(x) & 0x7fffffff; };
    const int diag = max(upper(e.xx), max(upper(e.yy), upper(e.zz)));
    const int mixed = max(upper(e.xy), max(upper(e.xz), upper(e.yz)));
    if (diag >= 0x407c0000 || mixed >= 0x405c0000) *wide = 1;  // 448 and 112
    e.xx += 1.0, e.yy += 1.0, e.zz += 1.0;
    const double g = det3(e);
    double C = 0.0;
    const double gersh =
        fmin(fmin(e.xx - fabs(e.xy) - fabs(e.xz), e.yy - fabs(e.xy) - fabs(e.yz)),
             e.zz - fabs(e.xz) - fabs(e.yz));
    if (sp.climiter == 1 || gersh < sp.xi_m) C = climit(sp.climiter, sp.xi_m, min_eig_sym3(e));
    const double Sigma = 1.0 - m[c];
    const double E = g - sp.v_m > 0.0 ? -2.0 * fabs(Sigma) : 0.0;
    return Sigma + C + E;
}

// C = E = 0 where FP32 certifies that every eigenvalue of e exceeds xi_m
// (Sylvester's criterion) and, e being positive definite then, that its trace
// stays below 3 v_m^(1/3) (det e <= (tr e / 3)^3) and below 100, which bounds
// every entry; the FP64 form looks for wide nodes among the others.  pwide: 1
// where there is one.
template <int GK>
__global__ void __launch_bounds__(GT, GPERSM) k_source_stream(Dims d, SourceParams sp, float trace_max,
                                                                  const double* __restrict__ phi,
                                                                  const float* __restrict__ phi32,
                                                                  const double* __restrict__ m,
                                                                  double* __restrict__ t,
                                                                  double* __restrict__ psum,
                                                                  double* __restrict__ pwide) {
    constexpr int GPK = Tile<GK>::PK;
    __shared__ float buf[2][1][Tile<GK>::N];
    __shared__ int list[GT / 32][64];
    const int lj = threadIdx.x / GK, lk = threadIdx.x % GK;
    const int own = Tile<GK>::own();
    const float xi = (float)sp.xi_m * (1.f + 4.f * kU);  // not below xi_m
    WarpList todo{list[threadIdx.x / 32], 0};
    Column32<GPK> col{};
    double s = 0.0;
    __shared__ int wide;
    if (threadIdx.x == 0) wide = 0;  // (a barrier comes before the first node)
    auto exact = [&] {
        const int c = todo.take();
        if (c >= 0) {
            const double v = source64(d, sp, phi, m, c, &wide);
            t[c] = v;
            s += v;
        }
    };
    const float* const fields[1] = {phi32};
    stream_planes<GK, 1>(
        d, fields, buf, [&] { col = Column32<GPK>{}; },
        [&](int p, bool done, int j0, int k0, int w) {
            float gy, gz;
            const int c = done ? cell_index(d, p - 1, j0 + lj, k0 + lk) : 0;
            const double mass = done ? m[c] : 0.0;
            const Hess32 h = col.feed(buf[w][0] + own, gy, gz);
            if (!done) return;
            const float xx = 1.f + h.xx, yy = 1.f + h.yy, zz = 1.f + h.zz;
            const float big = fmaxf(fmaxf(fabsf(xx), fabsf(yy)), fabsf(zz));
            const float eps = 32.0f * kU * h.vmax + 4.0f * kU * (big + 1.0f);
            const bool plain = sp.climiter != 1 && sylvester32(xx, yy, zz, h.xy, h.xz, h.yz, xi, eps) > 0 &&
                               (xx + yy) + zz + 4.f * eps < trace_max;
            if (plain) {
                const double v = 1.0 - mass;
                t[c] = v;
                s += v;
            }
            todo.add(!plain, c);
            if (todo.n >= 32) exact();
        });
    while (todo.n > 0) exact();
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) put_partial(psum, s, kRedBlocks), put_partial(pwide, wide ? 1.0 : 0.0, kRedBlocks);
}

// Any grid, every node in FP64.
__global__ void k_source_node(Dims d, SourceParams sp, const double* __restrict__ phi,
                              const double* __restrict__ m, double* __restrict__ t, double* __restrict__ psum,
                              double* __restrict__ pwide) {
    double s = 0.0;
    __shared__ int wide;
    if (threadIdx.x == 0) wide = 0;
    __syncthreads();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells; c += gridDim.x * blockDim.x) {
        const double v = source64(d, sp, phi, m, c, &wide);
        t[c] = v;
        s += v;
    }
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) psum[blockIdx.x] = s, pwide[blockIdx.x] = wide ? 1.0 : 0.0;
}

// Step limiter at one node in FP64: the smallest k in [0, kmax] with
// lambda_min(I + Hess phi + 2^-k Hess dphi) > floor, kmax + 1 if none.
__device__ __noinline__ int limiter64(const Dims& d, const LimiterParams& lp, const double* __restrict__ phi,
                                      const double* __restrict__ dphi, int c) {
    int i, j, k;
    cell_coords(d, c, i, j, k);
    Sym3 e = hessian(d, phi, i, j, k);
    e.xx += 1.0, e.yy += 1.0, e.zz += 1.0;
    const Sym3 h = hessian(d, dphi, i, j, k);
    double al = 1.0;
    for (int q = 0; q <= lp.kmax; ++q, al *= 0.5) {
        Sym3 M;
        M.xx = e.xx + al * h.xx, M.yy = e.yy + al * h.yy, M.zz = e.zz + al * h.zz;
        M.xy = e.xy + al * h.xy, M.xz = e.xz + al * h.xz, M.yz = e.yz + al * h.yz;
        if (pd_above(M, lp.lambda_floor)) return q;
    }
    return lp.kmax + 1;
}

// twice the largest |central difference| of dphi at node c
__device__ inline double gradient64(const Dims& d, const double* __restrict__ dphi, int i, int j, int k) {
    const double gx = dphi[cell_index(d, i + 1, j, k)] - dphi[cell_index(d, i - 1, j, k)];
    const double gy = dphi[cell_index(d, i, j + 1, k)] - dphi[cell_index(d, i, j - 1, k)];
    const double gz = dphi[cell_index(d, i, j, k + 1)] - dphi[cell_index(d, i, j, k - 1)];
    return fmax(fabs(gx), fmax(fabs(gy), fabs(gz)));
}

// The Hessian of an FP32 field at one node (Column32's values from memory) and
// twice its gradient.
__device__ inline Hess32 hess32_at(const Dims& d, const float* __restrict__ f, int i, int j, int k, float& gx,
                                   float& gy, float& gz) {
    auto at = [&](int a, int b, int c) { return f[cell_index(d, i + a, j + b, k + c)]; };
    Hess32 h;
    const float c = at(0, 0, 0);
    h.vmax = fabsf(c);
    auto second = [&](float p, float m, float& g) {
        h.vmax = fmaxf(h.vmax, fmaxf(fabsf(p), fabsf(m)));
        g = p - m;
        return (p - 2.f * c) + m;
    };
    auto mixed = [&](float pp, float pm, float mp, float mm) {
        h.vmax = fmaxf(fmaxf(h.vmax, fmaxf(fabsf(pp), fabsf(pm))), fmaxf(fabsf(mp), fabsf(mm)));
        return 0.25f * ((pp - pm) - (mp - mm));
    };
    h.xx = second(at(1, 0, 0), at(-1, 0, 0), gx);
    h.yy = second(at(0, 1, 0), at(0, -1, 0), gy);
    h.zz = second(at(0, 0, 1), at(0, 0, -1), gz);
    h.xy = mixed(at(1, 1, 0), at(1, -1, 0), at(-1, 1, 0), at(-1, -1, 0));
    h.xz = mixed(at(1, 0, 1), at(1, 0, -1), at(-1, 0, 1), at(-1, 0, -1));
    h.yz = mixed(at(0, 1, 1), at(0, 1, -1), at(0, -1, 1), at(0, -1, -1));
    return h;
}

// Step limiter: the largest over the nodes of the smallest k in [0, kmax] with
// lambda_min(e + 2^-k Hess dphi) > floor (kmax + 1 if none), and max_a |central
// grad_a dphi|.  A node that passes at the largest k its warp has found so far
// does not change the result, and where it fails FP32 finds its own k, unless a
// verdict on the way is open (then the FP64 form does).  The gradient's maximum is FP64 too: a node
// is evaluated only where FP32 does not show it to be below the largest value
// its warp has found.  Every lane of a warp takes part in each call.
struct LimiterScreen {
    int kk = 0;            // the warp's largest k so far, and 2^-kk
    float al = 1.f;
    double gm = 0.0;       // this lane's largest |2 G|
    float gw = 0.f;        // the warp's, rounded down

    __device__ __forceinline__ void raise(int k) {
        kk = max(kk, __reduce_max_sync(0xffffffffu, k));
        al = kk < 126 ? __int_as_float((127 - kk) << 23) : 0.f;
    }
    // g: FP32's largest |difference| (within 8 u vmax of the FP64 one, exact())
    template <typename Exact>
    __device__ __forceinline__ void gradient(float g, float vmax, Exact&& exact) {
        const bool higher = !(g + 8.f * kU * vmax < gw);
        if (__any_sync(0xffffffffu, higher)) {
            if (higher) gm = fmax(gm, exact());
            float f = __double2float_rd(gm);
            for (int o = 16; o > 0; o >>= 1) f = fmaxf(f, __shfl_xor_sync(0xffffffffu, f, o));
            gw = f;
        }
    }
    // a node's Hessians of phi and dphi; returns whether the FP64 form has to
    // find its k
    __device__ __forceinline__ bool node(const LimiterParams& lp, float floor32, const Hess32& a, const Hess32& b) {
        // FP32's verdict at step length l: the entries' error is that of
        // the inputs and Hessians, then of the two additions forming M
        auto verdict = [&](float l) {
            const float mxx = 1.0f + a.xx + l * b.xx, myy = 1.0f + a.yy + l * b.yy;
            const float mzz = 1.0f + a.zz + l * b.zz, mxy = a.xy + l * b.xy;
            const float mxz = a.xz + l * b.xz, myz = a.yz + l * b.yz;
            const float big = fmaxf(fmaxf(fabsf(mxx), fabsf(myy)),
                                    fmaxf(fabsf(mzz), fmaxf(fabsf(mxy), fmaxf(fabsf(mxz), fabsf(myz)))));
            const float eps = 32.0f * kU * (a.vmax + l * b.vmax) + 4.0f * kU * (big + 1.0f);
            return sylvester32(mxx, myy, mzz, mxy, mxz, myz, floor32, eps);
        };
        bool unsure = false;
        if (kk <= lp.kmax) {
            const bool passes = verdict(al) > 0;
            if (__any_sync(0xffffffffu, !passes)) {
                int k = 0;
                if (!passes) {  // the node's own k, as far as FP32 tells
                    float l = 1.f;
                    int v = -1;
                    for (; k <= lp.kmax && (v = verdict(l)) < 0; ++k) l *= 0.5f;
                    unsure = v == 0;
                }
                raise(unsure ? 0 : k);
            }
        }
        return unsure;
    }
    // the block's partials
    __device__ __forceinline__ void put(double* pk, double* pg) {
        const double k = block_reduce<OpMax>((double)kk);
        const double g = block_reduce<OpMax>(0.5 * gm);
        if (threadIdx.x == 0) put_partial(pk, k, kRedBlocks), put_partial(pg, g, kRedBlocks);
    }
};

template <int GK>
__global__ void __launch_bounds__(GT, GPERSM) k_limiter_stream(Dims d, LimiterParams lp,
                                                                   const double* __restrict__ phi,
                                                                   const double* __restrict__ dphi,
                                                                   const float* __restrict__ phi32,
                                                                   const float* __restrict__ dphi32,
                                                                   double* __restrict__ pk,
                                                                   double* __restrict__ pg) {
    constexpr int GPK = Tile<GK>::PK;
    __shared__ float buf[2][2][Tile<GK>::N];
    __shared__ int list[GT / 32][64];
    const int lj = threadIdx.x / GK, lk = threadIdx.x % GK;
    const int own = Tile<GK>::own();
    const float floor32 = (float)lp.lambda_floor;
    WarpList todo{list[threadIdx.x / 32], 0};
    Column32<GPK> A{}, B{};
    LimiterScreen screen;
    auto exact = [&] {
        const int c = todo.take();
        screen.raise(c >= 0 ? limiter64(d, lp, phi, dphi, c) : 0);
    };
    const float* const fields[2] = {phi32, dphi32};
    stream_planes<GK, 2>(
        d, fields, buf, [&] { A = Column32<GPK>{}, B = Column32<GPK>{}; },
        [&](int p, bool done, int j0, int k0, int w) {
            float gy, gz, ay, az;
            const Hess32 a = A.feed(buf[w][0] + own, ay, az);
            const Hess32 b = B.feed(buf[w][1] + own, gy, gz);
            if (!done) return;
            const int c = cell_index(d, p - 1, j0 + lj, k0 + lk);
            const float g = fmaxf(fabsf(B.gx), fmaxf(fabsf(gy), fabsf(gz)));
            screen.gradient(g, b.vmax, [&] { return gradient64(d, dphi, p - 1, j0 + lj, k0 + lk); });
            todo.add(screen.node(lp, floor32, a, b), c);
            if (todo.n >= 32) exact();
        });
    while (todo.n > 0) exact();
    screen.put(pk, pg);
}

// Any grid, a thread a node from memory (whole warps have nodes or none: the
// cells are a multiple of 32).  1024 x 512 x 8: 577 us with the FP64 form at
// every node, 66 with this screen.
__global__ void k_limiter_node(Dims d, LimiterParams lp, const double* __restrict__ phi,
                               const double* __restrict__ dphi, const float* __restrict__ phi32,
                               const float* __restrict__ dphi32, double* __restrict__ pk,
                               double* __restrict__ pg) {
    const float floor32 = (float)lp.lambda_floor;
    LimiterScreen screen;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells; c += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_coords(d, c, i, j, k);
        float gx, gy, gz, ax, ay, az;
        const Hess32 a = hess32_at(d, phi32, i, j, k, ax, ay, az);
        const Hess32 b = hess32_at(d, dphi32, i, j, k, gx, gy, gz);
        screen.gradient(fmaxf(fabsf(gx), fmaxf(fabsf(gy), fabsf(gz))), b.vmax,
                        [&] { return gradient64(d, dphi, i, j, k); });
        const bool unsure = screen.node(lp, floor32, a, b);
        if (__any_sync(0xffffffffu, unsure)) screen.raise(unsure ? limiter64(d, lp, phi, dphi, c) : 0);
    }
    screen.put(pk, pg);
}

// The outputs of one node in FP64.  Not inlined, so that the fields and the
// closing statistics come from the same instructions.
__device__ __noinline__ double det64(const Sym3& e) { return det3(e); }
__device__ __noinline__ double lambda64(const Sym3& e) { return min_eig_sym3(e); }
__device__ __noinline__ Sym3 triad64(const Dims& d, const double* __restrict__ phi, int i, int j, int k) {
    Sym3 e = hessian(d, phi, i, j, k);
    e.xx += 1.0, e.yy += 1.0, e.zz += 1.0;
    return e;
}
// delta_r = -lap f with the 7-point Laplacian.
__device__ __noinline__ double delta_r_at(const Dims& d, const double* __restrict__ f, int i, int j, int k) {
    const double p = f[cell_index(d, i, j, k)];
    return -((f[cell_index(d, i + 1, j, k)] - 2.0 * p + f[cell_index(d, i - 1, j, k)]) +
             (f[cell_index(d, i, j + 1, k)] - 2.0 * p + f[cell_index(d, i, j - 1, k)]) +
             (f[cell_index(d, i, j, k + 1)] - 2.0 * p + f[cell_index(d, i, j, k - 1)]));
}


__global__ void k_delta_r(Dims d, const double* __restrict__ phi, double* __restrict__ out,
                          double* __restrict__ pmax) {
    double mx = -INFINITY;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells; c += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_coords(d, c, i, j, k);
        const double v = delta_r_at(d, phi, i, j, k);
        out[c] = v;
        mx = fmax(mx, v);
    }
    mx = block_reduce<OpMax>(mx);
    if (threadIdx.x == 0) pmax[blockIdx.x] = mx;
}

__global__ void k_geometry_out(Dims d, const double* __restrict__ phi, double* __restrict__ det,
                               double* __restrict__ lam, double* __restrict__ pdet,
                               double* __restrict__ plam) {
    double md = INFINITY, ml = INFINITY;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells; c += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_coords(d, c, i, j, k);
        const Sym3 e = triad64(d, phi, i, j, k);
        const double g = det64(e);
        if (det) det[c] = g;
        md = fmin(md, g);
        // lambda0 >= the Gershgorin bound, so without a per-node output the
        // eigenvalue is needed only where that bound is below the running min
        const double gersh =
            fmin(fmin(e.xx - fabs(e.xy) - fabs(e.xz), e.yy - fabs(e.xy) - fabs(e.yz)),
                 e.zz - fabs(e.xz) - fabs(e.yz));
        if (lam || gersh < ml) {
            const double l = lambda64(e);
            if (lam) lam[c] = l;
            ml = fmin(ml, l);
        }
    }
    md = block_reduce<OpMin>(md);
    if (threadIdx.x == 0) pdet[blockIdx.x] = md;
    ml = block_reduce<OpMin>(ml);
    if (threadIdx.x == 0) plam[blockIdx.x] = ml;
}

// The solve's closing statistics: min det e, min lambda0 and max delta_r, each
// the FP64 value of the node that attains it.  The first pass (EXACT = false)
// bounds them from FP32 values (the smallest upper bounds, the largest lower
// one), the second evaluates in FP64 the nodes that the bounds leave open.
// Bound by instruction issue (79% of the slots).  512^3: 26 -> 2.0 ms for all
// three (FP64 at every node, 23 of them for det and lambda0).
template <int GK, bool EXACT>
__global__ void __launch_bounds__(GT, GPERSM) k_extrema_stream(Dims d, const double* __restrict__ phi,
                                                                   const float* __restrict__ phi32,
                                                                   const double* __restrict__ bounds,
                                                                   double* __restrict__ pdet,
                                                                   double* __restrict__ plam,
                                                                   double* __restrict__ pdr) {
    constexpr int GPK = Tile<GK>::PK;
    __shared__ float buf[2][1][Tile<GK>::N];
    const int lj = threadIdx.x / GK, lk = threadIdx.x % GK;
    const int own = Tile<GK>::own();
    const float bd = EXACT ? __double2float_ru(bounds[0]) : 0.f, bl = EXACT ? __double2float_ru(bounds[1]) : 0.f,
                br = EXACT ? __double2float_rd(bounds[2]) : 0.f;
    Column32<GPK> col{};
    float fd = INFINITY, fl = INFINITY, fr = -INFINITY;
    double md = INFINITY, ml = INFINITY, mr = -INFINITY;
    const float* const fields[1] = {phi32};
    stream_planes<GK, 1>(
        d, fields, buf, [&] { col = Column32<GPK>{}; },
        [&](int p, bool done, int j0, int k0, int w) {
            float gy, gz;
            const Hess32 h = col.feed(buf[w][0] + own, gy, gz);
            if (!done) return;
            const float xx = 1.f + h.xx, yy = 1.f + h.yy, zz = 1.f + h.zz;
            const float big = fmaxf(fmaxf(fmaxf(fabsf(xx), fabsf(yy)), fabsf(zz)),
                                    fmaxf(fabsf(h.xy), fmaxf(fabsf(h.xz), fabsf(h.yz))));
            const float eps = 32.0f * kU * h.vmax + 4.0f * kU * (big + 1.0f);
            const float det = xx * (yy * zz - h.yz * h.yz) - h.xy * (h.xy * zz - h.yz * h.xz) +
                              h.xz * (h.xy * h.yz - yy * h.xz);
            const float ed = 9.0f * eps * big * big + 3.0f * eps * eps * big + eps * eps * eps +
                             72.0f * kU * big * big * big;
            float el;
            const float lam = lambda32(h.xx, h.yy, h.zz, h.xy, h.xz, h.yz, big, eps, el);
            const float dr = -(h.xx + h.yy + h.zz), er = 3.f * eps + 8.f * kU * (big + 1.f);
            if (!EXACT) {
                fd = fminf(fd, det + ed), fl = fminf(fl, lam + el), fr = fmaxf(fr, dr - er);
            } else {
                const bool od = !(det - ed > bd), ol = !(lam - el > bl), orr = !(dr + er < br);
                if (od || ol || orr) {
                    const int i = p - 1, j = j0 + lj, k = k0 + lk;
                    const Sym3 e = triad64(d, phi, i, j, k);
                    md = fmin(md, det64(e));
                    if (ol) ml = fmin(ml, lambda64(e));
                    if (orr) mr = fmax(mr, delta_r_at(d, phi, i, j, k));
                }
            }
        });
    md = block_reduce<OpMin>(EXACT ? md : (double)fd);
    ml = block_reduce<OpMin>(EXACT ? ml : (double)fl);
    mr = block_reduce<OpMax>(EXACT ? mr : (double)fr);
    if (threadIdx.x == 0)
        for (int b = blockIdx.x, first = 1; b < kRedBlocks; b += gridDim.x, first = 0) {
            pdet[b] = first ? md : INFINITY, plam[b] = first ? ml : INFINITY, pdr[b] = first ? mr : -INFINITY;
        }
}

// The triad e = I + Hess phi (6 x cells: xx, yy, zz, xy, xz, yz), for the
// adjoint and App. A's density update.
__global__ void k_triad(Dims d, const double* __restrict__ phi, double* __restrict__ e6) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const Sym3 e = hessian(d, phi, i, j, k);
    const size_t n = (size_t)d.cells;
    e6[c] = 1.0 + e.xx, e6[n + c] = 1.0 + e.yy, e6[2 * n + c] = 1.0 + e.zz;
    e6[3 * n + c] = e.xy, e6[4 * n + c] = e.xz, e6[5 * n + c] = e.yz;
}

// The tile's nodes along k on this grid (0: none fits).
int tile_k(const Dims& d) {
    return d.n2 % 32 == 0 && d.n1 % 8 == 0 ? 32 : d.n2 % 16 == 0 && d.n1 % 16 == 0 ? 16 : 0;
}

}  // namespace

int bounds_fail_screened() { return bounds_fail_take(); }

void launch_source(const Dims& d, const SourceParams& sp, const double* phi, const float* phi32, const double* m,
                   double* t, double* part_sum, double* part_wide, cudaStream_t st) {
    launch_counter()++;
    if (const int tk = tile_k(d)) {
        const float trace_max = (float)fmin(100.0, 3.0 * cbrt(sp.v_m) * (1.0 - 1e-5));
        auto fn = tk == 32 ? k_source_stream<32> : k_source_stream<16>;
        fn<<<GBLOCKS, GT, 0, st>>>(d, sp, trace_max, phi, phi32, m, t, part_sum, part_wide);
        return;
    }
    k_source_node<<<kRedBlocks, kRedThreads, 0, st>>>(d, sp, phi, m, t, part_sum, part_wide);
}

void launch_limiter(const Dims& d, const LimiterParams& lp, const double* phi, const double* dphi,
                    const float* phi32, const float* dphi32, double* part_k, double* part_g,
                    cudaStream_t st) {
    launch_counter()++;
    if (const int tk = tile_k(d)) {
        auto fn = tk == 32 ? k_limiter_stream<32> : k_limiter_stream<16>;
        fn<<<GBLOCKS, GT, 0, st>>>(d, lp, phi, dphi, phi32, dphi32, part_k, part_g);
        return;
    }
    k_limiter_node<<<kRedBlocks, kRedThreads, 0, st>>>(d, lp, phi, dphi, phi32, dphi32, part_k, part_g);
}

void launch_delta_r(const Dims& d, const double* phi, double* out, double* part_max,
                    cudaStream_t st) {
    launch_counter()++;
    k_delta_r<<<kRedBlocks, kRedThreads, 0, st>>>(d, phi, out, part_max);
}

void launch_geometry_out(const Dims& d, const double* phi, double* det, double* lam,
                         double* part_min_det, double* part_min_lam, cudaStream_t st) {
    launch_counter()++;
    k_geometry_out<<<kRedBlocks, kRedThreads, 0, st>>>(d, phi, det, lam, part_min_det, part_min_lam);
}

int launch_extrema(const Dims& d, const double* phi, const float* phi32, double* scratch, double* part_det,
                   double* part_lam, double* part_dr, double* scal, cudaStream_t st) {
    const FinishList fin{3, {{part_det, 1, SC_MIN_DET}, {part_lam, 1, SC_MIN_LAM}, {part_dr, 2, SC_MAX_DR}}};
    const int tk = tile_k(d);
    if (tk) {
        static_assert(SC_MIN_LAM == SC_MIN_DET + 1 && SC_MAX_DR == SC_MIN_DET + 2, "the bounds are adjacent");
        launch_counter() += 2;
        auto bound = tk == 32 ? k_extrema_stream<32, false> : k_extrema_stream<16, false>;
        auto exact = tk == 32 ? k_extrema_stream<32, true> : k_extrema_stream<16, true>;
        bound<<<GBLOCKS, GT, 0, st>>>(d, phi, phi32, nullptr, part_det, part_lam, part_dr);
        finish_reduces(fin, scal, st);
        exact<<<GBLOCKS, GT, 0, st>>>(d, phi, phi32, scal + SC_MIN_DET, part_det, part_lam,
                                                            part_dr);
    } else {
        launch_geometry_out(d, phi, nullptr, nullptr, part_det, part_lam, st);
        launch_delta_r(d, phi, scratch, part_dr, st);
    }
    finish_reduces(fin, scal, st);
    return tk ? 4 : 3;
}

void launch_triad(const Dims& d, const double* phi, double* e6, cudaStream_t st) {
    launch_counter()++;
    k_triad<<<(d.cells + 255) / 256, 256, 0, st>>>(d, phi, e6);
}

}  // namespace recon
