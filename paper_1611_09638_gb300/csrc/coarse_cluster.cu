// coarse_cluster.cu -- the coarse end of the FP32 V-cycle (App. A's multigrid)
// from a 32^3 level down, in one launch of one thread-block cluster.
//
// A level of 32^3 nodes is too large for one block's shared memory and too
// small to fill the GPU: it is bound by latency, by the barriers between its
// some twenty phases and by what a phase costs one SM.  Here a cluster of kCR
// blocks holds the 32^3 level in registers, and the first block runs the
// 16^3, 8^3 and 4^3 levels alone (a block barrier takes a fraction of a
// cluster barrier, and 4096 nodes are four a thread).
//
// The 32^3 level: a block owns four i-planes, a thread the four nodes of one
// (j, k) column, as two pairs of planes (2Q, 2Q + 1).  One node of a pair is
// red (i + j + k even) and one black, so a thread's red and black values sit
// in registers of their own, every colour phase updates one node of each pair,
// and all neighbours of a red node are the black nodes of the same pair (in
// the columns around it) or of the pair above or below in its own column:
//     (j + k) even: red on plane 2Q, black on 2Q + 1; odd: the other way.
// A phase reads the other colour's values, [pair][j][k] in shared memory,
// without bank conflicts, and stores its own; the values that the next block
// needs are stored straight into that block's shared memory (one a thread),
// before the cluster's hardware barrier that ends the phase.  Coefficients are
// face sums G (a_c + a_n, or the stored face sums of Level::face) and 1 / sum
// G, in registers for the whole launch: u = (sum G u_n - f / hh) / sum G with
// hh = h^-2 / 2 a power of two.
//
// After a full sweep the residual of the black nodes is zero but for rounding,
// so only red nodes are evaluated, and 13 of the 27 points of the full
// weighting carry anything.  A red update does not read the node's own old
// value, so the prolongation is added to black nodes only where a sweep
// follows.  Several V-cycles can run in one launch where the 32^3 level is the
// finest one; its state then stays in registers between them.
//
// One V(1, 1) of a 32^3 level takes 19 us and six in a launch 87 us;
// with every level in distributed shared memory, every node's face sums and
// division in every phase and a cluster barrier after each phase down to 16^3
// a cycle took 30 us.
#include <cooperative_groups.h>

#include "async_copy.cuh"
#include "checked.cuh"
#include "mg_stencil.cuh"
#include "recon_internal.cuh"

namespace cg = cooperative_groups;

namespace recon {

namespace {

constexpr int kCR = 8;              // blocks of the cluster (portable cluster size)
constexpr int kCN = 32;             // edge of the top level
constexpr int kCT = kCN * kCN;      // threads per block: one per (j, k) column
constexpr int kCol = kCN * kCN;     // nodes of a plane of the top level
static_assert(kCN == 4 * kCR, "four planes, two pairs, per block");

// ---- levels held by one block, [i][j][k] -----------------------------------

struct SLev {
    float *gx, *gy, *gz;  // face sums (entry c: the face between c and its +1 neighbour)
    float *rd;            // 1 / sum of a node's six face sums
    float *u, *f, *r;
    float hh, s;          // h^-2 / 2 and its inverse
};

// The t-th node of a colour (0 red, 1 black): consecutive threads take
// consecutive k, the plane of the pair follows from the parity, so that a
// warp's accesses fall into distinct banks.
template <int N>
__device__ __forceinline__ int colour_node(int t, int colour, int& i, int& j, int& k) {
    k = t & (N - 1), j = (t / N) & (N - 1);
    i = 2 * (t / (N * N)) + ((j + k + colour) & 1);
    return (i * N + j) * N + k;
}

template <int N>
struct Nb {
    int xp, xm, yp, ym, zp, zm;
};
template <int N>
__device__ __forceinline__ Nb<N> neighbours(int i, int j, int k) {
    constexpr int m = N - 1;
    Nb<N> b;
    b.xp = (((i + 1) & m) * N + j) * N + k, b.xm = (((i - 1) & m) * N + j) * N + k;
    b.yp = (i * N + ((j + 1) & m)) * N + k, b.ym = (i * N + ((j - 1) & m)) * N + k;
    b.zp = (i * N + j) * N + ((k + 1) & m), b.zm = (i * N + j) * N + ((k - 1) & m);
    return b;
}

template <int N>
__device__ __forceinline__ float off_sum(const SLev& L, int c, const Nb<N>& b) {
    return (L.gx[c] * L.u[b.xp] + L.gx[b.xm] * L.u[b.xm]) + (L.gy[c] * L.u[b.yp] + L.gy[b.ym] * L.u[b.ym]) +
           (L.gz[c] * L.u[b.zp] + L.gz[b.zm] * L.u[b.zm]);
}

template <int N>
__device__ __forceinline__ float face_total(const SLev& L, int c, const Nb<N>& b) {
    return (L.gx[c] + L.gx[b.xm]) + (L.gy[c] + L.gy[b.ym]) + (L.gz[c] + L.gz[b.zm]);
}

// One colour of a sweep.  zero: u = 0 on entry (the red colour of the first
// sweep reads nothing).
template <int N>
__device__ void s_sweep(const SLev& L, int colour, bool zero) {
    for (int t = threadIdx.x; t < N * N * N / 2; t += kCT) {
        int i, j, k;
        const int c = colour_node<N>(t, colour, i, j, k);
        const float o = zero ? 0.f : off_sum<N>(L, c, neighbours<N>(i, j, k));
        L.u[c] = fmaf(-L.s, L.f[c], o) * L.rd[c];
    }
    __syncthreads();
}

// r = f - L u at the nodes of one colour.
template <int N>
__device__ void s_resid(const SLev& L, int colour) {
    for (int t = threadIdx.x; t < N * N * N / 2; t += kCT) {
        int i, j, k;
        const int c = colour_node<N>(t, colour, i, j, k);
        const Nb<N> b = neighbours<N>(i, j, k);
        L.r[c] = L.f[c] - L.hh * (off_sum<N>(L, c, b) - face_total<N>(L, c, b) * L.u[c]);
    }
}

// Full weighting at coarse node (I, J, K) of an N^3 level's residual r.  red:
// only the red nodes carry one (the centre, weight 1/8, and the twelve edges,
// 1/32).
template <int N, typename R>
__device__ __forceinline__ float weighted(R&& r, int I, int J, int K, bool red) {
    const int i = 2 * I, j = 2 * J, k = 2 * K;
    float edges = 0.f;
#pragma unroll
    for (int p = -1; p <= 1; p += 2)
#pragma unroll
        for (int q = -1; q <= 1; q += 2)
            edges += (r(i, j + p, k + q) + r(i + p, j + q, k)) + r(i + p, j, k + q);
    float acc = fmaf(0.125f, r(i, j, k), 0.03125f * edges);
    if (!red) {
        float faces = 0.f, corners = 0.f;
        for (int p = -1; p <= 1; p += 2) {
            faces += (r(i + p, j, k) + r(i, j + p, k)) + r(i, j, k + p);
            for (int q = -1; q <= 1; q += 2) corners += r(i + p, j + q, k - 1) + r(i + p, j + q, k + 1);
        }
        acc += fmaf(0.0625f, faces, 0.015625f * corners);
    }
    return acc;
}

// Bilinear interpolation at fine (j, k) in one plane of a coarse field: the
// four values around it, equal ones where j or k is even, so that no lane
// takes another path than its neighbours.
template <int CN>
__device__ __forceinline__ float in_plane(const float* plane, int j, int k) {
    constexpr int m = CN - 1;
    const int J = (j >> 1) * CN, J1 = (((j + 1) >> 1) & m) * CN, K = k >> 1, K1 = ((k + 1) >> 1) & m;
    return 0.25f * ((plane[J + K] + plane[J + K1]) + (plane[J1 + K] + plane[J1 + K1]));
}

// u += P(uc) at the nodes of one colour of an N^3 level.
template <int N>
__device__ void s_prolong(const SLev& L, const float* uc, int colour) {
    constexpr int cn = N / 2, cm = cn - 1;
    for (int t = threadIdx.x; t < N * N * N / 2; t += kCT) {
        int i, j, k;
        const int c = colour_node<N>(t, colour, i, j, k);
        L.u[c] += 0.5f * (in_plane<cn>(uc + (i >> 1) * (cn * cn), j, k) +
                          in_plane<cn>(uc + (((i + 1) >> 1) & cm) * (cn * cn), j, k));
    }
}

// Sweeps down on a level, and its residual restricted into fc.
template <int N, typename T>
__device__ void s_down(const SLev& L, int nu1, T* fc) {
    if (nu1 == 0)
        for (int c = threadIdx.x; c < N * N * N; c += kCT) L.u[c] = 0.f;
    for (int s = 0; s < nu1; ++s) s_sweep<N>(L, 0, s == 0), s_sweep<N>(L, 1, false);
    if (nu1 == 0) {
        __syncthreads();
        s_resid<N>(L, 1);
    }
    s_resid<N>(L, 0);
    __syncthreads();
    constexpr int cn = N / 2, m = N - 1;
    auto r = [&](int i, int j, int k) { return L.r[((i & m) * N + (j & m)) * N + (k & m)]; };
    for (int c = threadIdx.x; c < cn * cn * cn; c += kCT)
        fc[c] = weighted<N>(r, c / (cn * cn), (c / cn) & (cn - 1), c & (cn - 1), nu1 > 0);
    __syncthreads();
}

template <int N>
__device__ void s_up(const SLev& L, int nu2, const float* uc) {
    if (nu2 == 0) s_prolong<N>(L, uc, 0);
    s_prolong<N>(L, uc, 1);
    __syncthreads();
    for (int s = 0; s < nu2; ++s) s_sweep<N>(L, 0, false), s_sweep<N>(L, 1, false);
}

// A level's coefficient into shared memory by 16-byte copies (waited for by
// s_setup): the three face-sum arrays, or the nodal a (in the place of rd).
template <int N, bool FACE>
__device__ void s_fetch(const SLev& L, const float* a) {
    constexpr int n = N * N * N;
    if (FACE) {
        for (int c = 4 * threadIdx.x; c < 3 * n; c += 4 * kCT) cp_async16(L.gx + c, a + c);  // gx, gy, gz are adjacent
    } else {
        for (int c = 4 * threadIdx.x; c < n; c += 4 * kCT) cp_async16(L.r + c, a + c);
    }
}

template <int N, bool FACE>
__device__ void s_setup(const SLev& L) {
    constexpr int n = N * N * N;
    if (!FACE) {
        for (int c = threadIdx.x; c < n; c += kCT) {
            const Nb<N> b = neighbours<N>(c / (N * N), (c / N) & (N - 1), c & (N - 1));
            L.gx[c] = L.r[c] + L.r[b.xp], L.gy[c] = L.r[c] + L.r[b.yp], L.gz[c] = L.r[c] + L.r[b.zp];
        }
        __syncthreads();
    }
    for (int c = threadIdx.x; c < n; c += kCT)
        L.rd[c] = 1.f / face_total<N>(L, c, neighbours<N>(c / (N * N), (c / N) & (N - 1), c & (N - 1)));
}

constexpr int N1 = kCN / 2, N2 = kCN / 4, N3 = kCN / 8;
static_assert(N3 * N3 * N3 == kNc, "the last level is 4^3");
constexpr int kLev1 = 7 * N1 * N1 * N1, kLev2 = 7 * N2 * N2 * N2;

// Shared memory, in floats: the top level's red and black values and red and
// black residuals ([pair -1 .. 2][column]), four coarse planes, then block 0's
// levels and the 4^3 matrix (16-byte aligned).
constexpr int kTop = 4 * kCol, kTopAll = 4 * kTop, kCoarse = 4 * N1 * N1;
constexpr int kClusterSmem = (kTopAll + kCoarse + kLev1 + kLev2 + kNc) * (int)sizeof(float) +
                             (kNc + 1) * kNc * (int)sizeof(double);
static_assert((kTopAll + kCoarse + kLev1 + kLev2) % 4 == 0, "the 4^3 matrix is 16-byte aligned");
static_assert(kClusterSmem <= 227 * 1024, "shared memory of a block");

// The levels' coefficients and h^-2 / 2 as FP32, formed on the host: an FP64
// operation in each of a block's 1024 threads takes its SM 512 cycles (two
// lanes a clock), and the divisions of a first version took 8 of 28 us.
struct ClusterSet {
    int nu1, nu2;
    float hh[3];
    const float* a[3];
};

template <bool FACE>
__global__ void __cluster_dims__(kCR, 1, 1) __launch_bounds__(kCT)
    k_coarse_cluster(ClusterSet cs, const float* __restrict__ f_top, float* __restrict__ u_top,
                     const double* __restrict__ minv_g, int zero_u, int cycles) {
    cg::cluster_group cluster = cg::this_cluster();
    const int self = (int)cluster.block_rank();
    extern __shared__ __align__(16) float smem[];
    float* sR = smem;             // red values: slot q + 1 holds pair q, slots 0 and 3 the neighbours' pairs
    float* sB = sR + kTop;        // black values
    float* sP = sB + kTop;        // residuals at red nodes
    float* sQ = sP + kTop;        // residuals at black nodes (no sweep before the restriction)
    float* sC = sQ + kTop;        // coarse planes 2 self - 1 .. 2 self + 2 of the 16^3 correction
    SLev L1, L2;
    {
        float* q = sC + kCoarse;
        auto take = [&](SLev& L, int n, float hh) {
            L.gx = q, L.gy = q + n, L.gz = q + 2 * n, L.rd = q + 3 * n;
            L.u = q + 4 * n, L.f = q + 5 * n, L.r = q + 6 * n;
            L.hh = hh, L.s = 1.f / hh;
            q += 7 * n;
        };
        take(L1, N1 * N1 * N1, cs.hh[1]);
        take(L2, N2 * N2 * N2, cs.hh[2]);
    }
    double* minv = reinterpret_cast<double*>(L2.gx + kLev2);
    double* f3 = minv + kNc * kNc;  // (converted once, not in each of the 64 rows)
    float* u3 = reinterpret_cast<float*>(f3 + kNc);

    const int t = threadIdx.x, j = t / kCN, k = t & (kCN - 1);
    const int s0 = (j + k) & 1;
    constexpr int m = kCN - 1;
    const int jp = ((j + 1) & m) * kCN + k, jm = ((j - 1) & m) * kCN + k;
    const int kp = j * kCN + ((k + 1) & m), km = j * kCN + ((k - 1) & m);
    const int prev = (self + kCR - 1) % kCR, next = (self + 1) % kCR;
    // the neighbour that takes this thread's value of a colour, and the slot
    // there: pair 1 goes to the next block's slot 0, pair 0 to the previous
    // one's slot 3.  Red: (j + k) even holds plane 0, odd plane 3.
    // (RC_OFF: checked against the extent in the RECON_CHECKED build)
    const int first = RC_OFF(t, kTop, 302), fourth = RC_OFF(3 * kCol + t, kTop, 303);
    float* const outR = cluster.map_shared_rank(sR, s0 ? next : prev) + (s0 ? first : fourth);
    float* const outB = cluster.map_shared_rank(sB, s0 ? prev : next) + (s0 ? fourth : first);

    if (self == 0) {
        s_fetch<N1, FACE>(L1, cs.a[1]);
        s_fetch<N2, FACE>(L2, cs.a[2]);
        for (int e = 2 * t; e < kNc * kNc; e += 2 * kCT)
            cp_async16(reinterpret_cast<float*>(minv + e), reinterpret_cast<const float*>(minv_g + e));
        cp_commit();
    }
    // ---- the top level's coefficients, right-hand side and first guess
    float gA[2], gRo[2], gBo[2];        // to the pair's other node; from red / black to the next pair
    float gR[2][4], gB[2][4];           // to j + 1, j - 1, k + 1, k - 1
    float rR[2], rB[2], fR[2], fB[2], uR[2], uB[2];
    const float hh = cs.hh[0], sf = 1.f / hh;
    {
        const float* a = cs.a[0];
        constexpr int n = kCN * kCol;
        auto plane = [&](int p) { return RC_OFF(((4 * self + p) & m) * kCol, kCN * kCol - kCol + 1, 306); };
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int pr = plane(2 * q + s0), pb = plane(2 * q + 1 - s0);
            if (FACE) {
                const float *gy = a + n, *gz = a + 2 * n;
                gA[q] = a[plane(2 * q) + t];
                gRo[q] = a[plane(2 * q + (s0 ? 1 : -1)) + t];
                gBo[q] = a[plane(2 * q + (s0 ? -1 : 1)) + t];
                gR[q][0] = gy[pr + t], gR[q][1] = gy[pr + jm], gR[q][2] = gz[pr + t], gR[q][3] = gz[pr + km];
                gB[q][0] = gy[pb + t], gB[q][1] = gy[pb + jm], gB[q][2] = gz[pb + t], gB[q][3] = gz[pb + km];
            } else {
                const float ar = a[pr + t], ab = a[pb + t];
                gA[q] = ar + ab;
                gRo[q] = ar + a[plane(2 * q + (s0 ? 2 : -1)) + t];
                gBo[q] = ab + a[plane(2 * q + (s0 ? -1 : 2)) + t];
                gR[q][0] = ar + a[pr + jp], gR[q][1] = ar + a[pr + jm];
                gR[q][2] = ar + a[pr + kp], gR[q][3] = ar + a[pr + km];
                gB[q][0] = ab + a[pb + jp], gB[q][1] = ab + a[pb + jm];
                gB[q][2] = ab + a[pb + kp], gB[q][3] = ab + a[pb + km];
            }
            rR[q] = 1.f / ((gA[q] + gRo[q]) + (gR[q][0] + gR[q][1]) + (gR[q][2] + gR[q][3]));
            rB[q] = 1.f / ((gA[q] + gBo[q]) + (gB[q][0] + gB[q][1]) + (gB[q][2] + gB[q][3]));
            fR[q] = f_top[pr + t], fB[q] = f_top[pb + t];
            uR[q] = zero_u ? 0.f : u_top[pr + t], uB[q] = zero_u ? 0.f : u_top[pb + t];
        }
    }
    auto put_red = [&] {
        sR[kCol + t] = uR[0], sR[2 * kCol + t] = uR[1];
        *outR = s0 ? uR[1] : uR[0];
    };
    auto put_black = [&] {
        sB[kCol + t] = uB[0], sB[2 * kCol + t] = uB[1];
        *outB = s0 ? uB[0] : uB[1];
    };
    // sum G u_n of the red (black) node of pair q from the other colour's values
    auto off_red = [&](int q) {
        const float* x = sB + (q + 1) * kCol;
        return (gA[q] * uB[q] + gRo[q] * x[(s0 ? kCol : -kCol) + t]) + (gR[q][0] * x[jp] + gR[q][1] * x[jm]) +
               (gR[q][2] * x[kp] + gR[q][3] * x[km]);
    };
    auto off_black = [&](int q) {
        const float* x = sR + (q + 1) * kCol;
        return (gA[q] * uR[q] + gBo[q] * x[(s0 ? -kCol : kCol) + t]) + (gB[q][0] * x[jp] + gB[q][1] * x[jm]) +
               (gB[q][2] * x[kp] + gB[q][3] * x[km]);
    };
    auto sweep = [&](bool zero) {
#pragma unroll
        for (int q = 0; q < 2; ++q) uR[q] = fmaf(-sf, fR[q], zero ? 0.f : off_red(q)) * rR[q];
        put_red();
        cluster.sync();
#pragma unroll
        for (int q = 0; q < 2; ++q) uB[q] = fmaf(-sf, fB[q], off_black(q)) * rB[q];
        put_black();
        cluster.sync();
    };

    if (self == 0) {
        cp_wait_all();
        __syncthreads();
        s_setup<N1, FACE>(L1);
        s_setup<N2, FACE>(L2);
    }
    cluster.sync();  // every block runs before its shared memory is written from outside
    bool zero = zero_u != 0;
    if (!zero || cs.nu1 == 0) {
        put_red();
        put_black();
        cluster.sync();
        zero = false;
    }
    for (int cyc = 0; cyc < cycles; ++cyc) {
        for (int s = 0; s < cs.nu1; ++s) sweep(zero && s == 0);
        zero = false;
        // residuals, [pair][column] like the values; the coarse planes of a
        // block reach into pair -1: red (j + k) odd, black (j + k) even
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const float dr = (gA[q] + gRo[q]) + (gR[q][0] + gR[q][1]) + (gR[q][2] + gR[q][3]);
            const float r = fR[q] - hh * (off_red(q) - dr * uR[q]);
            sP[(q + 1) * kCol + t] = r;
            if (q == 1 && s0) cluster.map_shared_rank(sP, next)[t] = r;
            if (cs.nu1 == 0) {
                const float db = (gA[q] + gBo[q]) + (gB[q][0] + gB[q][1]) + (gB[q][2] + gB[q][3]);
                const float b = fB[q] - hh * (off_black(q) - db * uB[q]);
                sQ[(q + 1) * kCol + t] = b;
                if (q == 1 && !s0) cluster.map_shared_rank(sQ, next)[t] = b;
            }
        }
        cluster.sync();
        if (t < 2 * N1 * N1) {
            const int q = t / (N1 * N1), J = (t / N1) & (N1 - 1), K = t & (N1 - 1);
            // plane p of the block (-1 .. 3): pair p >> 1
            auto r = [&](int p, int jj, int kk) {
                jj &= m, kk &= m;
                const int at = RC_OFF(((p >> 1) + 1) * kCol + jj * kCN + kk, kTop, 304);
                return ((p + jj + kk) & 1) ? sQ[at] : sP[at];
            };
            const float v = weighted<kCN>(r, q, J, K, cs.nu1 > 0);
            cluster.map_shared_rank(L1.f, 0)[RC_OFF((2 * self + q) * (N1 * N1) + J * N1 + K, N1 * N1 * N1, 301)] = v;
        }
        cluster.sync();
        if (self == 0) {
            s_down<N1>(L1, cs.nu1, L2.f);
            s_down<N2>(L2, cs.nu1, f3);
            if (t < 4 * kNc) {  // the 4^3 level: u = M f in FP64, four threads a row
                double acc = 0.0;
                for (int c = t & 3; c < kNc; c += 4) acc = fma(minv[(t >> 2) * kNc + c], f3[c], acc);
                acc += __shfl_xor_sync(0xffffffffu, acc, 1);
                acc += __shfl_xor_sync(0xffffffffu, acc, 2);
                if ((t & 3) == 0) u3[t >> 2] = (float)acc;
            }
            __syncthreads();
            s_up<N2>(L2, cs.nu2, u3);
            s_up<N1>(L1, cs.nu2, L2.u);
        }
        cluster.sync();
        // the 16^3 correction around this block, then u += P of it, on the
        // neighbours' pairs too, so that no exchange is needed
        sC[t] = cluster.map_shared_rank(L1.u, 0)[RC_OFF(
            ((2 * self - 1 + t / (N1 * N1)) & (N1 - 1)) * (N1 * N1) + (t & (N1 * N1 - 1)), N1 * N1 * N1, 305)];
        static_assert(kCoarse == kCT, "one coarse value a thread");
        __syncthreads();
        // interpolated in the coarse planes -1 .. 2, then P on planes -1 .. 4
        float v[4];
#pragma unroll
        for (int I = 0; I < 4; ++I) v[I] = in_plane<N1>(sC + I * (N1 * N1), j, k);
        const float p[6] = {0.5f * (v[0] + v[1]), v[1], 0.5f * (v[1] + v[2]), v[2], 0.5f * (v[2] + v[3]), v[3]};
        // black: planes 0, 2, 4 where j + k is odd, else -1, 1, 3
        uB[0] += s0 ? p[1] : p[2], uB[1] += s0 ? p[3] : p[4];
        sB[kCol + t] = uB[0], sB[2 * kCol + t] = uB[1];
        sB[(s0 ? 3 * kCol : 0) + t] += s0 ? p[5] : p[0];
        if (cs.nu2 == 0) {  // red: the other way
            uR[0] += s0 ? p[2] : p[1], uR[1] += s0 ? p[4] : p[3];
            sR[kCol + t] = uR[0], sR[2 * kCol + t] = uR[1];
            sR[(s0 ? 0 : 3 * kCol) + t] += s0 ? p[0] : p[5];
        }
        // (without a sweep the neighbours' red values were written above, and
        // theirs may come in the next cycle's first phase)
        if (cs.nu2 == 0) cluster.sync();
        else __syncthreads();
        for (int s = 0; s < cs.nu2; ++s) sweep(false);
    }
    {
        auto plane = [&](int p) { return RC_OFF(((4 * self + p) & m) * kCol, kCN * kCol - kCol + 1, 306); };
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            u_top[plane(2 * q + s0) + t] = uR[q];
            u_top[plane(2 * q + 1 - s0) + t] = uB[q];
        }
    }
    // (the last phase above ended with a cluster barrier: no block ends while
    // another may still read or write its shared memory)
}

}  // namespace

bool coarse_cluster_fits(const CoarseSet& cs) {
    if (cs.nlev != 4) return false;
    for (int l = 0; l < 4; ++l) {
        const Level& L = cs.lv[l];
        if (L.face != cs.lv[0].face) return false;  // one form for the whole set
        if (L.h2i[0] != L.h2i[1] || L.h2i[1] != L.h2i[2]) return false;
        const int n = kCN >> l;
        if (L.d.n0 != n || L.d.n1 != n || L.d.n2 != n) return false;
        if (l < 3 && !(L.coarsen[0] && L.coarsen[1] && L.coarsen[2])) return false;
    }
    return true;
}

bool launch_coarse_cluster(const CoarseSet& cs, const float* f, float* u, const double* minv, bool zero_u,
                           int cycles, cudaStream_t st) {
    if (!coarse_cluster_fits(cs)) return false;
    launch_counter()++;
    ClusterSet set{};
    set.nu1 = cs.nu1, set.nu2 = cs.nu2;
    for (int l = 0; l < 3; ++l) set.hh[l] = (float)(0.5 * cs.lv[l].h2i[0]), set.a[l] = (const float*)cs.a[l];
    auto fn = cs.lv[0].face ? k_coarse_cluster<true> : k_coarse_cluster<false>;
    allow_smem((const void*)fn, kClusterSmem);
    fn<<<kCR, kCT, kClusterSmem, st>>>(set, f, u, minv, zero_u ? 1 : 0, cycles);
    return true;
}

int bounds_fail_cluster() { return bounds_fail_take(); }

}  // namespace recon
