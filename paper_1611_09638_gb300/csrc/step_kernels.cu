// step_kernels.cu -- kernels of one moving-mesh step (Sec. II, App. A): CIC
// deposits in 64-bit fixed point, the checks of the inputs, the smoothing
// operator S, the mesh advance, App. A's density update, the mesh positions, and
// the ends of the reductions.  (Source, limiter, triad and the outputs det,
// lambda0 and delta_r: screened.cu; node displacements: displacement.cu.)
#include "fixed_point.cuh"
#include "geometry.cuh"
#include "recon_internal.cuh"
#include "reduce.cuh"

namespace recon {

namespace {

constexpr int kThreads = 256;
inline int nblocks(long long work) { return (int)((work + kThreads - 1) / kThreads); }

// ---------------------------------------------------------------- helpers

// 1 / n for a power of two n (< 2^1023), exactly, from the exponent bits
// (integer work only; x * inv_pow2(n) equals x / n bit for bit).
__device__ inline double inv_pow2(int n) {
    return __longlong_as_double((long long)(1023 - (__ffs(n) - 1)) << 52);
}

// The eight CIC corner charges of one tracer in fixed point.  The offset of
// the tracer from its home node is rounded on each axis to 2^-52 of a cell
// (fixed_axis): the lower node is home + floor and f the fraction in units of
// 2^-52.  The mass M = llrint(w scale) is split exactly,
// first along x into M1 = M f_x / 2^52 rounded to nearest and M0 = M - M1, then each part
// along y, then along z, so the charges are non-negative integers that sum to
// M exactly (mass conservation per tracer).  The splits are 64 x 64-bit
// integer multiplies (upper halves): the FP64 work per tracer is four
// scalings and four conversions, against some 35 FP64 instructions for FP64
// corner weights.  The rounding of a charge is below one unit (1 / scale) of
// the fixed point, like llrint of an FP64 product, and the position's below
// 2^-53 cells, the rounding of an FP64 offset between 1/2 and 1 cell.
struct CicCharges {
    int i0, j0, k0;               // lower corner
    unsigned long long c[2][2][2];  // charges at (i0 + di, j0 + dj, k0 + dk)
};

constexpr int kFracBits = 52;

// The fixed-point position of a tracer along one axis: the offset from its
// home node rounded to 2^-kFracBits of a cell (-2^11 <= off < 2^11), as the lower
// node and the fraction f in [0, 2^kFracBits).  Below 2^10 cells the rounding is
// integer work.
__device__ inline void fixed_axis(int home, double off, int& i0, unsigned long long& f) {
    const bool near = ((int)(__double_as_longlong(off) >> 52) & 0x7ff) < 1023 + 10;
    const long long q = near ? to_fixed(off, kFracBits) : __double2ll_rn(off * 4503599627370496.0);
    i0 = home + (int)(q >> kFracBits);                              // floor
    f = (unsigned long long)q & ((1ull << kFracBits) - 1);
}

// m f / 2^52 rounded to nearest (the upper half of m (f 2^12), plus one where
// the lower half is at least 2^63) and the rest m - that: an exact split
// without a bias toward either side.
__device__ inline void split_fixed(unsigned long long m, unsigned long long f, unsigned long long& lo,
                                   unsigned long long& hi) {
    const unsigned long long y = f << (64 - kFracBits);
    hi = __umul64hi(m, y) + ((m * y) >> 63);
    lo = m - hi;
}

// The split of M over the corners for the fractions fx, fy, fz.
__device__ inline void split_charges(unsigned long long M, unsigned long long fx, unsigned long long fy,
                                     unsigned long long fz, CicCharges& r) {
    unsigned long long mx[2], mxy[2][2];
    split_fixed(M, fx, mx[0], mx[1]);
#pragma unroll
    for (int di = 0; di < 2; ++di) {
        split_fixed(mx[di], fy, mxy[di][0], mxy[di][1]);
#pragma unroll
        for (int dj = 0; dj < 2; ++dj) split_fixed(mxy[di][dj], fz, r.c[di][dj][0], r.c[di][dj][1]);
    }
}

__device__ inline CicCharges cic_charges(int i, int j, int k, double ox, double oy, double oz, double w,
                                         double scale) {
    CicCharges r;
    unsigned long long fx, fy, fz;
    fixed_axis(i, ox, r.i0, fx);
    fixed_axis(j, oy, r.j0, fy);
    fixed_axis(k, oz, r.k0, fz);
    split_charges((unsigned long long)__double2ll_rn(w * scale), fx, fy, fz, r);
    return r;
}


// ---------------------------------------------------------------- kernels

__global__ void k_validate_grid(int cells, const double* __restrict__ rho, double* ps, double* pb) {
    double s = 0.0, bad = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += gridDim.x * blockDim.x) {
        const double v = rho[c];
        if (!(v >= 0.0) || !isfinite(v)) bad = 1.0;
        else s += v;
    }
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) ps[blockIdx.x] = s;
    bad = block_reduce<OpMax>(bad);
    if (threadIdx.x == 0) pb[blockIdx.x] = bad;
}

__global__ void k_validate_particles(int64_t np, const double* __restrict__ pos,
                                     const double* __restrict__ mass, double* ps, double* pb) {
    double s = 0.0, bad = 0.0;
    for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < np;
         p += (int64_t)gridDim.x * blockDim.x) {
        const double x = pos[3 * p], y = pos[3 * p + 1], z = pos[3 * p + 2];
        if (!isfinite(x) || !isfinite(y) || !isfinite(z)) bad = 1.0;
        const double m = mass ? mass[p] : 1.0;
        if (!(m >= 0.0) || !isfinite(m)) bad = 1.0;
        else s += m;
    }
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) ps[blockIdx.x] = s;
    bad = block_reduce<OpMax>(bad);
    if (threadIdx.x == 0) pb[blockIdx.x] = bad;
}

// The scale of the fixed point for a total mass known on the device (total;
// what fixed_scale gives on the host), or the given one.
__device__ inline double deposit_scale(const double* __restrict__ total, double scale) {
    if (!total) return scale;
    const int e = (int)(__double_as_longlong(*total) >> 52) - 1022;  // total < 2^e
    return __longlong_as_double((long long)(1023 + 61 - min(max(e, 1), 1024)) << 52);
}

// bad: null, or set to 1 where a position is not finite (unit masses: such a
// deposit needs no pass over the particles before it).
__global__ void k_deposit_particles(Dims d, int64_t np, const double* __restrict__ pos,
                                    const double* __restrict__ mass, double inv_h, double given,
                                    const double* __restrict__ total, double* __restrict__ bad,
                                    unsigned long long* __restrict__ mfix) {
    const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (bad) {
        const bool off = p < np && !(isfinite(pos[3 * p]) && isfinite(pos[3 * p + 1]) && isfinite(pos[3 * p + 2]));
        if (off) *bad = 1.0;
    }
    const double scale = deposit_scale(total, given);
    // the position as an offset from node 0 (the same integer charges as the
    // tracers'; cell_index wraps it), first wrapped into [0, n) grid units where
    // it is 2^10 cells away or more (x * inv_pow2(n) is x / n exactly), and from
    // there into [-2^11, 2^11), which is what fixed_axis holds (n <= 4096)
    auto wrap = [](double x, int n) {
        if (fabs(x) < 1024.0) return x;
        const double y = x - (double)n * floor(x * inv_pow2(n));
        return y < 2048.0 ? y : y - (double)n;
    };
    CicCharges q{};
    if (p < np) {
        unsigned long long fx, fy, fz;
        fixed_axis(0, wrap(pos[3 * p] * inv_h, d.n0), q.i0, fx);
        fixed_axis(0, wrap(pos[3 * p + 1] * inv_h, d.n1), q.j0, fy);
        fixed_axis(0, wrap(pos[3 * p + 2] * inv_h, d.n2), q.k0, fz);
        const double m = mass ? mass[p] : 1.0;
        split_charges((unsigned long long)__double2ll_rn(m * scale), fx, fy, fz, q);
    }
    // Two lanes add one particle's pair of cells along k, so that an atomic
    // instruction of particles in no order touches half as many sectors, which
    // bound it: 20 million in random order on 256^3 1.43 -> 1.19 ms, one a cell of
    // 512^3 in order 6.6 -> 3.0 ms (4.2 of that with the FP64 wrap and scalings
    // left out).
    const int lane = threadIdx.x & 31, dk = lane & 1;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const int src = (lane >> 1) + 16 * s;
        const int i0 = __shfl_sync(0xffffffffu, q.i0, src), j0 = __shfl_sync(0xffffffffu, q.j0, src);
        const int k = __shfl_sync(0xffffffffu, q.k0, src) + dk;
#pragma unroll
        for (int di = 0; di < 2; ++di)
#pragma unroll
            for (int dj = 0; dj < 2; ++dj) {
                const unsigned long long a = __shfl_sync(0xffffffffu, q.c[di][dj][0], src);
                const unsigned long long b = __shfl_sync(0xffffffffu, q.c[di][dj][1], src);
                const unsigned long long v = dk ? b : a;
                if (v) atomicAdd(&mfix[cell_index(d, i0 + di, j0 + dj, k)], v);
            }
    }
}

// 1 / 2^n of a power of two by its exponent bits.
__device__ inline double inv_of_pow2(double x) {
    return __longlong_as_double((2046ll << 52) - __double_as_longlong(x));
}

__global__ void k_fix_to_double(int cells, unsigned long long* __restrict__ mfix, double given,
                                const double* __restrict__ total, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cells) return;
    const double inv_scale = inv_of_pow2(deposit_scale(total, given));
    out[c] = (double)(long long)mfix[c] * inv_scale;
    mfix[c] = 0ull;
}

// The same with the sum of the density and the checks of k_validate_grid, for
// grids of at most 2^20 cells: one launch instead of two (64^3: 2.5 us of a 69 us
// deposit); on larger grids the two passes are faster (256^3: 116 us against
// 181).
__global__ void k_fix_validate(int cells, unsigned long long* __restrict__ mfix, double given,
                               const double* __restrict__ total, double* __restrict__ out, double* ps, double* pb) {
    double s = 0.0, bad = 0.0;
    const double inv_scale = inv_of_pow2(deposit_scale(total, given));
    const int stride = gridDim.x * blockDim.x;
    auto one = [&](int c, long long q) {
        const double v = (double)q * inv_scale;
        mfix[c] = 0ull;
        out[c] = v;
        if (q < 0) bad = 1.0;
        else s += v;
    };
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    for (; c < cells; c += stride) one(c, (long long)mfix[c]);
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) ps[blockIdx.x] = s;
    bad = block_reduce<OpMax>(bad);
    if (threadIdx.x == 0) pb[blockIdx.x] = bad;
}

__global__ void k_init_tracers(int cells, const double* __restrict__ rho,
                               const double* __restrict__ sum_rho,
                               double* __restrict__ w, double* __restrict__ ox,
                               double* __restrict__ oy, double* __restrict__ oz,
                               double* __restrict__ phi, float* __restrict__ phi32) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    __shared__ double inv;  // (a division in every thread bound this kernel: 512^3 3.54 -> 1.00 ms)
    if (threadIdx.x == 0) inv = 1.0 / (*sum_rho / (double)cells);
    __syncthreads();
    if (c >= cells) return;
    const double inv_rho_bar = inv;
    w[c] = rho[c] * inv_rho_bar;
    ox[c] = 0.0, oy[c] = 0.0, oz[c] = 0.0;
    phi[c] = 0.0;
    phi32[c] = 0.0f;
}

// Deposit of the tracers on the deformed mesh: tracer c (home node c, mass
// w_c) sits at curvilinear coordinate c + offset.  Neighbouring tracers stay
// neighbours, so a warp's atomics fall into few sectors of L2, which adds them
// faster than tiles accumulated in shared memory first: 512^3 1.69 ms against
// 2.70, 256^3 223 us against 352, 128^3 34 against 77, 32^3 (8 tiles) 3.0 against 33.
__global__ void k_deposit_tracers(Dims d, const double* __restrict__ ox,
                                  const double* __restrict__ oy, const double* __restrict__ oz,
                                  const double* __restrict__ w, double scale,
                                  unsigned long long* __restrict__ mfix) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const CicCharges q = cic_charges(i, j, k, ox[c], oy[c], oz[c], w[c], scale);
    for (int di = 0; di < 2; ++di)
        for (int dj = 0; dj < 2; ++dj)
            for (int dk = 0; dk < 2; ++dk)
                atomicAdd(&mfix[cell_index(d, q.i0 + di, q.j0 + dj, q.k0 + dk)], q.c[di][dj][dk]);
}

// m from the fixed-point accumulator (which is cleared for the next deposit),
// coefficient a = max(m, a_min) in FP64 and FP32, and partial sums of m.
__global__ void k_mass_coef(int cells, unsigned long long* __restrict__ mfix, double inv_scale,
                            double a_min, double* __restrict__ m, double* __restrict__ a64,
                            float* __restrict__ a32, double* __restrict__ part) {
    double s = 0.0;
    const int stride = gridDim.x * blockDim.x;
    auto one = [&](int c, long long q) {
        const double v = (double)q * inv_scale;
        mfix[c] = 0ull;
        m[c] = v;
        const double a = v > a_min ? v : a_min;
        a64[c] = a;
        if (a32) a32[c] = (float)a;
        s += v;
    };
    int c = blockIdx.x * blockDim.x + threadIdx.x;
    // four loads in flight per thread; the nodes are summed in the same order
    for (; c + 3 * stride < cells; c += 4 * stride) {
        long long q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = (long long)mfix[c + u * stride];
#pragma unroll
        for (int u = 0; u < 4; ++u) one(c + u * stride, q[u]);
    }
    for (; c < cells; c += stride) one(c, (long long)mfix[c]);
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// One axis of the smoothing operator S (a weighted mean over the 3x3x3
// neighbourhood, separable into (w, 1-2w, w) along each axis): out =
// w in[-1] + (1-2w) in[0] + w in[+1] along `axis`, minus (*shift_sum / cells)
// when shift_sum is given; optional per-block sums of out and out^2.  Three
// passes (k, j, i) cost 9 FP64 instructions per node against 27 for the
// direct 27-point sum.
__global__ void k_smooth_axis(Dims d, int axis, double ws, const double* __restrict__ in,
                              const double* __restrict__ shift_sum, double* __restrict__ out,
                              float* __restrict__ out32, double* __restrict__ psum,
                              double* __restrict__ psq) {
    const double w1 = 1.0 - 2.0 * ws;
    const double shift = shift_sum ? *shift_sum / (double)d.cells : 0.0;
    const int di = axis == 0, dj = axis == 1, dk = axis == 2;
    double s = 0.0, q = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < d.cells; c += gridDim.x * blockDim.x) {
        int i, j, k;
        cell_coords(d, c, i, j, k);
        const double v = fma(ws, in[cell_index(d, i - di, j - dj, k - dk)] +
                                     in[cell_index(d, i + di, j + dj, k + dk)],
                             w1 * in[c]) - shift;
        out[c] = v;
        if (out32) out32[c] = (float)v;
        s += v;
        q = fma(v, v, q);
    }
    if (psum) {
        s = block_reduce<OpSum>(s);
        if (threadIdx.x == 0) psum[blockIdx.x] = s;
    }
    if (psq) {
        q = block_reduce<OpSum>(q);
        if (threadIdx.x == 0) psq[blockIdx.x] = q;
    }
}

// S in one pass.  A block takes an SJ x SK tile of the (j, k) plane, a warp a
// row and a lane a node of it, and streams planes along i: a plane is smoothed
// along k by warp shuffles, along j through shared memory, and along i from
// the last two planes' values, which each thread keeps in registers.  The
// planes of all tiles form one sequence that the blocks split evenly, so that
// small grids use as many blocks as they have planes; a piece that starts
// inside a tile's column first smooths the plane before it.  The grid is one
// round of resident blocks, six per SM (at kRedBlocks, 1.33 rounds, a third of
// the FP64 issue slots stayed empty).
//
// Bound by the FP64 rate (2 lanes a clock and SM).  QUARTER (side weight 1/4,
// the default): a + 2 b + c per axis and one exact factor 1/64 at the end, 2
// instructions an axis instead of 3.  SUM: the FP32 copy and the sum; SQ: the
// sum of squares.  512^3: 3.87 -> 2.87 ms (FP64 pipe 72% busy), 32^3 (8 blocks in the
// former split): 36.5 -> 9.8 us.
constexpr int SJ = 8, SK = 32;
constexpr int kSPerSM = 6, kSBlocks = kSPerSM * (kRedBlocks / 8);

template <bool QUARTER, bool SUM, bool SQ>
__global__ void __launch_bounds__(SJ* SK, kSPerSM) k_smooth_S_stream(
    Dims d, double ws, const double* __restrict__ in, const double* __restrict__ shift_sum,
    double* __restrict__ out, float* __restrict__ out32, double* __restrict__ part) {
    __shared__ double sk[2][SJ + 2][SK];  // planes smoothed along k
    const double w1 = 1.0 - 2.0 * ws;
    const double shift = shift_sum ? *shift_sum * inv_pow2(d.cells) : 0.0;
    const int lj = threadIdx.x / SK, lk = threadIdx.x % SK;
    const int tiles_k = d.n2 / SK;
    auto mix = [&](double m, double c, double p) {
        return QUARTER ? fma(2.0, c, m + p) : fma(ws, m + p, w1 * c);
    };
    // a warp's row, with the values before and after it
    struct Row {
        double v, e;
    };
    auto load = [&](int i, int j, int k0) {
        Row r;
        r.v = in[cell_index(d, i, j, k0 + lk)];
        if (lk == 0) r.e = in[cell_index(d, i, j, k0 - 1)];
        if (lk == SK - 1) r.e = in[cell_index(d, i, j, k0 + SK)];
        return r;
    };
    auto along_k = [&](const Row& r) {
        double m = __shfl_up_sync(0xffffffffu, r.v, 1), p = __shfl_down_sync(0xffffffffu, r.v, 1);
        if (lk == 0) m = r.e;
        if (lk == SK - 1) p = r.e;
        return mix(m, r.v, p);
    };
    const long long planes = (long long)tiles_k * (d.n1 / SJ) * d.n0;
    long long at = planes * blockIdx.x / gridDim.x;
    const long long end = planes * (blockIdx.x + 1) / gridDim.x;
    double acc = 0.0;
    while (at < end) {
        const int col = (int)(at / d.n0), i0 = (int)(at % d.n0);
        const int i1 = (int)min((long long)d.n0, i0 + (end - at));
        at += i1 - i0;
        const int k0 = (col % tiles_k) * SK, j0 = (col / tiles_k) * SJ;
        // warps 0 and 1 also smooth the rows before and after the tile
        const int je = lj == 0 ? j0 - 1 : j0 + SJ, re = lj == 0 ? 0 : SJ + 1;
        double a2 = 0.0, a1 = 0.0;  // (j, k)-smoothed values of planes p - 2, p - 1
        Row own = load(i0 - 1, j0 + lj, k0), edge{};
        if (lj < 2) edge = load(i0 - 1, je, k0);
        for (int p = i0 - 1; p <= i1; ++p) {
            double(*row)[SK] = sk[(p - i0 + 1) & 1];
            const double c = along_k(own);
            row[lj + 1][lk] = c;
            if (lj < 2) row[re][lk] = along_k(edge);
            if (p < i1) {
                own = load(p + 1, j0 + lj, k0);
                if (lj < 2) edge = load(p + 1, je, k0);
            }
            __syncthreads();  // (the other buffer is read until the next one)
            const double v = mix(row[lj][lk], c, row[lj + 2][lk]);
            if (p > i0) {  // plane p - 1 is complete
                const double x = mix(a2, a1, v);
                const double o = QUARTER ? fma(x, 1.0 / 64.0, -shift) : x - shift;
                const int e = cell_index(d, p - 1, j0 + lj, k0 + lk);
                out[e] = o;
                if (SUM) {
                    out32[e] = (float)o;
                    acc += o;
                }
                if (SQ) acc = fma(o, o, acc);
            }
            a2 = a1, a1 = v;
        }
        __syncthreads();
    }
    if (SUM || SQ) {
        acc = block_reduce<OpSum>(acc);
        if (threadIdx.x == 0) put_partial(part, acc, kRedBlocks);
    }
}

template <bool QUARTER>
void launch_smooth_stream(const Dims& d, double ws, const double* in, const double* shift_sum, double* out,
                          float* out32, double* part_sum, double* part_sq, cudaStream_t st) {
    if (part_sum)
        k_smooth_S_stream<QUARTER, true, false><<<kSBlocks, SJ * SK, 0, st>>>(d, ws, in, shift_sum, out, out32, part_sum);
    else if (part_sq)
        k_smooth_S_stream<QUARTER, false, true><<<kSBlocks, SJ * SK, 0, st>>>(d, ws, in, shift_sum, out, out32, part_sq);
    else
        k_smooth_S_stream<QUARTER, false, false><<<kSBlocks, SJ * SK, 0, st>>>(d, ws, in, shift_sum, out, out32, nullptr);
}

// V = e^-1 G at every node: e = I + Hess phi (before the step; stored by
// launch_triad), G the central-difference gradient of dphi; e^-1 from
// the adjugate of the symmetric e.
__global__ void k_node_velocity(Dims d, const double* __restrict__ e6,
                                const double* __restrict__ dphi, double* __restrict__ vx,
                                double* __restrict__ vy, double* __restrict__ vz) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const size_t n = (size_t)d.cells;
    Sym3 e;
    e.xx = e6[c], e.yy = e6[n + c], e.zz = e6[2 * n + c];
    e.xy = e6[3 * n + c], e.xz = e6[4 * n + c], e.yz = e6[5 * n + c];
    // twice the central-difference gradient of dphi (the 1/2 goes with 1/det)
    const double gx = dphi[cell_index(d, i + 1, j, k)] - dphi[cell_index(d, i - 1, j, k)];
    const double gy = dphi[cell_index(d, i, j + 1, k)] - dphi[cell_index(d, i, j - 1, k)];
    const double gz = dphi[cell_index(d, i, j, k + 1)] - dphi[cell_index(d, i, j, k - 1)];
    // e^-1 = adj(e) / det e with the six cofactors of the symmetric e
    const double Axx = e.yy * e.zz - e.yz * e.yz, Ayy = e.xx * e.zz - e.xz * e.xz;
    const double Azz = e.xx * e.yy - e.xy * e.xy, Axy = e.xz * e.yz - e.xy * e.zz;
    const double Axz = e.xy * e.yz - e.yy * e.xz, Ayz = e.xy * e.xz - e.xx * e.yz;
    const double hinv = 0.5 / (e.xx * Axx + e.xy * Axy + e.xz * Axz);
    vx[c] = (Axx * gx + Axy * gy + Axz * gz) * hinv;
    vy[c] = (Axy * gx + Ayy * gy + Ayz * gz) * hinv;
    vz[c] = (Axz * gx + Ayz * gy + Azz * gz) * hinv;
}

// App. A's linear density update (the variant that carries m instead of
// re-depositing tracers): K = m e^-1 at every node, e = I + Hess phi the
// stored triad (symmetric, so K is too: xx, yy, zz, xy, xz, yz).
__global__ void k_mass_tensor(Dims d, const double* __restrict__ e6, const double* __restrict__ m,
                              double* __restrict__ K6) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    const size_t n = (size_t)d.cells;
    Sym3 e;
    e.xx = e6[c], e.yy = e6[n + c], e.zz = e6[2 * n + c];
    e.xy = e6[3 * n + c], e.xz = e6[4 * n + c], e.yz = e6[5 * n + c];
    const double cxx = e.yy * e.zz - e.yz * e.yz, cyy = e.xx * e.zz - e.xz * e.xz;
    const double czz = e.xx * e.yy - e.xy * e.xy, cxy = e.xz * e.yz - e.xy * e.zz;
    const double cxz = e.xy * e.yz - e.xz * e.yy, cyz = e.xy * e.xz - e.xx * e.yz;
    const double s = m[c] / det3(e);
    K6[c] = cxx * s, K6[n + c] = cyy * s, K6[2 * n + c] = czz * s;
    K6[3 * n + c] = cxy * s, K6[4 * n + c] = cxz * s, K6[5 * n + c] = cyz * s;
}

// m += alpha d_mu(K^{mu nu} d_nu v) in flux form: per axis the second
// difference with face coefficients (K_c + K_n)/2, per axis pair the
// difference of centred differences taken at the two neighbours.
__global__ void k_mass_update(Dims d, const double* __restrict__ K6, const double* __restrict__ v,
                              const double* __restrict__ alpha_p, double* __restrict__ m) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    const double alpha = *alpha_p;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const size_t n = (size_t)d.cells;
    const int o[3][3] = {{1, 0, 0}, {0, 1, 0}, {0, 0, 1}};
    const int off[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};  // K6 slot of (a, b)
    const double vc = v[c];
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int pl = cell_index(d, i + o[a][0], j + o[a][1], k + o[a][2]);
        const int mi = cell_index(d, i - o[a][0], j - o[a][1], k - o[a][2]);
        const double* Ka = K6 + off[a][a] * n;
        acc += 0.5 * (Ka[c] + Ka[pl]) * (v[pl] - vc) - 0.5 * (Ka[c] + Ka[mi]) * (vc - v[mi]);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            if (b == a) continue;
            const double* Kab = K6 + off[a][b] * n;
            const int pi = i + o[a][0], pj = j + o[a][1], pk = k + o[a][2];
            const int qi = i - o[a][0], qj = j - o[a][1], qk = k - o[a][2];
            const double dp = v[cell_index(d, pi + o[b][0], pj + o[b][1], pk + o[b][2])] -
                              v[cell_index(d, pi - o[b][0], pj - o[b][1], pk - o[b][2])];
            const double dm = v[cell_index(d, qi + o[b][0], qj + o[b][1], qk + o[b][2])] -
                              v[cell_index(d, qi - o[b][0], qj - o[b][1], qk - o[b][2])];
            acc += 0.25 * (Kab[pl] * dp - Kab[mi] * dm);
        }
    }
    m[c] += alpha * acc;
}

// a = max(m, a_min) in FP64 (and FP32) with partial sums of m, for the
// variant whose m is carried rather than deposited.
__global__ void k_coef_from_m(int cells, const double* __restrict__ m, double a_min,
                              double* __restrict__ a64, float* __restrict__ a32,
                              double* __restrict__ part) {
    double s = 0.0;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < cells; c += gridDim.x * blockDim.x) {
        const double v = m[c];
        const double a = v > a_min ? v : a_min;
        a64[c] = a;
        if (a32) a32[c] = (float)a;
        s += v;
    }
    s = block_reduce<OpSum>(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// phi += alpha (dphi - mean) without moving tracers.
__global__ void k_phi_advance(int cells, const double* __restrict__ alpha_p,
                              const double* __restrict__ dphi, const double* __restrict__ sum_dphi,
                              double* __restrict__ phi, float* __restrict__ phi32) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= cells) return;
    const double alpha = *alpha_p;
    const double mean = *sum_dphi * inv_pow2(cells);
    const double pn = phi[c] + alpha * (dphi[c] - mean);
    phi[c] = pn;
    phi32[c] = (float)pn;
}

// (b - a) f / 2^52 rounded to nearest, added to a: one step of linear
// interpolation of fixed-point values with a fraction f of fixed_axis
// (|b - a| <= 2^61; the 128-bit product's upper half is the floor, its lower
// half's top bit the rounding).
__device__ inline long long lerp_fixed(long long a, long long b, unsigned long long f) {
    const long long x = (b - a) * 2, y = (long long)(f << (63 - kFracBits));
    const unsigned long long low = (unsigned long long)x * (unsigned long long)y;
    return a + __mul64hi(x, y) + (long long)(low >> 63);
}

// Tracers move by -alpha V(xi), V CIC-interpolated from the nodes, in fixed
// point: the offsets are rounded to 2^-52 cell as in cic_charges, and the
// node displacements alpha V (displacement.cu, 2^-53 cells) are
// interpolated by integer linear interpolation along k, then j, then i, each
// step rounded to nearest (rounding down instead biases every move by about a
// unit the same way, which the 40-step 32^3 trajectory amplified to 3e-6 in
// R_k); the result leaves as one FP64 subtraction per axis.
// phi += alpha (dphi - mean), mean = *sum_dphi / cells.
__global__ void k_advance(Dims d, const long long* __restrict__ dx, const long long* __restrict__ dy,
                          const long long* __restrict__ dz, const double* __restrict__ alpha_p,
                          const double* __restrict__ dphi, const double* __restrict__ sum_dphi,
                          double* __restrict__ ox, double* __restrict__ oy,
                          double* __restrict__ oz, double* __restrict__ phi,
                          float* __restrict__ phi32) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    const double alpha = *alpha_p;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const double px = ox[c], py = oy[c], pz = oz[c];
    int i0, j0, k0;
    unsigned long long fx, fy, fz;
    fixed_axis(i, px, i0, fx);
    fixed_axis(j, py, j0, fy);
    fixed_axis(k, pz, k0, fz);
    int nb[2][2][2];
#pragma unroll
    for (int di = 0; di < 2; ++di)
#pragma unroll
        for (int dj = 0; dj < 2; ++dj)
#pragma unroll
            for (int dk = 0; dk < 2; ++dk) nb[di][dj][dk] = cell_index(d, i0 + di, j0 + dj, k0 + dk);
    auto interp = [&](const long long* __restrict__ D) {
        long long cx[2];
#pragma unroll
        for (int di = 0; di < 2; ++di) {
            const long long c0 = lerp_fixed(D[nb[di][0][0]], D[nb[di][0][1]], fz);
            const long long c1 = lerp_fixed(D[nb[di][1][0]], D[nb[di][1][1]], fz);
            cx[di] = lerp_fixed(c0, c1, fy);
        }
        return lerp_fixed(cx[0], cx[1], fx);
    };
    constexpr double unit = 1.0 / 9007199254740992.0;  // 2^-53
    ox[c] = fma(-(double)interp(dx), unit, px);
    oy[c] = fma(-(double)interp(dy), unit, py);
    oz[c] = fma(-(double)interp(dz), unit, pz);
    const double mean = *sum_dphi * inv_pow2(d.cells);
    const double pn = phi[c] + alpha * (dphi[c] - mean);
    phi[c] = pn;
    phi32[c] = (float)pn;
}

__global__ void k_mesh_x(Dims d, const double* __restrict__ phi, double h, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    out[3 * c + 0] = ((double)i + 0.5 * (phi[cell_index(d, i + 1, j, k)] - phi[cell_index(d, i - 1, j, k)])) * h;
    out[3 * c + 1] = ((double)j + 0.5 * (phi[cell_index(d, i, j + 1, k)] - phi[cell_index(d, i, j - 1, k)])) * h;
    out[3 * c + 2] = ((double)k + 0.5 * (phi[cell_index(d, i, j, k + 1)] - phi[cell_index(d, i, j, k - 1)])) * h;
}

__global__ void k_scale(int cells, const double* __restrict__ in, double s, double* __restrict__ out) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < cells) out[c] = in[c] * s;
}

template <class Op>
__device__ void finish(const double* __restrict__ partials, double* __restrict__ scalars, int slot) {
    double v = Op::id();
    for (int b = threadIdx.x; b < kRedBlocks; b += blockDim.x) v = Op::op(v, partials[b]);
    v = block_reduce<Op>(v);
    if (threadIdx.x == 0) scalars[slot] = v;
}

// Finishes several reductions, a block each.
__global__ void k_finish(FinishList l, double* __restrict__ scalars) {
    const Finish f = l.f[blockIdx.x];
    if (f.op == 0) finish<OpSum>(f.partials, scalars, f.slot);
    else if (f.op == 1) finish<OpMin>(f.partials, scalars, f.slot);
    else finish<OpMax>(f.partials, scalars, f.slot);
}

}  // namespace

void finish_reduces(const FinishList& l, double* scalars, cudaStream_t st) {
    launch_counter()++;
    k_finish<<<l.n, 256, 0, st>>>(l, scalars);
}

void finish_reduce(const double* partials, int op, double* scalars, int slot, cudaStream_t st) {
    finish_reduces(FinishList{1, {{partials, op, slot}}}, scalars, st);
}

void launch_validate_grid(int cells, const double* rho, double* ps, double* pb, cudaStream_t st) {
    launch_counter()++;
    k_validate_grid<<<kRedBlocks, kRedThreads, 0, st>>>(cells, rho, ps, pb);
}

void launch_validate_particles(int64_t np, const double* pos, const double* mass, double* ps,
                               double* pb, cudaStream_t st) {
    launch_counter()++;
    k_validate_particles<<<kRedBlocks, kRedThreads, 0, st>>>(np, pos, mass, ps, pb);
}

void launch_deposit_particles(const Dims& d, int64_t np, const double* pos, const double* mass,
                              double inv_h, double scale, const double* total, double* bad,
                              unsigned long long* mfix, cudaStream_t st) {
    if (np <= 0) return;
    launch_counter()++;
    k_deposit_particles<<<(unsigned)((np + kThreads - 1) / kThreads), kThreads, 0, st>>>(
        d, np, pos, mass, inv_h, scale, total, bad, mfix);
}

void launch_fix_validate(int cells, unsigned long long* mfix, double scale, const double* total, double* out,
                         double* ps, double* pb, cudaStream_t st) {
    if (cells > 1 << 20) {
        launch_fix_to_double(cells, mfix, scale, total, out, st);
        launch_validate_grid(cells, out, ps, pb, st);
        return;
    }
    launch_counter()++;
    k_fix_validate<<<kRedBlocks, kRedThreads, 0, st>>>(cells, mfix, scale, total, out, ps, pb);
}

void launch_fix_to_double(int cells, unsigned long long* mfix, double scale, const double* total, double* out,
                          cudaStream_t st) {
    launch_counter()++;
    k_fix_to_double<<<nblocks(cells), kThreads, 0, st>>>(cells, mfix, scale, total, out);
}

void launch_init_tracers(int cells, const double* rho, const double* sum_rho, double* w,
                         double* ox, double* oy, double* oz, double* phi, float* phi32,
                         cudaStream_t st) {
    launch_counter()++;
    k_init_tracers<<<nblocks(cells), kThreads, 0, st>>>(cells, rho, sum_rho, w, ox, oy, oz, phi,
                                                        phi32);
}

void launch_deposit_tracers(const Dims& d, const double* ox, const double* oy, const double* oz,
                            const double* w, double scale, unsigned long long* mfix,
                            cudaStream_t st) {
    launch_counter()++;
    k_deposit_tracers<<<nblocks(d.cells), kThreads, 0, st>>>(d, ox, oy, oz, w, scale, mfix);
}

void launch_mass_coef(int cells, unsigned long long* mfix, double inv_scale, double a_min,
                      double* m, double* a64, float* a32, double* partials, cudaStream_t st) {
    launch_counter()++;
    k_mass_coef<<<kRedBlocks, kRedThreads, 0, st>>>(cells, mfix, inv_scale, a_min, m, a64, a32,
                                                    partials);
}

void launch_smooth_S(const Dims& d, double s_side, const double* in, const double* shift_sum,
                     double* out, float* out32, double* tmp2, double* part_sum, double* part_sq,
                     cudaStream_t st) {
    if (d.n2 % SK == 0 && d.n1 % SJ == 0 && !(part_sum && part_sq)) {
        launch_counter()++;
        auto launch = s_side == 0.25 ? launch_smooth_stream<true> : launch_smooth_stream<false>;
        launch(d, s_side, in, shift_sum, out, out32, part_sum, part_sq, st);
        return;
    }
    launch_counter() += 3;
    k_smooth_axis<<<kRedBlocks, kRedThreads, 0, st>>>(d, 2, s_side, in, nullptr, tmp2, nullptr,
                                                      nullptr, nullptr);
    k_smooth_axis<<<kRedBlocks, kRedThreads, 0, st>>>(d, 1, s_side, tmp2, nullptr,
                                                      tmp2 + d.cells, nullptr, nullptr, nullptr);
    k_smooth_axis<<<kRedBlocks, kRedThreads, 0, st>>>(d, 0, s_side, tmp2 + d.cells, shift_sum,
                                                      out, out32, part_sum, part_sq);
}

void launch_node_velocity(const Dims& d, const double* e6, const double* dphi, double* vx,
                          double* vy, double* vz, cudaStream_t st) {
    launch_counter()++;
    k_node_velocity<<<nblocks(d.cells), kThreads, 0, st>>>(d, e6, dphi, vx, vy, vz);
}

void launch_advance(const Dims& d, const long long* dx, const long long* dy, const long long* dz,
                    const double* alpha, const double* dphi, const double* sum_dphi, double* ox,
                    double* oy, double* oz, double* phi, float* phi32, cudaStream_t st) {
    launch_counter()++;
    k_advance<<<nblocks(d.cells), kThreads, 0, st>>>(d, dx, dy, dz, alpha, dphi, sum_dphi, ox, oy,
                                                     oz, phi, phi32);
}

void launch_mass_literal(const Dims& d, const double* e6, const double* dphi,
                         const double* alpha, double* m, double* K6, cudaStream_t st) {
    launch_counter() += 2;
    k_mass_tensor<<<nblocks(d.cells), kThreads, 0, st>>>(d, e6, m, K6);
    k_mass_update<<<nblocks(d.cells), kThreads, 0, st>>>(d, K6, dphi, alpha, m);
}

void launch_coef_from_m(int cells, const double* m, double a_min, double* a64, float* a32,
                        double* partials, cudaStream_t st) {
    launch_counter()++;
    k_coef_from_m<<<kRedBlocks, kRedThreads, 0, st>>>(cells, m, a_min, a64, a32, partials);
}

void launch_phi_advance(int cells, const double* alpha, const double* dphi,
                        const double* sum_dphi, double* phi, float* phi32, cudaStream_t st) {
    launch_counter()++;
    k_phi_advance<<<nblocks(cells), kThreads, 0, st>>>(cells, alpha, dphi, sum_dphi, phi, phi32);
}

void launch_mesh_x(const Dims& d, const double* phi, double h, double* out, cudaStream_t st) {
    launch_counter()++;
    k_mesh_x<<<nblocks(d.cells), kThreads, 0, st>>>(d, phi, h, out);
}

void launch_scale(int cells, const double* in, double s, double* out, cudaStream_t st) {
    launch_counter()++;
    k_scale<<<nblocks(cells), kThreads, 0, st>>>(cells, in, s, out);
}


}  // namespace recon
