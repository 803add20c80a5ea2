// displacement.cu -- the node displacements of a step, alpha V = alpha e^-1 G
// with e = I + Hess phi and G the central-difference gradient of dphi (the
// mesh points' motion seen by the tracers, Sec. II of Zhu et al. 2016), in
// fixed point with kDispBits fractional bits for the tracer advance.
//
// In FP64 a node takes some 70 instructions (the Hessian, six cofactors, a
// division, three products), 10 ms at 512^3 with the Hessian read back from
// memory.  Here only FP32 and integer instructions run: phi and dphi are
// brought to 64-bit fixed point as a plane is loaded (phi to 2^-54 whatever its
// size, modulo 2^64: the source's pass over the same phi shows that every
// second difference fits; dphi to 2^-Qd from the limiter's largest gradient), Hessian and gradient are
// exact integer sums, and e U = alpha G is solved by iterative refinement: X ~
// e^-1 in FP32 gives a first U, and each further piece comes from the exact
// residual alpha G - e U, formed modulo 2^64 (its leading bits cancel, so the
// low 64 bits of the products suffice).  A piece carries 18 bits, so two or
// three residuals leave an error below the 2^-53 cells of the result; badly
// conditioned nodes take smaller pieces and more of them.  Nodes that do not
// converge, and steps whose numbers do not fit (disp_scales), are computed in
// FP64.  Against exact rational arithmetic (smooth fields with |phi| up to 4, 60
// and 166 cells^2, alpha V up to half a cell) the error is 0.29 units of 2^-53 cells rms and
// 0.57 at most, also at the nodes of the large fields where phi is small; that
// of the FP64 form 0.29, 0.61 and 4.9 rms (0.29, 0.44 and 0.33 where |phi| < 6),
// 148 at most (rounding to the unit alone: 0.289).
//
// A block streams planes along i over an 8 x 32 (or 16 x 16) tile; a thread keeps its
// column's sums of the last planes in registers, so that a plane's 340 nodes
// are converted once and read back from shared memory 14 times a thread.
// Bound by instruction issue (70% of the slots, 54% of the integer pipe):
// 512^3 10.06 -> 3.49 ms; it reads 16 and writes 24 bytes a node (0.8 ms at the
// copy rate).
#include "checked.cuh"
#include "displacement_solve.cuh"
#include "geometry.cuh"
#include "recon_internal.cuh"

namespace recon {

namespace {

constexpr long long kDispMax = 1ll << (kDispBits + 7);  // 128 cells

constexpr int DT = 256;  // nodes of a tile, DK of them along k
constexpr int DPERSM = 3, DBLOCKS = DPERSM * (kRedBlocks / 8);

// alpha V at one node in FP64, rounded to fixed point; values beyond kDispMax
// cells, which no valid step produces, are held at that bound.
__device__ __noinline__ void displacement64(const Dims& d, const double* __restrict__ phi,
                                            const double* __restrict__ dphi, double alpha, int i, int j, int k,
                                            long long (&out)[3]) {
    Sym3 e = hessian(d, phi, i, j, k);
    e.xx += 1.0, e.yy += 1.0, e.zz += 1.0;
    const double gx = dphi[cell_index(d, i + 1, j, k)] - dphi[cell_index(d, i - 1, j, k)];
    const double gy = dphi[cell_index(d, i, j + 1, k)] - dphi[cell_index(d, i, j - 1, k)];
    const double gz = dphi[cell_index(d, i, j, k + 1)] - dphi[cell_index(d, i, j, k - 1)];
    const double Axx = e.yy * e.zz - e.yz * e.yz, Ayy = e.xx * e.zz - e.xz * e.xz;
    const double Azz = e.xx * e.yy - e.xy * e.xy, Axy = e.xz * e.yz - e.xy * e.zz;
    const double Axz = e.xy * e.yz - e.yy * e.xz, Ayz = e.xy * e.xz - e.xx * e.yz;
    // 1/2 of the central differences, alpha and 2^kDispBits in one factor
    const double hinv = (0.5 * 9007199254740992.0) * alpha / (e.xx * Axx + e.xy * Axy + e.xz * Axz);
    auto fix = [](double v) {
        const long long q = __double2ll_rn(v);  // saturates beyond the int64 range
        return q > kDispMax ? kDispMax : (q < -kDispMax ? -kDispMax : q);
    };
    out[0] = fix((Axx * gx + Axy * gy + Axz * gz) * hinv);
    out[1] = fix((Axy * gx + Ayy * gy + Ayz * gz) * hinv);
    out[2] = fix((Axz * gx + Ayz * gy + Azz * gz) * hinv);
}

template <int DK>
__global__ void __launch_bounds__(DT, DPERSM) k_displacement_stream(
    Dims d, const double* __restrict__ scal, const double* __restrict__ phi, const double* __restrict__ dphi,
    long long* __restrict__ dx, long long* __restrict__ dy, long long* __restrict__ dz) {
    constexpr int DJ = DT / DK, DPK = DK + 2, DN = (DJ + 2) * DPK;  // rows, and with the ring
    static_assert(DN <= 2 * DT, "two values a thread and field");
    __shared__ U64 sp[2][DN], sd[2][DN];
    const DispScales sc = disp_scales(scal[SC_ALPHA], scal[SC_MAX_G], scal[SC_SUM_DPHI], scal[SC_WIDE] != 0.0);
    const int t = threadIdx.x, lj = t / DK, lk = t % DK;
    // (with the ring around it; RC_OFF: checked against the extent in the
    // RECON_CHECKED build)
    const int own = DPK + 1 + RC_OFF(lj * DPK + lk, DN - 2 * DPK - 2, 501);
    const int tiles_k = d.n2 / DK;
    const long long planes = (long long)tiles_k * (d.n1 / DJ) * d.n0;
    long long at = planes * blockIdx.x / gridDim.x;
    const long long end = planes * (blockIdx.x + 1) / gridDim.x;
    if (!sc.ok) {  // every node in FP64
        for (; at < end; ++at) {
            const int col = (int)(at / d.n0), i = (int)(at % d.n0);
            const int j = (col / tiles_k) * DJ + lj, k = (col % tiles_k) * DK + lk;
            long long o[3];
            displacement64(d, phi, dphi, scal[SC_ALPHA], i, j, k, o);
            const int c = cell_index(d, i, j, k);
            dx[c] = o[0], dy[c] = o[1], dz[c] = o[2];
        }
        return;
    }
    // this thread's nodes of a plane with its ring
    const int e1 = t + DT;
    const bool two = e1 < DN;
    while (at < end) {
        const int col = (int)(at / d.n0), i0 = (int)(at % d.n0);
        const int i1 = (int)min((long long)d.n0, i0 + (end - at));
        at += i1 - i0;
        const int k0 = (col % tiles_k) * DK, j0 = (col / tiles_k) * DJ;
        const int c0 = cell_index(d, 0, j0 - 1 + t / DPK, k0 - 1 + t % DPK);
        const int c1 = two ? cell_index(d, 0, j0 - 1 + e1 / DPK, k0 - 1 + e1 % DPK) : 0;
        const int plane = d.n1 * d.n2;
        double p0, p1 = 0.0, q0, q1 = 0.0;
        auto load = [&](int i) {
            const int b = (i & (d.n0 - 1)) * plane;
            const int g0 = RC_OFF(b + c0, d.cells, 502), g1 = RC_OFF(b + c1, d.cells, 503);
            p0 = phi[g0], q0 = dphi[g0];
            if (two) p1 = phi[g1], q1 = dphi[g1];
        };
        DispColumn sums{};
        load(i0 - 1);
        for (int p = i0 - 1; p <= i1; ++p) {
            const int buf = (p - i0 + 1) & 1;
            sp[buf][t] = to_fixed_mod(p0, kPhiBits), sd[buf][t] = to_fixed_mod(q0, sc.Qd);
            if (two) sp[buf][e1] = to_fixed_mod(p1, kPhiBits), sd[buf][e1] = to_fixed_mod(q1, sc.Qd);
            if (p < i1) load(p + 1);
            __syncthreads();  // (the other buffer is read until the next one)
            long long h[6], g[3];
            sums.feed(sp[buf] + own, sd[buf] + own, DPK, h, g);
            if (p > i0) {  // node (p - 1)
                long long o[3];
                if (!solve_fixed(sc, h, g, o)) displacement64(d, phi, dphi, scal[SC_ALPHA], p - 1, j0 + lj, k0 + lk, o);
                const int cell = cell_index(d, p - 1, j0 + lj, k0 + lk);
                dx[cell] = o[0], dy[cell] = o[1], dz[cell] = o[2];
            }
        }
        __syncthreads();
    }
}

// Any grid, a thread a node from memory, with the same sums (so the same bits).
// 1024 x 512 x 8: 497 us in FP64 throughout, 221 in this form.
__global__ void k_displacement_node(Dims d, const double* __restrict__ scal, const double* __restrict__ phi,
                                    const double* __restrict__ dphi, long long* __restrict__ dx,
                                    long long* __restrict__ dy, long long* __restrict__ dz) {
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= d.cells) return;
    int i, j, k;
    cell_coords(d, c, i, j, k);
    const double alpha = scal[SC_ALPHA];
    const DispScales sc = disp_scales(alpha, scal[SC_MAX_G], scal[SC_SUM_DPHI], scal[SC_WIDE] != 0.0);
    long long o[3];
    bool settled = false;
    if (sc.ok) {
        auto p = [&](int a, int b, int e) { return to_fixed_mod(phi[cell_index(d, i + a, j + b, k + e)], kPhiBits); };
        auto q = [&](int a, int b, int e) { return to_fixed_mod(dphi[cell_index(d, i + a, j + b, k + e)], sc.Qd); };
        const U64 two = 2 * p(0, 0, 0);
        const long long h[6] = {(long long)(p(1, 0, 0) + p(-1, 0, 0) - two), (long long)(p(0, 1, 0) + p(0, -1, 0) - two),
                                (long long)(p(0, 0, 1) + p(0, 0, -1) - two),
                                (long long)((p(1, 1, 0) - p(1, -1, 0)) - (p(-1, 1, 0) - p(-1, -1, 0))),
                                (long long)((p(1, 0, 1) - p(1, 0, -1)) - (p(-1, 0, 1) - p(-1, 0, -1))),
                                (long long)((p(0, 1, 1) - p(0, 1, -1)) - (p(0, -1, 1) - p(0, -1, -1)))};
        const long long g[3] = {(long long)(q(1, 0, 0) - q(-1, 0, 0)), (long long)(q(0, 1, 0) - q(0, -1, 0)),
                                (long long)(q(0, 0, 1) - q(0, 0, -1))};
        settled = solve_fixed(sc, h, g, o);
    }
    if (!settled) displacement64(d, phi, dphi, alpha, i, j, k, o);
    dx[c] = o[0], dy[c] = o[1], dz[c] = o[2];
}

}  // namespace

int bounds_fail_displacement() { return bounds_fail_take(); }

void launch_node_displacement(const Dims& d, const double* scal, const double* phi, const double* dphi,
                              long long* dx, long long* dy, long long* dz, cudaStream_t st) {
    launch_counter()++;
    if (d.n2 % 32 == 0 && d.n1 % 8 == 0) {
        k_displacement_stream<32><<<DBLOCKS, DT, 0, st>>>(d, scal, phi, dphi, dx, dy, dz);
        return;
    }
    if (d.n2 % 16 == 0 && d.n1 % 16 == 0) {
        k_displacement_stream<16><<<DBLOCKS, DT, 0, st>>>(d, scal, phi, dphi, dx, dy, dz);
        return;
    }
    k_displacement_node<<<(d.cells + 255) / 256, 256, 0, st>>>(d, scal, phi, dphi, dx, dy, dz);
}

}  // namespace recon
