// The node displacements' fixed-point arithmetic (displacement_solve.cuh), on
// the host.
#include "cuda_runtime.h"

#include "../../paper_1611_09638_gb300/csrc/displacement_solve.cuh"

// solve_fixed over a list of nodes; scales: Qd, kexp of each.
extern "C" void solve_nodes(int count, const int* scales, const long long* h, const long long* g, long long* out,
                            int* accepted) {
    for (int n = 0; n < count; ++n) {
        const recon::DispScales sc{scales[2 * n], scales[2 * n + 1], true};
        long long hn[6], gn[3], u[3] = {0, 0, 0};
        for (int q = 0; q < 6; ++q) hn[q] = h[6 * n + q];
        for (int q = 0; q < 3; ++q) gn[q] = g[3 * n + q];
        accepted[n] = recon::solve_fixed(sc, hn, gn, u);
        for (int q = 0; q < 3; ++q) out[3 * n + q] = u[q];
    }
}

// The whole of a node from the 3 x 3 x 3 values around it; the scales of a step
// with step length alpha and largest gradient max_g.
extern "C" void displace_nodes(int count, double alpha, double max_g, double sum_dphi, int wide, const double* phi,
                               const double* dphi, long long* out, int* accepted) {
    const recon::DispScales sc = recon::disp_scales(alpha, max_g, sum_dphi, wide != 0);
    for (int n = 0; n < count; ++n) {
        recon::DispColumn sums{};
        long long h[6], g[3], u[3] = {0, 0, 0};
        for (int p = 0; p < 3; ++p) {
            unsigned long long f[9], w[9];
            for (int q = 0; q < 9; ++q) {
                f[q] = recon::to_fixed_mod(phi[27 * n + 9 * p + q], recon::kPhiBits);
                w[q] = recon::to_fixed_mod(dphi[27 * n + 9 * p + q], sc.Qd);
            }
            sums.feed(f + 4, w + 4, 3, h, g);
        }
        accepted[n] = sc.ok && recon::solve_fixed(sc, h, g, u);
        for (int q = 0; q < 3; ++q) out[3 * n + q] = u[q];
    }
}

extern "C" void fixed_mod(int count, const double* x, int Q, unsigned long long* out) {
    for (int n = 0; n < count; ++n) out[n] = recon::to_fixed_mod(x[n], Q);
}
