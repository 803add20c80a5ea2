// solve_fixed (displacement_solve.cuh) over a list of nodes, on the host.
#include "cuda_runtime.h"

#include "../../paper_1611_09638_gb300/csrc/displacement_solve.cuh"

extern "C" void solve_nodes(int count, const int* scales, const long long* h, const long long* g, long long* out,
                            int* accepted) {
    for (int n = 0; n < count; ++n) {
        recon::DispScales sc{scales[3 * n], scales[3 * n + 1], scales[3 * n + 2], true};
        long long hn[6], gn[3], u[3] = {0, 0, 0};
        for (int q = 0; q < 6; ++q) hn[q] = h[6 * n + q];
        for (int q = 0; q < 3; ++q) gn[q] = g[3 * n + q];
        accepted[n] = recon::solve_fixed(sc, hn, gn, u);
        for (int q = 0; q < 3; ++q) out[3 * n + q] = u[q];
    }
}
