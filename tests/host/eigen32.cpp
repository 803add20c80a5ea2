// lambda32 (eigen32.cuh) over a list of Hessians, on the host.
#include "cuda_runtime.h"

#include "../../paper_1611_09638_gb300/csrc/eigen32.cuh"

extern "C" void lambdas(int count, const float* h, float* lam, float* el) {
    for (int n = 0; n < count; ++n, h += 6) {
        float big = 0.f;
        for (int q = 0; q < 6; ++q) big = std::max(big, fabsf(q < 3 ? 1.f + h[q] : h[q]));
        // entries that are exact but for forming 1 + h
        lam[n] = recon::lambda32(h[0], h[1], h[2], h[3], h[4], h[5], big, 4.f * recon::kU * (big + 1.f), el[n]);
    }
}
