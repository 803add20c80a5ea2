// The FP64 residual pass with its FP32 copy, called alone: sum of r^2.
#include "../../paper_1611_09638_gb300/csrc/mg_kernels.cu"

extern "C" int residual_partials(int n0, int n1, int n2, const double* u, const double* f, const double* F,
                                 const double* D, float* r32, double* partials) {
    recon::Level L{};
    L.d = recon::make_dims(n0, n1, n2);
    recon::launch_residual64_to32(L, u, f, F, D, r32, partials, nullptr);
    return (int)cudaDeviceSynchronize();
}

extern "C" int partials() { return recon::kRedBlocks; }
