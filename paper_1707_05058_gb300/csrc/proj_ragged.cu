// Instantiations and launchers of the standalone projection of ragged batches.
#include <algorithm>

#include "proj_ragged.cuh"

namespace cdsdp_dev {

cudaError_t launch_project_ragged(bool fp32, int p, int limit, const int* off, const int* size, const void* W, void* X,
                                  int max_sweeps, bool overlap, cudaStream_t st) {
    const double tolrel = jacobi_tolrel(32, fp32);
    if (fp32)
        return limit <= 16 ? launch_ragged<float, 16>(p, limit, off, size, W, X, tolrel, max_sweeps, overlap, st)
                           : launch_ragged<float, 32>(p, std::min(limit, 32), off, size, W, X, tolrel, max_sweeps, overlap, st);
    return limit <= 16 ? launch_ragged<double, 16>(p, limit, off, size, W, X, tolrel, max_sweeps, overlap, st)
                       : launch_ragged<double, 32>(p, std::min(limit, 32), off, size, W, X, tolrel, max_sweeps, overlap, st);
}

cudaError_t launch_project_cta_ragged(int p, int limit, const int* off, const int* size, const void* W, void* X,
                                      int max_sweeps, bool overlap, cudaStream_t st) {
    const size_t smem = CTAJacobiReg<64>::bytes;
    cudaError_t e = cudaFuncSetAttribute(k_project_cta_ragged, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_beside(overlap, k_project_cta_ragged, proj_cta_grid(p), kRaggedCtaThreads, smem, st, p,
                         std::min(limit, 64), off, size, (const float*)W, (float*)X, jacobi_tolrel(64, true), max_sweeps);
}

}  // namespace cdsdp_dev
