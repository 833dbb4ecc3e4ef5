// Instantiations of the gradient kernels for padded dimension 16.
#include "pm_fx_grad.cuh"

namespace pm {

template <typename Real, int INTEG>
static cudaError_t adjoint_launch(const GradParams &gp, int grid, int warps, size_t smem, cudaStream_t st) {
    auto k = adjoint_kernel<Real, 16, INTEG>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k<<<grid, warps * 32, smem, st>>>(gp);
    return cudaGetLastError();
}

template <typename Real, int INTEG>
static int adjoint_occupancy(int warps, size_t smem) {
    int nb = 0;
    auto k = adjoint_kernel<Real, 16, INTEG>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, warps * 32, smem);
    return e == cudaSuccess ? nb : 0;
}

// scans, then the adjoint: FP32 by groups of lanes on the CUDA cores, FP64 by the digit products (grid: the
// number of SMs, smem: the shared memory limit of a block there)
cudaError_t grad_run_d16(int fp64, int integ, const ScanParams &sp, const GradParams &gp, int grid, int warps,
                         size_t smem, cudaStream_t st) {
    cudaError_t e = fx::scan_run<16>(sp, sp.bpin, true, st);
    if (e != cudaSuccess) return e;
    switch (integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return adjoint_launch<float, kMidpoint>(gp, grid, warps, smem, st);
        case 1: return fx::adjoint_launch<16, kMidpoint>(gp, grid, smem, st);
        case 2: return adjoint_launch<float, kGL2>(gp, grid, warps, smem, st);
        case 3: return fx::adjoint_launch<16, kGL2>(gp, grid, smem, st);
        case 4: return adjoint_launch<float, kSimpson>(gp, grid, warps, smem, st);
        case 5: return fx::adjoint_launch<16, kSimpson>(gp, grid, smem, st);
    }
    return cudaErrorInvalidValue;
}

// exclusive prefixes of every leaf from the forward pass's leaf and block products
cudaError_t scan_run_d16(const ScanParams &sp, cudaStream_t st) { return fx::scan_run<16>(sp, sp.bpin, false, st); }

cudaError_t fx_trace_d16(const double *packed, const double *bnorm, int nb, void *out, cudaStream_t st) {
    return fx::trace_digits<16>(packed, bnorm, nb, out, st);
}
size_t fx_trace_bytes_d16(int nb) { return fx::trace_digit_bytes<16>(nb); }
size_t fx_adjoint_leaf_bytes_d16() { return fx::AdjCfg<16>::LEAF_BYTES; }

int adjoint_blocks_per_sm_d16(int fp64, int integ, int warps, size_t smem) {
    switch (integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return adjoint_occupancy<float, kMidpoint>(warps, smem);
        case 2: return adjoint_occupancy<float, kGL2>(warps, smem);
        case 4: return adjoint_occupancy<float, kSimpson>(warps, smem);
    }
    return 0;
}

size_t adjoint_smem_d16(int fp64, int K, int warps) {
    (void)fp64;  // FP64: sized by its own launch (pm_fx_grad.cuh)
    return adjoint_smem_bytes<float, 16>(K, warps);
}

}  // namespace pm
