// Instantiations of the fused propagation kernel for padded dimension 8
// (mode cheb: 0 = Taylor exponential, 1 = Chebyshev exponential, 2 = Taylor trajectory,
// 3 = FP64 Taylor on the FP64 pipe for callers without workspace).  FP64 Taylor (0, 2) runs on the
// exact digit products of pm_fx.cuh; legacy asks for the geometry of the FP64 fused kernel (1, 3, batched items).
#include "pm_fx.cuh"

namespace pm {

cudaError_t fused_dispatch_d8(int fp64, int integ, const FusedParams &p, int grid, int warps, size_t smem,
                               cudaStream_t st, int cheb) {
    switch (cheb * 6 + integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return launch_fused<float, 8, kMidpoint>(p, grid, warps, smem, st);
        case 1: return fx::launch<8, kMidpoint, false>(p, grid, warps, smem, st);
        case 2: return launch_fused<float, 8, kGL2>(p, grid, warps, smem, st);
        case 3: return fx::launch<8, kGL2, false>(p, grid, warps, smem, st);
        case 4: return launch_fused<float, 8, kSimpson>(p, grid, warps, smem, st);
        case 5: return fx::launch<8, kSimpson, false>(p, grid, warps, smem, st);
        case 6: return launch_fused<float, 8, kMidpoint, 1>(p, grid, warps, smem, st);
        case 7: return launch_fused<double, 8, kMidpoint, 1>(p, grid, warps, smem, st);
        case 8: return launch_fused<float, 8, kGL2, 1>(p, grid, warps, smem, st);
        case 9: return launch_fused<double, 8, kGL2, 1>(p, grid, warps, smem, st);
        case 10: return launch_fused<float, 8, kSimpson, 1>(p, grid, warps, smem, st);
        case 11: return launch_fused<double, 8, kSimpson, 1>(p, grid, warps, smem, st);
        case 12: return launch_fused<float, 8, kMidpoint, 2>(p, grid, warps, smem, st);
        case 13: return fx::launch<8, kMidpoint, true>(p, grid, warps, smem, st);
        case 14: return launch_fused<float, 8, kGL2, 2>(p, grid, warps, smem, st);
        case 15: return fx::launch<8, kGL2, true>(p, grid, warps, smem, st);
        case 16: return launch_fused<float, 8, kSimpson, 2>(p, grid, warps, smem, st);
        case 17: return fx::launch<8, kSimpson, true>(p, grid, warps, smem, st);
        case 19: return launch_fused<double, 8, kMidpoint>(p, grid, warps, smem, st);
        case 21: return launch_fused<double, 8, kGL2>(p, grid, warps, smem, st);
        case 23: return launch_fused<double, 8, kSimpson>(p, grid, warps, smem, st);
    }
    return cudaErrorInvalidValue;
}

int fused_blocks_per_sm_d8(int fp64, int integ, int warps, size_t smem, int cheb) {
    switch (cheb * 6 + integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return fused_max_blocks_per_sm<float, 8, kMidpoint>(warps, smem);
        case 1: return fx::max_blocks_per_sm<8, kMidpoint, false>(warps, smem);
        case 2: return fused_max_blocks_per_sm<float, 8, kGL2>(warps, smem);
        case 3: return fx::max_blocks_per_sm<8, kGL2, false>(warps, smem);
        case 4: return fused_max_blocks_per_sm<float, 8, kSimpson>(warps, smem);
        case 5: return fx::max_blocks_per_sm<8, kSimpson, false>(warps, smem);
        case 6: return fused_max_blocks_per_sm<float, 8, kMidpoint, 1>(warps, smem);
        case 7: return fused_max_blocks_per_sm<double, 8, kMidpoint, 1>(warps, smem);
        case 8: return fused_max_blocks_per_sm<float, 8, kGL2, 1>(warps, smem);
        case 9: return fused_max_blocks_per_sm<double, 8, kGL2, 1>(warps, smem);
        case 10: return fused_max_blocks_per_sm<float, 8, kSimpson, 1>(warps, smem);
        case 11: return fused_max_blocks_per_sm<double, 8, kSimpson, 1>(warps, smem);
        case 12: return fused_max_blocks_per_sm<float, 8, kMidpoint, 2>(warps, smem);
        case 13: return fx::max_blocks_per_sm<8, kMidpoint, true>(warps, smem);
        case 14: return fused_max_blocks_per_sm<float, 8, kGL2, 2>(warps, smem);
        case 15: return fx::max_blocks_per_sm<8, kGL2, true>(warps, smem);
        case 16: return fused_max_blocks_per_sm<float, 8, kSimpson, 2>(warps, smem);
        case 17: return fx::max_blocks_per_sm<8, kSimpson, true>(warps, smem);
        case 19: return fused_max_blocks_per_sm<double, 8, kMidpoint>(warps, smem);
        case 21: return fused_max_blocks_per_sm<double, 8, kGL2>(warps, smem);
        case 23: return fused_max_blocks_per_sm<double, 8, kSimpson>(warps, smem);
    }
    return 0;
}

size_t fused_smem_d8(int fp64, int n_basis, int warps, int legacy) {
    if (fp64 && !legacy) return fx::smem_bytes<8>(n_basis, warps);
    return fp64 ? fused_smem_bytes<double, 8>(n_basis, warps) : fused_smem_bytes<float, 8>(n_basis, warps);
}

int fused_groups_per_warp_d8(int fp64, int legacy) {
    return fp64 ? (legacy ? Geo<double, 8>::GPW : 1) : Geo<float, 8>::GPW;
}

int fused_max_warps_d8(int fp64, int legacy) {
    return fp64 ? (legacy ? Geo<double, 8>::MAXW : fx::Cfg<8>::MAXW) : Geo<float, 8>::MAXW;
}

cudaError_t fx_basis_d8(const double *packed, const double *bnorm, int nb, void *out, cudaStream_t st) {
    return fx::basis_digits<8>(packed, bnorm, nb, out, st);
}
size_t fx_basis_bytes_d8(int nb) { return fx::basis_digit_bytes<8>(nb); }
size_t fx_leaf_bytes_d8() { return fx::Cfg<8>::LEAF_BYTES; }

}  // namespace pm
