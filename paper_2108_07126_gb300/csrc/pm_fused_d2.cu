// Instantiations of the fused propagation kernel for padded dimension 2
// (mode cheb: 0 = U(T) by unit quaternions, 1 = Chebyshev exponential, 2 = Taylor trajectory, 3 = Taylor exponential
// with its degree and squarings).
#include "pm_fused.cuh"
#include "pm_su2.cuh"

namespace pm {

cudaError_t fused_dispatch_d2(int fp64, int integ, const FusedParams &p, int grid, int warps, size_t smem,
                               cudaStream_t st, int cheb) {
    // U(T) alone: unit quaternions, one thread per leaf (a leaf per lane in the fused kernel too, so that the caller's
    // geometry holds for both); the fused kernel where leaf or block products are kept or the degree is forced
    if (cheb == 3) {
        cheb = 0;
    } else if (cheb == 0 && !p.leaf_out && !p.block_out) {
        switch (integ * 2 + (fp64 ? 1 : 0)) {
            case 0: return su2::launch<float, kMidpoint>(p, grid, warps, st);
            case 1: return su2::launch<double, kMidpoint>(p, grid, warps, st);
            case 2: return su2::launch<float, kGL2>(p, grid, warps, st);
            case 3: return su2::launch<double, kGL2>(p, grid, warps, st);
            case 4: return su2::launch<float, kSimpson>(p, grid, warps, st);
            case 5: return su2::launch<double, kSimpson>(p, grid, warps, st);
        }
    }
    switch (cheb * 6 + integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return launch_fused<float, 2, kMidpoint>(p, grid, warps, smem, st);
        case 1: return launch_fused<double, 2, kMidpoint>(p, grid, warps, smem, st);
        case 2: return launch_fused<float, 2, kGL2>(p, grid, warps, smem, st);
        case 3: return launch_fused<double, 2, kGL2>(p, grid, warps, smem, st);
        case 4: return launch_fused<float, 2, kSimpson>(p, grid, warps, smem, st);
        case 5: return launch_fused<double, 2, kSimpson>(p, grid, warps, smem, st);
        case 6: return launch_fused<float, 2, kMidpoint, 1>(p, grid, warps, smem, st);
        case 7: return launch_fused<double, 2, kMidpoint, 1>(p, grid, warps, smem, st);
        case 8: return launch_fused<float, 2, kGL2, 1>(p, grid, warps, smem, st);
        case 9: return launch_fused<double, 2, kGL2, 1>(p, grid, warps, smem, st);
        case 10: return launch_fused<float, 2, kSimpson, 1>(p, grid, warps, smem, st);
        case 11: return launch_fused<double, 2, kSimpson, 1>(p, grid, warps, smem, st);
        case 12: return launch_fused<float, 2, kMidpoint, 2>(p, grid, warps, smem, st);
        case 13: return launch_fused<double, 2, kMidpoint, 2>(p, grid, warps, smem, st);
        case 14: return launch_fused<float, 2, kGL2, 2>(p, grid, warps, smem, st);
        case 15: return launch_fused<double, 2, kGL2, 2>(p, grid, warps, smem, st);
        case 16: return launch_fused<float, 2, kSimpson, 2>(p, grid, warps, smem, st);
        case 17: return launch_fused<double, 2, kSimpson, 2>(p, grid, warps, smem, st);
    }
    return cudaErrorInvalidValue;
}

int fused_blocks_per_sm_d2(int fp64, int integ, int warps, size_t smem, int cheb) {
    switch (cheb * 6 + integ * 2 + (fp64 ? 1 : 0)) {
        case 0: return fused_max_blocks_per_sm<float, 2, kMidpoint>(warps, smem);
        case 1: return fused_max_blocks_per_sm<double, 2, kMidpoint>(warps, smem);
        case 2: return fused_max_blocks_per_sm<float, 2, kGL2>(warps, smem);
        case 3: return fused_max_blocks_per_sm<double, 2, kGL2>(warps, smem);
        case 4: return fused_max_blocks_per_sm<float, 2, kSimpson>(warps, smem);
        case 5: return fused_max_blocks_per_sm<double, 2, kSimpson>(warps, smem);
        case 6: return fused_max_blocks_per_sm<float, 2, kMidpoint, 1>(warps, smem);
        case 7: return fused_max_blocks_per_sm<double, 2, kMidpoint, 1>(warps, smem);
        case 8: return fused_max_blocks_per_sm<float, 2, kGL2, 1>(warps, smem);
        case 9: return fused_max_blocks_per_sm<double, 2, kGL2, 1>(warps, smem);
        case 10: return fused_max_blocks_per_sm<float, 2, kSimpson, 1>(warps, smem);
        case 11: return fused_max_blocks_per_sm<double, 2, kSimpson, 1>(warps, smem);
        case 12: return fused_max_blocks_per_sm<float, 2, kMidpoint, 2>(warps, smem);
        case 13: return fused_max_blocks_per_sm<double, 2, kMidpoint, 2>(warps, smem);
        case 14: return fused_max_blocks_per_sm<float, 2, kGL2, 2>(warps, smem);
        case 15: return fused_max_blocks_per_sm<double, 2, kGL2, 2>(warps, smem);
        case 16: return fused_max_blocks_per_sm<float, 2, kSimpson, 2>(warps, smem);
        case 17: return fused_max_blocks_per_sm<double, 2, kSimpson, 2>(warps, smem);
    }
    return 0;
}

size_t fused_smem_d2(int fp64, int n_basis, int warps, int legacy) {
    (void)legacy;
    return fp64 ? fused_smem_bytes<double, 2>(n_basis, warps) : fused_smem_bytes<float, 2>(n_basis, warps);
}

int fused_groups_per_warp_d2(int fp64, int) { return fp64 ? Geo<double, 2>::GPW : Geo<float, 2>::GPW; }

int fused_max_warps_d2(int fp64, int) { return fp64 ? Geo<double, 2>::MAXW : Geo<float, 2>::MAXW; }

}  // namespace pm
