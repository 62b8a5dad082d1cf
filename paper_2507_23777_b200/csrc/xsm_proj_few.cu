// Instances of the projections over few token rows.
#include "xsm_proj_few.cuh"

namespace xsm {

cudaError_t launch_proj_few(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
    const FewShape f = few_shape(A.rows, A.kdim);
    if (!f.pack) return f.nt == 1 ? launch_few<8, 1, false, 4>(D, A, smem, L) : launch_few<8, 2, false, 4>(D, A, smem, L);
    return f.warps == 15 ? launch_few<15, 1, true, 9>(D, A, smem, L) : f.blocks == 8 ? launch_few<8, 1, true, 8>(D, A, smem, L) : launch_few<8, 1, true, 4>(D, A, smem, L);
}

}  // namespace xsm
