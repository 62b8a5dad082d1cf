// Instances of the projections over few token rows.
#include "xsm_proj_few.cuh"

namespace xsm {

cudaError_t few_8_1_packed_4(const Dev &, const ProjArgs &, int, const ChainLaunch &);
cudaError_t few_8_1_4(const Dev &, const ProjArgs &, int, const ChainLaunch &);
cudaError_t few_8_1_packed_8(const Dev &, const ProjArgs &, int, const ChainLaunch &);
cudaError_t few_8_1_8(const Dev &, const ProjArgs &, int, const ChainLaunch &);
cudaError_t few_8_2_4(const Dev &, const ProjArgs &, int, const ChainLaunch &);
cudaError_t few_8_2_8(const Dev &, const ProjArgs &, int, const ChainLaunch &);

static cudaError_t few_15_1_packed_9(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) { return launch_few<15, 1, true, 9>(D, A, smem, L); }
static cudaError_t few_15_1_9(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) { return launch_few<15, 1, false, 9>(D, A, smem, L); }
static cudaError_t few_15_2_4(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) { return launch_few<15, 2, false, 4>(D, A, smem, L); }

cudaError_t launch_proj_few(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) {
    const FewShape f = few_shape(A.rows, A.kdim);
    if (f.warps == 15) return f.nt == 2 ? few_15_2_4(D, A, smem, L) : f.pack ? few_15_1_packed_9(D, A, smem, L) : few_15_1_9(D, A, smem, L);
    if (f.blocks == 8) return f.nt == 2 ? few_8_2_8(D, A, smem, L) : f.pack ? few_8_1_packed_8(D, A, smem, L) : few_8_1_8(D, A, smem, L);
    return f.nt == 2 ? few_8_2_4(D, A, smem, L) : f.pack ? few_8_1_packed_4(D, A, smem, L) : few_8_1_4(D, A, smem, L);
}

}  // namespace xsm
