// Instances of the projections over few token rows.
#include "xsm_proj_few.cuh"

namespace xsm {

cudaError_t few_8_2_4(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) { return launch_few<8, 2, false, 4>(D, A, smem, L); }
cudaError_t few_8_2_8(const Dev &D, const ProjArgs &A, int smem, const ChainLaunch &L) { return launch_few<8, 2, false, 8>(D, A, smem, L); }

}  // namespace xsm
