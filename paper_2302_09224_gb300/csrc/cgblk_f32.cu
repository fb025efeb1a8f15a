// Resident CG blocks: FP32 links and spinors, FP32 compute.
#include "cg_block.cuh"

namespace hisq {
bool launch_cg_block_f32(int long_recon, const CGBlockShape &sh, const CGBlockArgs &a, cudaStream_t s)
{
    return launch_cg_block_t<G_F32, S_F32>(long_recon, sh, a, s);
}
}  // namespace hisq
