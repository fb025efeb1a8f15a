// Resident CG blocks: 16-bit links and spinors, FP32 compute.
#include "cg_block.cuh"

namespace hisq {
bool launch_cg_block_half(int long_recon, const CGBlockShape &sh, const CGBlockArgs &a, cudaStream_t s)
{
    return launch_cg_block_t<G_FIX16, S_HALF>(long_recon, sh, a, s);
}
}  // namespace hisq
