// Resident CG blocks: 16-bit links, 20-bit spinors, FP32 compute.
#include "cg_block.cuh"

namespace hisq {
bool launch_cg_block_int20(int long_recon, const CGBlockShape &sh, const CGBlockArgs &a, cudaStream_t s)
{
    return launch_cg_block_t<G_FIX16, S_INT20>(long_recon, sh, a, s);
}
}  // namespace hisq
