// Instantiations of the two-stream attention kernels for head_dim 64.
#include "attn_duo.cuh"

namespace wise {
cudaError_t launch_duo_d64(int block, int mode, const AttnLaunch& L) { return launch_duo_for_dim<64>(block, mode, L); }
}  // namespace wise
