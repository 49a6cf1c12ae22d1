// Instantiations of the two-stream attention kernels for head_dim 128.
#include "attn_duo.cuh"

namespace wise {
cudaError_t launch_duo_d128(int block, int mode, const AttnLaunch& L) { return launch_duo_for_dim<128>(block, mode, L); }
}  // namespace wise
