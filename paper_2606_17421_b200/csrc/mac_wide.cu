// The multiply-accumulate for rings with a ciphertext prime of 2^50 or more (instances apart: they compile side by side).
#include "mac_kernel.cuh"

namespace bf {

cudaError_t launch_mac_wide(const MacLaunch& m) { return launch_mac_ring<false>(m); }

}  // namespace bf
