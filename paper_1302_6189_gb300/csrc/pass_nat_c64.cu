// pass_nat_c64.cu -- the layout-keeping kernels of complex64.
#include "pass_nat.cuh"

namespace mdfft {
bool find_nat_kernel_c64(int64_t n, bool rows, PassKernel *k) { MDFFT_FIND_NAT(float, MDFFT_NAT_LENGTHS) }
}  // namespace mdfft
