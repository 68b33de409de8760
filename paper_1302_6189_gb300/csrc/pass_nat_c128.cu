// pass_nat_c128.cu -- the layout-keeping kernels of complex128.
#include "pass_nat.cuh"

namespace mdfft {
bool find_nat_kernel_c128(int64_t n, bool rows, PassKernel *k) { MDFFT_FIND_NAT(double, MDFFT_NAT_LENGTHS_C128) }
}  // namespace mdfft
