// pass_nat.cuh -- registry body of the layout-keeping kernels of one precision.
#pragma once

#include "fft_nat.cuh"
#include "passes.h"

namespace mdfft {

template <typename Real, int N> static PassKernel make_nat(bool rows) {
    using CC = ColCfg<Real, N>;
    using RC = RowCfg<Real, N>;
    if (rows)
        return PassKernel{(const void *)&fft_nat_row_kernel<Real, N>, RC::THREADS, RC::LINES, RC::Cfg::TL, RC::SMEM, RC::Cfg::plan};
    return PassKernel{(const void *)&fft_nat_col_kernel<Real, N>, CC::THREADS, CC::COLS, CC::Cfg::TL, CC::SMEM, CC::Cfg::plan};
}

template <typename Real> static bool find_nat(int64_t n, bool rows, PassKernel *k) {
    switch (n) {
#define MDFFT_CASE(N)                       \
    case N:                                 \
        *k = make_nat<Real, N>(rows);       \
        return true;
        MDFFT_NAT_LENGTHS(MDFFT_CASE)
#undef MDFFT_CASE
        default:
            return false;
    }
}

}  // namespace mdfft
