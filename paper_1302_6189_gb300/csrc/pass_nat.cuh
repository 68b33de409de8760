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

#define MDFFT_FIND_NAT(Real, LENGTHS)              \
    switch (n) {                                   \
        LENGTHS(MDFFT_NAT_CASE_##Real)             \
        default:                                   \
            return false;                          \
    }
#define MDFFT_NAT_CASE_float(N) \
    case N:                     \
        *k = make_nat<float, N>(rows); \
        return true;
#define MDFFT_NAT_CASE_double(N) \
    case N:                      \
        *k = make_nat<double, N>(rows); \
        return true;

}  // namespace mdfft
