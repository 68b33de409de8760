// pass_pair.cu -- the two-axis kernels of complex64 (fft_pair.cuh).
#include "fft_pair.cuh"
#include "passes.h"

namespace mdfft {

template <int N, bool ROWS> static PassKernel make_pair(int *row_tile, int *col_tile, int *g, int *r) {
    using PC = PairCfg<N, ROWS>;
    PassKernel k{};
    k.fn = (const void *)&fft_pair_kernel<N, ROWS>;
    k.threads = PC::THREADS;
    k.smem = PC::SMEM;
    k.persistent = 1;
    *row_tile = RowCfg<float, N>::LINES, *col_tile = ColCfg<float, N>::COLS, *g = PC::G, *r = PC::R;
    return k;
}

// 64, 128 and 256: the lengths whose two axes take clearly less than two trips
// through HBM (512-point columns take longer than a trip by themselves)
bool find_pair_kernel(int64_t n, bool rows, PassKernel *k, int *row_tile, int *col_tile, int *g, int *r) {
    if (n == 64) *k = rows ? make_pair<64, true>(row_tile, col_tile, g, r) : make_pair<64, false>(row_tile, col_tile, g, r);
    else if (n == 128) *k = rows ? make_pair<128, true>(row_tile, col_tile, g, r) : make_pair<128, false>(row_tile, col_tile, g, r);
    else if (n == 256) *k = rows ? make_pair<256, true>(row_tile, col_tile, g, r) : make_pair<256, false>(row_tile, col_tile, g, r);
    else return false;
    return true;
}

}  // namespace mdfft
