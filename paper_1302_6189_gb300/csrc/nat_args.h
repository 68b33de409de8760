// nat_args.h -- launch arguments of the layout-keeping kernels (fft_nat.cuh).
#pragma once

#include "fft_pass.cuh"

namespace mdfft {

struct NatArgs {
    const void *in;
    void *out;        // may be `in`
    const void *tw;   // twiddle table of radix_plan(N) (tw_offset layout)
    uint32_t nlines;  // line l starts at (l / stride) N stride + l mod stride
    int64_t stride;   // distance of a line's points (1: rows)
    FastDiv fd;       // the stride as a divisor
    int conj;         // bit 0 conjugates the loaded input, bit 1 the stored output
    int scaled;       // scale != 1
    double scale;     // multiplies every stored value
};

}  // namespace mdfft
