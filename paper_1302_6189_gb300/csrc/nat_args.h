// nat_args.h -- launch arguments of the layout-keeping kernels (fft_nat.cuh, fft_pair.cuh).
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

// Two neighbouring axes of equal length N in one launch (fft_pair.cuh).  Tile
// c of an operation on columns covers the lines (j, w block): j = c / k, which
// start at slab base + j step + (c mod k) COLS.
struct PairOp {
    NatArgs io;       // in, out, stride, conj, scale of the operation (nlines, fd, tw unused)
    uint32_t tiles;   // tiles of a whole slab
    uint32_t k;
    int64_t step;
};

struct PairArgs {
    PairOp op[2];
    const void *tw;
    uint32_t slabs, ahead;     // ahead: slabs that the first operation runs ahead of the second
    uint32_t wblocks;          // slabs per outer index (blocks of W inner points); 1: slabs of whole planes
    uint32_t W;
    int64_t outer;             // element distance of the slabs' outer index
    uint32_t units, per_slab;  // planes in all and per slab (blocks: outer indices, 1)
    uint32_t *sync;            // [0] ticket, [1] CTAs done, [2] abort, [3 + s] first operation's tiles done in slab s
    int *err;
    uint64_t wait_ns;          // a wait that takes longer gives up
};

}  // namespace mdfft
