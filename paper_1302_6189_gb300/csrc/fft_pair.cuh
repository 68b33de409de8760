// fft_pair.cuh -- two neighbouring axes of equal length of a complex64 array
// in one launch, with one trip through HBM instead of two.
//
// The lines of two axes depend on each other only inside a slab: the points
// that share all other coordinates (a plane, or some planes) or, for two outer
// axes, all of them but a block of neighbouring inner ones.  The kernel walks
// the slabs with both operations interleaved: A (the first axis) of slab
// i + D, then B (the second, in place) of slab i.  A slab is about 0.5 MB and
// D slabs are in flight, so B finds in L2 what A wrote and HBM sees the array
// read once and written once.
//
// Tiles are dealt by a ticket counter.  Tickets are drawn by running CTAs
// only, and every tile that a B tile waits for has a lower ticket, so it
// belongs to a CTA that runs or has finished; A tiles wait for nothing, hence
// every wait ends.  (Waits are bounded all the same: after wait_ns the kernel
// sets the plan's error flag and every CTA returns.)  The host chooses D so
// that the tickets between A's last tile of a slab and B's first cover all
// resident CTAs: B rarely waits.  The last CTA to leave zeroes the counters
// for the next launch: a CTA counts itself out with release and acquire, so
// that what it added to any counter comes before the zeroes.  (After complete waits the B
// tiles' acquires order this too; after one that gave up nothing else does.)
//
// What bounds it: the instructions of the two axes (27 to 31 us per axis and 2^24
// points at 256 points, where a trip through HBM takes 38; over the launch 60 %
// of the load/store data pipe and 58 % of the issue slots busy, most stalled
// warps at the CTA barriers, 50 % of the DRAM rate); both operations together
// take less than two trips, not one.  Whole transforms, one launch per axis
// before: 256^3 121 -> 109 us, 256^3 x 8 there and back 1,862 -> 1,639 us, 64^4 x 4
// 620 -> 539 us.
//
// A kernel per length: with every pair of lengths in one kernel (a switch) the
// tiles ran at 0.6 of this rate.
#pragma once

#include "fft_nat.cuh"
#include "ptx_sync.cuh"

namespace mdfft {

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t *p) {
    uint32_t v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void red_release(uint32_t *p, uint32_t v) {
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t add_acq_rel(uint32_t *p, uint32_t v) {
    uint32_t old;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
    return old;
}

// ticket -> operation, slab, tile: A of the first D slabs, then per slab i the
// A tiles of slab i + D and the B tiles of slab i, then B of the last D slabs
__device__ __forceinline__ void pair_ticket(const PairArgs &a, uint32_t t, int &op, uint32_t &slab, uint32_t &tile) {
    const uint32_t nA = a.op[0].tiles, nB = a.op[1].tiles, head = a.ahead * nA, steady = (a.slabs - a.ahead) * (nA + nB);
    if (t < head) {
        op = 0, slab = t / nA, tile = t - slab * nA;
    } else if (t - head < steady) {
        const uint32_t u = t - head, i = u / (nA + nB), r = u - i * (nA + nB);
        op = r < nA ? 0 : 1;
        slab = op ? i : i + a.ahead;
        tile = op ? r - nA : r;
    } else {
        const uint32_t u = t - head - steady, i = u / nB;
        op = 1, slab = a.slabs - a.ahead + i, tile = u - i * nB;
    }
}

// CTA: a row tile or G column tiles at a time (A of two outer axes: columns too)
template <int N, bool ROWS> struct PairCfg {
    using RC = RowCfg<float, N>;
    using CC = ColCfg<float, N>;
    static constexpr int THREADS = ROWS ? RC::THREADS : CC::THREADS, G = THREADS / CC::THREADS;
    static_assert(G * CC::THREADS == THREADS && N % CC::COLS == 0 && N % RC::LINES == 0, "whole tiles");
    static constexpr int NTW = tw_entries(radix_plan(N));
    static constexpr int BUF = ROWS && RC::LINES * RC::RS > G * N * CC::COLS ? RC::LINES * RC::RS : G * N * CC::COLS;
    static constexpr size_t SMEM = (size_t)(BUF + NTW) * sizeof(float2);
    static constexpr int MINB = 1280 / THREADS;
    // a ticket's tile is R of these: 128 bytes a thread, as much as leaves the
    // tiles of all resident CTAs (25 MB) well inside L2; smaller tickets cost
    // their barriers and fence more often
    static constexpr int POINTS = ROWS ? RC::LINES * N : N * CC::COLS;
    static constexpr int R = POINTS >= 16 * THREADS ? 1 : 16 * THREADS / POINTS;
};

template <int N, bool ROWS>
__global__ void __launch_bounds__(PairCfg<N, ROWS>::THREADS, PairCfg<N, ROWS>::MINB) fft_pair_kernel(const PairArgs a) {
    using PC = PairCfg<N, ROWS>;
    using CC = ColCfg<float, N>;
    using RC = RowCfg<float, N>;
    extern __shared__ __align__(16) unsigned char pair_smem[];
    __shared__ uint32_t s_ticket;
    float2 *buf = reinterpret_cast<float2 *>(pair_smem), *tw = buf + PC::BUF;
    const int tid = threadIdx.x;
    const uint32_t total = a.slabs * (a.op[0].tiles + a.op[1].tiles);
    follow_previous_launch();
    for (int i = tid; i < PC::NTW; i += PC::THREADS) tw[i] = __ldg(reinterpret_cast<const float2 *>(a.tw) + i);
    uint32_t next = 0;
    if (tid == 0) next = atomicAdd(a.sync, 1);
    for (;;) {
        int op = 0;
        uint32_t slab = 0, tile = 0;
        if (tid == 0) {
            if (next < total) {
                pair_ticket(a, next, op, slab, tile);
                if (op == 1 && ld_acquire(a.sync + 3 + slab) < a.op[0].tiles) {
                    const uint64_t t0 = global_timer_ns();
                    while (ld_acquire(a.sync + 3 + slab) < a.op[0].tiles) {
                        if (global_timer_ns() - t0 > a.wait_ns) {
                            atomicExch(a.sync + 2, 1);
                            if (a.err) *a.err = 1;
                        }
                        if (ld_acquire(a.sync + 2)) {
                            next = total;
                            break;
                        }
                    }
                }
            }
            s_ticket = next;
        }
        __syncthreads();
        const uint32_t t = s_ticket;
        if (t >= total) break;
        if (tid == 0) next = atomicAdd(a.sync, 1);  // (drawn a tile ahead: its latency is hidden)
        pair_ticket(a, t, op, slab, tile);
        const uint32_t u = slab / a.wblocks, wb = slab - u * a.wblocks;
        const int64_t base = (int64_t)u * a.outer + (int64_t)wb * a.W;
        // units (planes) of this slab; slabs of inner blocks hold one unit
        const uint32_t left = a.units - u * a.per_slab, units = left < a.per_slab ? left : a.per_slab;
#pragma unroll 1
        for (int r = 0; r < PC::R; ++r) {
            if (r > 0) __syncthreads();  // the exchange buffer is free again
            const uint32_t part = tile * PC::R + r;
            int me = tid;  // (opaque: a tile's addresses are worked out per tile, not kept around the loop)
            asm volatile("" : "+r"(me));
            if (ROWS && op == 0) {
                if (part * RC::LINES < units * N) {
                    const int64_t at = base + (int64_t)part * (RC::LINES * N);
                    RowParts<float, N, 0, true>::run(reinterpret_cast<const float2 *>(a.op[0].io.in) + at,
                                                     reinterpret_cast<float2 *>(a.op[0].io.out) + at, buf, tw, me, RC::LINES, a.op[0].io);
                }
            } else {
                const int sub = PC::G > 1 ? me / CC::THREADS : 0, m = me - sub * CC::THREADS;
                const int col = m % CC::COLS, th = m / CC::COLS;
                const PairOp &o = a.op[ROWS ? 1 : 0];  // (columns: lengths and blocks of both operations alike)
                const uint32_t ct = part * PC::G + sub, j = ct / o.k;
                const bool ok = !ROWS || j < units;
                const int64_t wat = base + (int64_t)(ct - j * o.k) * CC::COLS + col;
                if (ROWS || op == 1) {
                    const int64_t at = wat + (int64_t)j * a.op[1].step;
                    ColParts<float, N, 0, true>::run(reinterpret_cast<const float2 *>(a.op[1].io.in) + at,
                                                     reinterpret_cast<float2 *>(a.op[1].io.out) + at, buf + sub * (N * CC::COLS), tw,
                                                     col, th, ok, a.op[1].io);
                } else {
                    const int64_t at = wat + (int64_t)j * a.op[0].step;
                    ColParts<float, N, 0, true>::run(reinterpret_cast<const float2 *>(a.op[0].io.in) + at,
                                                     reinterpret_cast<float2 *>(a.op[0].io.out) + at, buf + sub * (N * CC::COLS), tw,
                                                     col, th, ok, a.op[0].io);
                }
            }
        }
        __syncthreads();  // every store of the tile is issued, shared memory is free
        if (op == 0 && tid == 0) {
            __threadfence();
            red_release(a.sync + 3 + slab, 1);
        }
    }
    if (tid == 0 && add_acq_rel(a.sync + 1, 1) == gridDim.x - 1) {  // last one out
        for (uint32_t s = 0; s < a.slabs; ++s) a.sync[3 + s] = 0;
        a.sync[0] = a.sync[1] = a.sync[2] = 0;
    }
}

}  // namespace mdfft
