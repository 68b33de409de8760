// fft_nat.cuh -- line transforms of one axis of a dense row-major array that
// keep its layout: every line is stored back to the places it was read from.
//
// A redistribution changes which process owns a point, not its value; on one
// GPU every process's chunk lies in the same HBM, so an execution that does
// not count moved points can transform the axes of a plan's transpose order
// one after another without moving anything.  The butterflies, twiddles and
// their order are those of fft_pass_kernel (the default radix plan), so the
// results are bit-identical to the pass kernels'.
//
// What changes is the work around the butterflies.  A pass kernel exchanges
// the line between its radix stages through shared memory and then transposes
// the tile through shared memory once more, with a CTA barrier on each side.
// Here the stages run in place: stage s leaves its R outputs where its R
// inputs were (the digits of the index come out reversed), so one barrier
// lies between stages and the last one stores straight from registers, at the
// output index its digits stand for.
//  * columns (fft_nat_col_kernel): an axis whose points lie `stride` apart.
//    A CTA takes COLS lines that are neighbours in memory; a thread works on
//    one of them, lanes side by side, so loads and stores are runs of COLS
//    points and the exchange buffer [point][column] has no bank conflicts.
//  * rows (fft_nat_row_kernel): the contiguous axis.  TL threads share a line;
//    if they lie in one warp no CTA barrier is needed at all.
// Stages are merged into parts of about 16 points that one thread runs in
// registers (Parts): 12 = 4 x 3 or 20 = 4 x 5 take no exchange, 96 = 8 x (4 x 3)
// one instead of two.
//
// What bounds them: HBM or, for arrays under about 100 MB, L2 (both at 0.9 and
// more of the rate for 8 to 128 and 256 points; the lengths with a third part
// or an odd last part at 0.75 to 0.9, by instructions and barriers).  Measured
// per launch over 2^25 points, GB/s, the pass kernel before (row and column
// launches together: N x N planes), rows and columns now: N = 24 3,000 -> 6,070,
// 32 4,040 -> 6,020, 96 4,130 -> 5,180, 160 3,940 -> 5,090, 256 5,520 -> 5,960,
// 512 4,610 -> 5,180; whole transforms: 24^5 170 -> 76 us (64 MB, in L2), 256^3
// 142 -> 121 us (109 with fft_pair.cuh), 512^3 1,190 -> 1,060 us.  Counters
// (single precision): 256-point columns 74 % of the DRAM rate and 48 % of the
// load/store data pipe; 24-point rows 90 % of that pipe, their columns 60 %;
// 512-point rows 79 % of it at 85 % of the DRAM rate, their columns 30 warps per
// SM (63 registers) at 70 %; 240-point columns 19 warps (80 registers).
// Double precision: the FP64 units (a warp instruction holds one for 64
// cycles), so lanes must not idle and small grids need many short-lived warps
// spread over the SMs: 32^3 25.6 -> 14.9 us, 64^3 44.2 -> 32.8, 128^3 274 -> 245,
// 48 x 48 planes (2^22 points) 390 -> 270, 256 x 256 399 -> 371; 256^3 runs 22.25
// FP64 instructions per point and axis in 2,121 us, their issue time being 2,119.
#pragma once

#include "nat_args.h"

namespace mdfft {

// Consecutive radix stages of a plan merged into parts that one thread runs
// in registers: as few parts as a size of at most `lim` points allows, then
// the smallest largest part.
struct Parts {
    int n = 0;
    int size[12] = {0}, first[12] = {0}, count[12] = {0};
    int max = 1;
};
__host__ __device__ constexpr Parts parts_of(const RadixPlan &p, int lim) {
    Parts best;
    if (p.S <= 0) return best;
    best.n = 100;
    for (int cut = 0; cut < (1 << (p.S - 1)); ++cut) {
        Parts c;
        int sz = 1, f = 0;
        bool ok = true;
        for (int s = 0; s < p.S; ++s) {
            sz *= p.R[s];
            if (s != p.S - 1 && !((cut >> s) & 1)) continue;
            ok = ok && sz <= lim;
            c.size[c.n] = sz, c.first[c.n] = f, c.count[c.n] = s + 1 - f;
            c.max = sz > c.max ? sz : c.max;
            c.n++;
            sz = 1, f = s + 1;
        }
        if (ok && (c.n < best.n || (c.n == best.n && c.max < best.max))) best = c;
    }
    return best;
}

// radix of stage S and points combined before it, as plain constants (usable in device code)
template <int N, int S> constexpr int kRadix = radix_plan(N).R[S];
__host__ __device__ constexpr int ns_of(const RadixPlan &p, int s) {
    int v = 1;
    for (int i = 0; i < s; ++i) v *= p.R[i];
    return v;
}
template <int N, int S> constexpr int kNs = ns_of(radix_plan(N), S);

// index k (twiddle / output order) of the first S stages' digits -> their
// place p: k = r_0 + r_1 R_0 + ..., p = (r_0 R_1 + r_1) R_2 + ...
template <int N, int S, int AT = 0> __device__ __forceinline__ int digits_place(int k, int p = 0) {
    if constexpr (AT == S) {
        return p;
    } else {
        constexpr int R = kRadix<N, AT>;
        return digits_place<N, S, AT + 1>((int)((unsigned)k / (unsigned)R), p * R + (int)((unsigned)k % (unsigned)R));
    }
}
// output index of place idx of the digits of stages [F, F + C), most significant digit first
template <int N, int F, int C> __host__ __device__ constexpr int digits_out(int idx) {
    if constexpr (C == 0) {
        return 0;
    } else {
        constexpr int R = kRadix<N, F + C - 1>, NS = kNs<N, F + C - 1>;
        return (idx % R) * NS + digits_out<N, F, C - 1>(idx / R);
    }
}

// Size limit of a part.  Columns and rows of one kernel launch over 2^25
// points, GB/s: 192 = 8 x 8 x 3 6,190 / 5,680, as 8 x 24 (fewer exchanges, 80
// registers) 5,030 / 4,740; 512 = 16 x 16 x 2 5,380 / 6,400, as 16 x 32 4,520 /
// 5,590; but 480 = 32 x 15 5,090 in columns, as 8 x 4 x 15 4,080.
__host__ __device__ constexpr int nat_lim(int n, bool dbl, bool rows) {
    // double precision: chains as short as the widest stage allows below 60
    // points, where small grids leave most FP64 units idle
    if (dbl) return n >= 60 ? 16 : radix_plan(n).maxR > 8 ? radix_plan(n).maxR : 8;
    return n <= 20 ? 20 : n == 480 && !rows ? 32 : 16;
}

template <typename Real, int N, bool ROWS> struct NatCfg {
    using C = typename Cx<Real>::T;
    static constexpr RadixPlan plan = radix_plan(N);
    static constexpr Parts parts = parts_of(plan, nat_lim(N, sizeof(Real) == 8, ROWS));
    static_assert(parts.n >= 1 && parts.n <= 4, "line length");
    static constexpr int TL = N / parts.max;  // threads per line
    __host__ __device__ static constexpr int before(int i) {  // product of the parts before part i
        int v = 1;
        for (int q = 0; q < i; ++q) v *= parts.size[q];
        return v;
    }
    __host__ __device__ static constexpr int dist(int i) { return N / (before(i) * parts.size[i]); }  // element distance in part i
};

// The radix stages of part PI on the SIZE points of v; twk: the twiddle table
// advanced by the output index of the digits before the part.
template <typename Real, int N, bool ROWS, int PI, int SI = 0> struct PartStages {
    using Cfg = NatCfg<Real, N, ROWS>;
    using C = typename Cfg::C;
    static constexpr Parts P = Cfg::parts;
    static constexpr int FIRST = P.first[PI], COUNT = P.count[PI], SIZE = P.size[PI];
    static constexpr int S = FIRST + SI, R = kRadix<N, S>, NS = kNs<N, S>;
    static constexpr int TWOFF = tw_offset(Cfg::plan, S);
    // place of a point: (digits done, digit of this stage, digits to come)
    static constexpr int D = SIZE * ns_of(Cfg::plan, FIRST) / ns_of(Cfg::plan, S + 1);
    static constexpr int PB = SIZE / (R * D);
    template <int B> __device__ __forceinline__ static void block(C (&v)[SIZE], const C *twk) {
        if constexpr (B < PB) {
            constexpr int K = digits_out<N, FIRST, SI>(B);
            C w[R];
            if constexpr (NS > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) w[r] = twk[TWOFF + r * NS + K];
            }
#pragma unroll
            for (int q = 0; q < D; ++q) {
                C u[R];
#pragma unroll
                for (int r = 0; r < R; ++r) u[r] = v[(B * R + r) * D + q];
                if constexpr (NS > 1) {
#pragma unroll
                    for (int r = 1; r < R; ++r) u[r] = cmul(u[r], w[r]);
                }
                dft<R>(u);
#pragma unroll
                for (int r = 0; r < R; ++r) v[(B * R + r) * D + q] = u[r];
            }
            block<B + 1>(v, twk);
        }
    }
    __device__ __forceinline__ static void run(C (&v)[SIZE], const C *twk) {
        block<0>(v, twk);
        if constexpr (SI + 1 < COUNT) PartStages<Real, N, ROWS, PI, SI + 1>::run(v, twk);
    }
};

// (the data passes through once: no L1 allocation, so that the twiddles stay;
// an ordinary load, as the same kernel stores to these places in place)
__device__ __forceinline__ float2 ld_stream(const float2 *p) {
    float2 v;
    asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_stream(const double2 *p) {
    double2 v;
    asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// (written by other SMs in the same launch, fft_pair.cuh: not from L1)
__device__ __forceinline__ float2 ld_l2(const float2 *p) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
// (runs shorter than a sector or two: the rest of the sector is read soon, from L1)
__device__ __forceinline__ float2 ld_cached(const float2 *p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ double2 ld_cached(const double2 *p) {
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p));
    return v;
}

// The launches of an execution follow each other by programmatic dependence:
// the next one is set up as this one's CTAs leave, and waits here until this
// one is complete and its stores are visible.  (60 x 240 x 160: 28.7 -> 21.8 us
// for three launches, 24^5 87.1 -> 75.6 us for five, 256^3 130 -> 121 us.)  The
// kernels do not let it start any earlier (griddepcontrol.launch_dependents):
// CTAs set up while others still run take the places that happen to be free,
// and the uneven spread cost more than the wait saved (80^3 13.4 us against
// 8.7, 128^3 19.0 / 15.3, 16^5 20.4 / 13.9; complex128 64^3 87 / 34.5).
__device__ __forceinline__ void follow_previous_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// In double precision nothing but the butterflies may issue FP64 instructions:
// one that is predicated off takes its 64 cycles all the same, and the compiler
// predicates these short blocks.  So a sign is flipped as an integer, and the
// scaled stores stand in a block of their own, which stays a branch.  (48-point
// columns: 911 FP64 instructions per CTA as predicated blocks, 764 needed.)
__device__ __forceinline__ double flip_sign(double x, unsigned on) {
    return __hiloint2double(__double2hiint(x) ^ (int)(on << 31), __double2loint(x));
}
// conjugation of the first pass's input
template <typename C, int SIZE> __device__ __forceinline__ void load_conj(C (&v)[SIZE], const NatArgs &a) {
    if constexpr (sizeof(v[0].x) == 8) {
#pragma unroll
        for (int r = 0; r < SIZE; ++r) v[r].y = flip_sign(v[r].y, a.conj & 1);
    } else if (a.conj & 1) {
#pragma unroll
        for (int r = 0; r < SIZE; ++r) v[r].y = -v[r].y;
    }
}
template <typename C, int SIZE> __device__ __forceinline__ void zero_all(C (&v)[SIZE]) {
#pragma unroll
    for (int r = 0; r < SIZE; ++r) v[r] = C{0, 0};
}
// conjugation and scale of the last pass, as store_tile applies them, and the
// store: put(r, value) for every point
template <typename C, int SIZE, typename Put> __device__ __forceinline__ void finish_store(C (&v)[SIZE], const NatArgs &a, const Put &put) {
    using Real = decltype(v[0].x);
    if constexpr (sizeof(Real) == 8) {
#pragma unroll
        for (int r = 0; r < SIZE; ++r) v[r].y = flip_sign(v[r].y, (a.conj >> 1) & 1);
        if (a.scaled) {
#pragma unroll
            for (int r = 0; r < SIZE; ++r) put(r, C{v[r].x * a.scale, v[r].y * a.scale});
            asm volatile("" ::: "memory");  // (the two blocks' stores are not merged)
            return;
        }
    } else if ((a.conj & 2) || a.scaled) {
        const Real sc = (Real)a.scale, sy = (a.conj & 2) ? -sc : sc;
#pragma unroll
        for (int r = 0; r < SIZE; ++r) v[r] = C{v[r].x * sc, v[r].y * sy};
    }
#pragma unroll
    for (int r = 0; r < SIZE; ++r) put(r, v[r]);
}

// ------------------------------------------------------------------ columns

template <typename Real, int N> struct ColCfg {
    using Cfg = NatCfg<Real, N, false>;
    using C = typename Cfg::C;
    // runs of at least 128 bytes (64-byte runs with half the threads: 384
    // columns 4,890 GB/s against 6,070), and at least 128 threads (96 columns
    // 5,970 GB/s with 128 threads, 5,530 with 256)
    static constexpr int MINC = 128 / (int)sizeof(C);
    // double precision: an FP64 instruction takes a full warp's time whatever
    // its live lanes, so a warp's 32 / c butterflies of a line have to fit every
    // part's count up to 1/15 of idle lanes; then the smallest CTA
    __host__ __device__ static constexpr bool full_warps(int c) {
        const int w = 32 / c;
        if (Cfg::TL % w && Cfg::TL != 15) return false;
        for (int i = 0; i < Cfg::parts.n; ++i) {
            const int nb = N / Cfg::parts.size[i];
            if (15 * ((nb + w - 1) / w * w) > 16 * nb) return false;
        }
        return true;
    }
    static constexpr int cols() {
        int c = MINC;
        if (sizeof(Real) == 8) {
            while (c < 32 && !full_warps(c) && 2 * c * Cfg::TL <= 512) c *= 2;
            while (c * Cfg::TL < 32) c *= 2;
        } else {
            while (c * Cfg::TL < 96 && c < 128) c *= 2;
        }
        return c;
    }
    static constexpr int COLS = cols();
    static constexpr int THREADS = COLS * Cfg::TL;
    static_assert(THREADS <= 1024, "CTA shape");
    // exchange buffer [N][COLS], then the twiddle table
    static constexpr size_t SMEM = Cfg::parts.n == 1 ? 0 : ((size_t)N * COLS + tw_entries(Cfg::plan)) * sizeof(C);
};

// LOOP: the tile runs in a loop over tiles.  Points of absent lines then get
// defined values: left alone, their registers would stay live around the loop
// (and defining them where there is none costs 10 to 50 registers).
template <typename Real, int N, int PI, bool LOOP> struct ColParts {
    using Cfg = NatCfg<Real, N, false>;
    using C = typename Cfg::C;
    static constexpr int COLS = ColCfg<Real, N>::COLS;
    static constexpr int SIZE = Cfg::parts.size[PI], D = Cfg::dist(PI), B = Cfg::before(PI);
    static constexpr int STAGES = Cfg::parts.first[PI], COUNT = Cfg::parts.count[PI];
    static constexpr int NB = N / SIZE, PER = (NB + Cfg::TL - 1) / Cfg::TL;  // butterflies per line, per thread
    static constexpr bool FIRST = PI == 0, LAST = PI == Cfg::parts.n - 1;

    __device__ __forceinline__ static void run(const C *src, C *dst, C *buf, const C *tw, int col, int t, bool ok,
                                               const NatArgs &a) {
        C v[PER][SIZE];
        int k[PER], at[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            // butterfly b: output index k of the digits before this part, then the place of its first point
            const int b = t + i * Cfg::TL;
            const bool live = NB % Cfg::TL == 0 || b < NB;
            k[i] = (int)((unsigned)b % (unsigned)B);
            at[i] = digits_place<N, STAGES>(k[i]) * (N / B) + (int)((unsigned)b / (unsigned)B);
            if constexpr (FIRST) {
                if (live && ok) {
                    const C *p = src + (int64_t)at[i] * a.stride;
#pragma unroll
                    for (int r = 0; r < SIZE; ++r) {
                        if constexpr (LOOP) v[i][r] = ld_l2(p + (int64_t)(r * D) * a.stride);
                        else v[i][r] = ld_stream(p + (int64_t)(r * D) * a.stride);
                    }
                    load_conj(v[i], a);
                } else if constexpr (LOOP) {
                    zero_all(v[i]);
                }
            } else if (live) {
#pragma unroll
                for (int r = 0; r < SIZE; ++r) v[i][r] = buf[(at[i] + r * D) * COLS + col];
            } else if constexpr (LOOP) {
                zero_all(v[i]);
            }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int b = t + i * Cfg::TL;
            if (NB % Cfg::TL != 0 && b >= NB) continue;
            PartStages<Real, N, false, PI>::run(v[i], tw + k[i]);
            if constexpr (!LAST) {
#pragma unroll
                for (int r = 0; r < SIZE; ++r) buf[(at[i] + r * D) * COLS + col] = v[i][r];
            } else if (ok) {
                C *p = dst + (int64_t)k[i] * a.stride;
                finish_store(v[i], a, [&](int r, C x) { p[(int64_t)digits_out<N, STAGES, COUNT>(r) * a.stride] = x; });
            }
        }
        if constexpr (!LAST) {
            __syncthreads();
            ColParts<Real, N, PI + 1, LOOP>::run(src, dst, buf, tw, col, t, ok, a);
        }
    }
};

// Lines l0 .. l0 + COLS - 1 by the whole CTA (tw: the twiddles, staged when the length has an exchange).
template <typename Real, int N, bool LOOP = false, typename C = typename Cx<Real>::T>
__device__ __forceinline__ void nat_col_tile(const C *in, C *out, C *buf, const C *tw, int tid, uint32_t l0, const NatArgs &a) {
    using CC = ColCfg<Real, N>;
    const int col = tid % CC::COLS, t = tid / CC::COLS;
    const uint32_t l = l0 + col, o = fastdiv(l, a.fd);
    const int64_t base = (int64_t)o * N * a.stride + (l - o * a.fd.d);
    ColParts<Real, N, 0, LOOP>::run(in + base, out + base, buf, tw, col, t, l < a.nlines, a);
}

template <typename Real, int N>
__global__ void __launch_bounds__(ColCfg<Real, N>::THREADS) fft_nat_col_kernel(const NatArgs a) {
    using CC = ColCfg<Real, N>;
    using Cfg = NatCfg<Real, N, false>;
    using C = typename Cfg::C;
    extern __shared__ __align__(16) unsigned char nat_smem[];
    C *buf = reinterpret_cast<C *>(nat_smem);
    const int tid = threadIdx.x;
    const C *tw = reinterpret_cast<const C *>(a.tw);
    follow_previous_launch();
    if constexpr (Cfg::parts.n > 1) {  // twiddles to shared memory; the barrier after the first part covers them
        C *stw = buf + N * CC::COLS;
        for (int q = tid; q < tw_entries(Cfg::plan); q += CC::THREADS) stw[q] = __ldg(tw + q);
        tw = stw;
        if constexpr (Cfg::parts.count[0] > 1) __syncthreads();
    }
    nat_col_tile<Real, N>(reinterpret_cast<const C *>(a.in), reinterpret_cast<C *>(a.out), buf, tw, tid, blockIdx.x * CC::COLS, a);
}

// ------------------------------------------------------------------ rows

// Shared-memory place of point x of a row: one element of padding every g,
// rows of N + N / g + e elements.  Per length the pair whose accesses, replayed
// for every part (half-warps; quarter-warps in double precision), take the
// fewest wavefronts: at most 1.6 (480 points) times the conflict-free count.
struct NatPad {
    int n, g, e;
};
__host__ __device__ constexpr NatPad nat_pad(int n, bool dbl, int parts) {
    constexpr int none = 4096;
    constexpr NatPad c64[] = {{24, 3, 3},    {30, none, 5}, {32, 8, 0},   {40, 5, 5},    {48, none, 3}, {60, none, 0},
                              {64, 8, 0},    {80, none, 5}, {96, 48, 0},  {120, none, 0}, {128, 16, 0}, {160, 10, 5},
                              {192, 12, 1},  {240, none, 0}, {256, 16, 0}, {320, 20, 1},  {384, 48, 0}, {480, 10, 0},
                              {512, 32, 0},  {640, 40, 8},  {768, 48, 0}, {960, 20, 0},  {1024, 64, 0}};
    constexpr NatPad c128[] = {{10, 5, 1},    {12, none, 0}, {15, none, 0},  {20, 5, 5},   {24, none, 3}, {30, none, 1},
                               {32, 8, 0},    {40, none, 5}, {48, none, 3},  {60, 64, 0},  {64, 8, 0},    {80, none, 5},
                               {96, 24, 0},   {120, none, 7}, {128, 8, 0},   {160, 40, 0}, {192, 24, 0},  {240, none, 7},
                               {256, 16, 0},  {320, 40, 0},  {384, 24, 0},   {480, 20, 6}, {512, 32, 0},  {640, 40, 0},
                               {768, 48, 0},  {960, 40, 0},  {1024, 64, 0}};
    if (parts > 1) {
        if (dbl) {
            for (const NatPad &p : c128)
                if (p.n == n) return p;
        } else {
            for (const NatPad &p : c64)
                if (p.n == n) return p;
        }
    }
    return {n, none, n % 2 ? 0 : 1};  // one thread per row: odd row stride
}

template <typename Real, int N> struct RowCfg {
    using Cfg = NatCfg<Real, N, true>;
    using C = typename Cfg::C;
    static constexpr NatPad PAD = nat_pad(N, sizeof(Real) == 8, Cfg::parts.n);
    static constexpr int G = PAD.g, RS = N + N / G + PAD.e;
    // every part has TL butterflies per line, and a line's threads lie in one warp
    __host__ __device__ static constexpr bool even() {
        for (int i = 0; i < Cfg::parts.n; ++i)
            if (Cfg::parts.size[i] != Cfg::parts.max) return false;
        return 32 % Cfg::TL == 0;
    }
    static constexpr bool WARP = even();
    static constexpr int lines() {
        if (sizeof(Real) == 8) {  // full warps in every part (see ColCfg), in a small CTA
            for (int c = 1; c * Cfg::TL <= 160; ++c) {
                bool full = c * Cfg::TL > 16 && (Cfg::parts.n > 1 || c % 32 == 0);
                for (int i = 0; i < Cfg::parts.n; ++i) {
                    const int items = c * (N / Cfg::parts.size[i]);
                    full = full && 15 * ((items + 31) / 32 * 32) <= 16 * items;
                }
                if (full) return c;
            }
            return 160 / Cfg::TL;
        }
        const int l = (Cfg::parts.n == 1 ? 128 : 256) / Cfg::TL;
        return l < 1 ? 1 : l;
    }
    static constexpr int LINES = lines();
    static constexpr int THREADS = sizeof(Real) == 8 ? (LINES * Cfg::TL + 31) / 32 * 32 : LINES * Cfg::TL;
    static_assert(THREADS <= 1024, "CTA shape");
    static constexpr size_t SMEM = (size_t)LINES * RS * sizeof(C);
    // registers for 40 warps per SM (48 a thread; 32 warps with a 15-point part
    // or a multiple of 80 points, whose parts need more; 6 CTAs where a thread
    // holds a line of 20 points): uncapped the compiler spends 60 to 110 on the
    // same code and the warps are missed
    static constexpr int MINB = sizeof(Real) == 8      ? 1
                                : Cfg::parts.n == 1    ? (N >= 20 ? 6 : 1)
                                : Cfg::parts.max == 15 || N % 80 == 0 ? 1024 / THREADS
                                                       : 1280 / THREADS;
    __host__ __device__ static constexpr int pad(int x) { return x + x / G; }
};

template <typename Real, int N, int PI, bool LOOP> struct RowParts {
    using Cfg = NatCfg<Real, N, true>;
    using RC = RowCfg<Real, N>;
    using C = typename Cfg::C;
    static constexpr int SIZE = Cfg::parts.size[PI], D = Cfg::dist(PI), B = Cfg::before(PI);
    static constexpr int STAGES = Cfg::parts.first[PI], COUNT = Cfg::parts.count[PI];
    static constexpr int NB = N / SIZE, ITEMS = RC::LINES * NB, PER = (ITEMS + RC::THREADS - 1) / RC::THREADS;
    static constexpr bool FIRST = PI == 0, LAST = PI == Cfg::parts.n - 1;

    __device__ __forceinline__ static void run(const C *in, C *out, C *buf, const C *tw, int tid, int have,
                                               const NatArgs &a) {
        C v[PER][SIZE];
        int k[PER], at[PER], line[PER];
        bool live[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            const int it = tid + i * RC::THREADS;
            line[i] = (int)((unsigned)it / (unsigned)NB);
            const int b = it - line[i] * NB;
            live[i] = line[i] < have;
            k[i] = (int)((unsigned)b % (unsigned)B);
            at[i] = digits_place<N, STAGES>(k[i]) * (N / B) + (int)((unsigned)b / (unsigned)B);
            if (!live[i]) {
                if constexpr (LOOP) zero_all(v[i]);
                continue;
            }
            if constexpr (FIRST) {
                const C *src = in + line[i] * N + at[i];
#pragma unroll
                for (int r = 0; r < SIZE; ++r) v[i][r] = D * (int)sizeof(C) >= 64 ? ld_stream(src + r * D) : ld_cached(src + r * D);
                load_conj(v[i], a);
            } else {
#pragma unroll
                for (int r = 0; r < SIZE; ++r) v[i][r] = buf[line[i] * RC::RS + RC::pad(at[i] + r * D)];
            }
        }
#pragma unroll
        for (int i = 0; i < PER; ++i) {
            if (!live[i]) continue;
            PartStages<Real, N, true, PI>::run(v[i], tw + k[i]);
            if constexpr (!LAST) {
#pragma unroll
                for (int r = 0; r < SIZE; ++r) buf[line[i] * RC::RS + RC::pad(at[i] + r * D)] = v[i][r];
            } else {
                C *dst = out + line[i] * N + k[i];
                finish_store(v[i], a, [&](int r, C x) { dst[digits_out<N, STAGES, COUNT>(r)] = x; });
            }
        }
        if constexpr (!LAST) {
            if constexpr (RC::WARP) __syncwarp();
            else __syncthreads();
            RowParts<Real, N, PI + 1, LOOP>::run(in, out, buf, tw, tid, have, a);
        }
    }
};

// Lines l0 .. l0 + LINES - 1 by the whole CTA.
template <typename Real, int N, bool LOOP = false, typename C = typename Cx<Real>::T>
__device__ __forceinline__ void nat_row_tile(const C *in, C *out, C *buf, const C *tw, int tid, uint32_t l0, const NatArgs &a) {
    using RC = RowCfg<Real, N>;
    using Cfg = NatCfg<Real, N, true>;
    if constexpr (Cfg::parts.n == 1) {
        // one thread per line: a warp copies its 32 lines (contiguous in
        // memory) through its own rows of shared memory, in and out
        const int lane = tid & 31;
        l0 += tid - lane;
        if (l0 >= a.nlines) return;  // (whole warps; no CTA barrier below)
        const int have = (int)(a.nlines - l0 < 32 ? a.nlines - l0 : 32) * N;
        C *rows = buf + (tid - lane) * RC::RS, *row = rows + lane * RC::RS;
        const int64_t base = (int64_t)l0 * N;
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = lane + 32 * i;
            if (e < have) rows[e / N * RC::RS + e % N] = ld_stream(in + base + e);
        }
        __syncwarp();
        C v[N];
#pragma unroll
        for (int r = 0; r < N; ++r) v[r] = row[r];
        load_conj(v, a);
        PartStages<Real, N, true, 0>::run(v, tw);
        finish_store(v, a, [&](int r, C x) { row[digits_out<N, 0, Cfg::parts.count[0]>(r)] = x; });
        __syncwarp();
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const int e = lane + 32 * i;
            if (e < have) out[base + e] = rows[e / N * RC::RS + e % N];
        }
    } else {
        const int64_t base = (int64_t)l0 * N;
        const uint32_t left = a.nlines - l0;
        RowParts<Real, N, 0, LOOP>::run(in + base, out + base, buf, tw, tid, left < RC::LINES ? (int)left : RC::LINES, a);
    }
}

template <typename Real, int N>
__global__ void __launch_bounds__(RowCfg<Real, N>::THREADS, RowCfg<Real, N>::MINB) fft_nat_row_kernel(const NatArgs a) {
    using C = typename Cx<Real>::T;
    extern __shared__ __align__(16) unsigned char nat_smem[];
    follow_previous_launch();
    nat_row_tile<Real, N>(reinterpret_cast<const C *>(a.in), reinterpret_cast<C *>(a.out), reinterpret_cast<C *>(nat_smem),
                          reinterpret_cast<const C *>(a.tw), threadIdx.x, blockIdx.x * RowCfg<Real, N>::LINES, a);
}

}  // namespace mdfft
