// serve.cu -- batched serving of M-D FFT requests of different shapes.
//
// Continuous batching at pass granularity.  Every step launches the next axis
// (in the order of the plan's passes) of every request in flight, whatever its
// shape; a request that arrives while others are on the GPU joins at the next
// step, as soon as the HBM budget and a slot allow, and leaves after its last
// axis.  One step is one launch of a CUDA graph: the copy of the step's work
// table from pinned host memory, then one kernel per line length and kind
// (rows or columns, fft_nat.cuh) that has work, as parallel branches, so that
// the tail of one overlaps the others.  The graphs of the table slots are made
// with the server; a step enables the kernels it needs and sets their grids.
//
// A kernel per length, and not one persistent kernel with all lengths in a
// switch: that one ran every length at the registers and the shared memory of
// the longest (64 registers, 4 CTAs per SM), staged the twiddles per tile and
// closed every tile with four CTA barriers; the 100-request mix moved its data
// at half the copy rate.  There is no device-side waiting: the axes of one
// request are in consecutive steps, ordered by the stream.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <deque>
#include <map>
#include <new>
#include <unordered_map>
#include <vector>

#include "fft_nat.cuh"
#include "plan_internal.h"

using mdfft::NatArgs;
using mdfft::PassArgs;
using mdfft::detail::cuda_fail;
using mdfft::detail::fail;

namespace mdfft {
namespace serve {

constexpr int kMaxItems = 512;  // axes per step (one per request)
constexpr int kSlots = 8;       // tables (and graphs) in flight

// line lengths with a kernel in the step's graph (complex64); other lengths
// run as launches of their own within the same step
#define MDFFT_SERVE_LENGTHS(X) X(0, 16) X(1, 24) X(2, 32) X(3, 48) X(4, 64) X(5, 96) X(6, 128) X(7, 160) X(8, 192) X(9, 256)
#define MDFFT_COUNT_KIND(i, N) +1
constexpr int kKinds = 0 MDFFT_SERVE_LENGTHS(MDFFT_COUNT_KIND);
#undef MDFFT_COUNT_KIND
static_assert(kKinds == 10, "serving kinds are numbered 0 .. kKinds - 1 in MDFFT_SERVE_LENGTHS");
constexpr int kGroups = 2 * kKinds;  // group 2 kind: columns, 2 kind + 1: rows

struct Item {
    NatArgs args;
    int64_t start;  // first tile of this item in its group's numbering
};

struct Group {
    int first, n;   // items[first, first + n)
    int chunk;      // consecutive tiles dealt to a CTA at a time
    int64_t total;  // tiles
};

struct Table {
    Group group[kGroups];
    Item items[kMaxItems];
};

int kind_of(int64_t n) {
    switch (n) {
#define MDFFT_KIND(i, N) \
    case N:              \
        return i;
        MDFFT_SERVE_LENGTHS(MDFFT_KIND)
#undef MDFFT_KIND
        default:
            return -1;
    }
}

// index of a length in MDFFT_SERVE_LENGTHS
template <int N> constexpr int kKindOf = [] {
    int k = -1;
#define MDFFT_KIND(i, n) k = N == n ? i : k;
    MDFFT_SERVE_LENGTHS(MDFFT_KIND)
#undef MDFFT_KIND
    return k;
}();

template <int N, bool ROWS> constexpr int axis_threads() { return ROWS ? RowCfg<float, N>::THREADS : ColCfg<float, N>::THREADS; }
// 40 warps per SM (48 registers; 72 with a whole line in registers)
template <int N, bool ROWS> constexpr int axis_min_ctas() {
    return (NatCfg<float, N, ROWS>::parts.n == 1 ? 896 : 1280) / axis_threads<N, ROWS>();
}

// A group's tiles: chunks of consecutive tiles dealt to the CTAs in turn.
// Consecutive tiles mostly belong to one item, so item lookups and argument
// copies are rare (items are in increasing tile order: lookups only advance).
// The twiddles of a length are the same in every plan: columns stage them once
// per CTA.
template <int N, bool ROWS>
__global__ void __launch_bounds__(axis_threads<N, ROWS>(), axis_min_ctas<N, ROWS>()) serve_axis_kernel(const Table *tab) {
    using CC = ColCfg<float, N>;
    using RC = RowCfg<float, N>;
    using Cfg = NatCfg<float, N, ROWS>;
    constexpr int LINES = ROWS ? RC::LINES : CC::COLS, THREADS = ROWS ? RC::THREADS : CC::THREADS;
    extern __shared__ __align__(16) unsigned char serve_smem[];
    __shared__ NatArgs a;
    float2 *buf = reinterpret_cast<float2 *>(serve_smem);
    const Group &g = tab->group[2 * kKindOf<N> + (ROWS ? 1 : 0)];
    const Item *items = tab->items + g.first;
    const int n = g.n, chunk = g.chunk, tid = threadIdx.x;
    const int64_t total = g.total;
    const float2 *tw = reinterpret_cast<const float2 *>(items[0].args.tw);
    if constexpr (!ROWS && Cfg::parts.n > 1) {
        float2 *stw = buf + N * CC::COLS;
        for (int q = tid; q < tw_entries(Cfg::plan); q += THREADS) stw[q] = __ldg(tw + q);
        tw = stw;
    }
    int cur = -1;
    int64_t cur_start = 0, cur_end = 0;
    for (int64_t c0 = (int64_t)blockIdx.x * chunk; c0 < total; c0 += (int64_t)gridDim.x * chunk)
        for (int64_t t = c0; t < c0 + chunk && t < total; ++t) {
            __syncthreads();  // shared memory of the previous tile is free
            if (t >= cur_end) {
                int lo = cur + 1, hi = n - 1;  // the last item after cur starting at or before t
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (items[mid].start <= t) lo = mid;
                    else hi = mid - 1;
                }
                cur = lo;
                cur_start = items[cur].start;
                cur_end = cur + 1 < n ? items[cur + 1].start : total;
                const int *src = reinterpret_cast<const int *>(&items[cur].args);
                int *dst = reinterpret_cast<int *>(&a);
                if (tid < (int)(sizeof(NatArgs) / sizeof(int))) dst[tid] = src[tid];
                __syncthreads();
            }
            const uint32_t l0 = (uint32_t)(t - cur_start) * LINES;
            // (opaque: a tile's addresses are worked out per tile; hoisted out
            // of the loop they cost twice the registers)
            int tt = tid;
            asm volatile("" : "+r"(tt));
            const float2 *in = reinterpret_cast<const float2 *>(a.in);
            float2 *out = reinterpret_cast<float2 *>(a.out);
            if constexpr (ROWS) {
                nat_row_tile<float, N, true>(in, out, buf, tw, tt, l0, a);
            } else {
                nat_col_tile<float, N, true>(in, out, buf, tw, tt, l0, a);
            }
        }
}
static_assert(sizeof(NatArgs) / sizeof(int) <= 64, "one word per thread");

struct AxisKernel {
    const void *fn;
    int threads, lines;
    size_t smem;
};
AxisKernel axis_kernel(int group) {
    switch (group) {
#define MDFFT_CASE(i, N)                                                                                            \
    case 2 * i:                                                                                                     \
        return {(const void *)&serve_axis_kernel<N, false>, ColCfg<float, N>::THREADS, ColCfg<float, N>::COLS,      \
                ColCfg<float, N>::SMEM};                                                                            \
    case 2 * i + 1:                                                                                                 \
        return {(const void *)&serve_axis_kernel<N, true>, RowCfg<float, N>::THREADS, RowCfg<float, N>::LINES,      \
                RowCfg<float, N>::SMEM};
        MDFFT_SERVE_LENGTHS(MDFFT_CASE)
#undef MDFFT_CASE
        default:
            return {nullptr, 0, 0, 0};
    }
}

// first-fit allocator over one device arena (offsets 256-byte aligned)
class Arena {
  public:
    void reset(size_t bytes) {
        free_.clear();
        if (bytes) free_[0] = bytes;
    }
    bool alloc(size_t bytes, size_t *off) {
        bytes = (bytes + 255) / 256 * 256;
        for (auto it = free_.begin(); it != free_.end(); ++it) {
            if (it->second >= bytes) {
                *off = it->first;
                const size_t rest = it->second - bytes, at = it->first + bytes;
                free_.erase(it);
                if (rest) free_[at] = rest;
                return true;
            }
        }
        return false;
    }
    void release(size_t off, size_t bytes) {
        bytes = (bytes + 255) / 256 * 256;
        auto it = free_.emplace(off, bytes).first;
        auto nx = std::next(it);
        if (nx != free_.end() && it->first + it->second == nx->first) {
            it->second += nx->second;
            free_.erase(nx);
        }
        if (it != free_.begin()) {
            auto pv = std::prev(it);
            if (pv->first + pv->second == it->first) {
                pv->second += it->second;
                free_.erase(it);
            }
        }
    }

  private:
    std::map<size_t, size_t> free_;
};

struct Request {
    int64_t id = 0;
    mdfft_plan_t plan = nullptr;
    const void *in = nullptr;
    void *out = nullptr;
    int dir = -1, normalize = 0;
    size_t bytes = 0;     // budget charge: input + output + workspace
    size_t ws_off = 0;
    bool has_ws = false;
    int next_pass = 0;
    bool admitted = false, finished = false;
    double done_ms = -1.0;  // completion on the server clock
    int slot = -1;          // slot of the step that ran the last pass
    int last_slot = -1;     // slot of the latest step that ran one of its passes
    bool cancelled = false;
};

struct Slot {
    Table *host = nullptr;  // pinned
    Table *dev = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    cudaGraphNode_t copy = nullptr;  // the table copy node (its size follows the step's item count)
    cudaGraphNode_t axis[kGroups] = {nullptr};  // kernel nodes, one per group
    bool enabled[kGroups] = {false};            // groups the executable graph runs
    cudaEvent_t done = nullptr;
    bool busy = false;
    bool direct = false;  // the step ran plain pass launches (low load)
    std::vector<Request *> finishing;
};

}  // namespace serve
}  // namespace mdfft

using namespace mdfft::serve;

struct mdfft_server_s {
    size_t budget = 0, in_use = 0;
    int max_inflight = 0;
    int64_t P = 64;
    cudaStream_t stream = nullptr;
    int grid = 0;        // CTAs of a group's kernel at most (0: one resident wave of each)
    int wave[kGroups] = {0};
    void *arena_mem = nullptr;
    size_t arena_bytes = 0;
    Arena arena;
    std::map<std::vector<int64_t>, mdfft_plan_t> plans;
    std::deque<Request *> queue;
    std::vector<Request *> inflight;
    std::unordered_map<int64_t, Request *> requests;
    int64_t next_id = 1;
    int depth = 2;  // steps in flight on the GPU at most; arrivals in between join the next step
    int chunk = 4;  // at most this many consecutive tiles dealt to a CTA at a time
    int direct = 4;  // low load: at most this many requests with passes left run them as plain launches
    Slot slots[kSlots];
    int next_slot = 0;
    cudaEvent_t t0 = nullptr;
    mdfft_server_stats stats{};
};

namespace {

// The graph of a slot: the table copy, then all groups' kernels (disabled until
// a step needs them) as parallel branches.
mdfft_status make_graph(Slot &sl) {
    cudaError_t e = cudaGraphCreate(&sl.graph, 0);
    if (e == cudaSuccess)
        e = cudaGraphAddMemcpyNode1D(&sl.copy, sl.graph, nullptr, 0, sl.dev, sl.host, sizeof(Table), cudaMemcpyHostToDevice);
    for (int g = 0; g < kGroups && e == cudaSuccess; ++g) {
        const AxisKernel k = axis_kernel(g);
        void *args[] = {&sl.dev};
        cudaKernelNodeParams np{};
        np.func = const_cast<void *>(k.fn);
        np.gridDim = dim3(1), np.blockDim = dim3((unsigned)k.threads);
        np.sharedMemBytes = (unsigned)k.smem;
        np.kernelParams = args;
        e = cudaGraphAddKernelNode(&sl.axis[g], sl.graph, &sl.copy, 1, &np);
    }
    if (e == cudaSuccess) e = cudaGraphInstantiate(&sl.exec, sl.graph, 0);
    for (int g = 0; g < kGroups && e == cudaSuccess; ++g) {
        e = cudaGraphNodeSetEnabled(sl.exec, sl.axis[g], 0);
        sl.enabled[g] = false;
    }
    return e == cudaSuccess ? MDFFT_OK : cuda_fail(e, "step graph");
}

// Number of launches a request needs: the axes of its plan (the pass kernels
// where a plan has none, e.g. all dims 1).
int request_ops(const Request *r) { return r->plan->nat.empty() ? r->plan->M : (int)r->plan->nat.size(); }

// Requests of a slot whose step has completed: record completion, free memory.
void resolve_slot(mdfft_server_t s, Slot &sl) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, s->t0, sl.done);
    for (Request *r : sl.finishing) {
        r->finished = true;
        r->done_ms = r->cancelled ? -1.0 : ms;
        if (r->has_ws) s->arena.release(r->ws_off, (size_t)r->plan->T * r->plan->elem);
        r->has_ws = false;
        s->in_use -= r->bytes;
        (r->cancelled ? s->stats.cancelled : s->stats.completed)++;
        s->inflight.erase(std::find(s->inflight.begin(), s->inflight.end(), r));
    }
    sl.finishing.clear();
    sl.busy = false;
}

void poll_slots(mdfft_server_t s) {
    for (Slot &sl : s->slots)
        if (sl.busy && cudaEventQuery(sl.done) == cudaSuccess) resolve_slot(s, sl);
}

mdfft_status get_plan(mdfft_server_t s, int M, const int64_t *N, mdfft_plan_t *out) {
    std::vector<int64_t> key(N, N + M);
    auto it = s->plans.find(key);
    if (it != s->plans.end()) {
        *out = it->second;
        return MDFFT_OK;
    }
    int64_t T = 1;
    for (int i = 0; i < M; ++i) T *= N[i];
    mdfft_plan_t p = nullptr;
    mdfft_status st = mdfft::detail::plan_create(&p, M, N, std::min<int64_t>(s->P, T), nullptr, MDFFT_C64, 0, false, 1);
    if (st != MDFFT_OK) return st;
    s->plans[key] = p;
    *out = p;
    return MDFFT_OK;
}

// Pass s of request r as launch arguments (buffers as in mdfft_exec: the
// last pass writes out, earlier ones alternate with the request's workspace).
PassArgs pass_args(mdfft_server_t s, const Request *r, int pass) {
    const mdfft_plan_s *p = r->plan;
    const int M = p->M;
    void *ws = (char *)s->arena_mem + r->ws_off;
    const void *src = r->in;
    void *dst = nullptr;
    for (int q = 0; q <= pass; ++q) {
        // destination of pass q going backwards from out
        dst = ((M - 1 - q) % 2 == 0) ? r->out : ws;
        if (q < pass) src = dst;
    }
    PassArgs a = p->pass[pass].args;
    a.in = src;
    a.out = dst;
    a.tw = (const char *)p->tw + p->pass[pass].tw_offset;
    a.conj = r->dir == 1 ? (pass == 0 ? 1 : 0) | (pass == M - 1 ? 2 : 0) : 0;
    a.scale = (pass == M - 1 && r->normalize) ? 1.0 / (double)p->T : 1.0;
    a.scaled = a.scale != 1.0;
    return a;
}

// Axis `op` of request r as launch arguments: in place on out after the first.
NatArgs axis_args(const Request *r, int op) {
    const mdfft_plan_s *p = r->plan;
    const mdfft::detail::NatOp &o = p->nat[op];
    const bool last = op + 1 == (int)p->nat.size();
    NatArgs a = o.args;
    a.in = op == 0 ? r->in : r->out;
    a.out = r->out;
    a.tw = (const char *)p->tw + p->pass[o.s].tw_offset;
    a.conj = r->dir == 1 ? (op == 0 ? 1 : 0) | (last ? 2 : 0) : 0;
    a.scale = (last && r->normalize) ? 1.0 / (double)p->T : 1.0;
    a.scaled = a.scale != 1.0;
    return a;
}

// Launch `op` of request r on its own.
cudaError_t launch_alone(mdfft_server_t s, const Request *r, int op) {
    if (r->plan->nat.empty()) {
        const mdfft::detail::Pass &ps = r->plan->pass[op];
        PassArgs a = pass_args(s, r, op);
        a.ntiles = ps.ctas;
        void *args[] = {&a};
        return cudaLaunchKernel(ps.k.fn, dim3((unsigned)ps.grid), dim3(ps.k.threads), args, ps.k.smem, s->stream);
    }
    const mdfft::PassKernel &k = r->plan->nat[op].k;
    NatArgs a = axis_args(r, op);
    void *args[] = {&a};
    return mdfft::detail::launch_following(k, (a.nlines + (unsigned)k.lines - 1) / (unsigned)k.lines, args, s->stream);
}

}  // namespace

extern "C" {

mdfft_status mdfft_server_create(mdfft_server_t *out, size_t budget_bytes, int max_inflight, int64_t P,
                                 mdfft_stream_t stream) {
    if (!out) return fail(MDFFT_E_ARG, "null argument");
    *out = nullptr;
    if (budget_bytes < 4096 || max_inflight < 1 || max_inflight > kMaxItems || P < 1)
        return fail(MDFFT_E_ARG, "budget >= 4096 bytes, 1 <= max_inflight <= 512, P >= 1");
    mdfft_server_s *s = new (std::nothrow) mdfft_server_s;
    if (!s) return fail(MDFFT_E_NOMEM, "host allocation");
    s->budget = budget_bytes;
    s->max_inflight = max_inflight;
    s->P = P;
    s->stream = reinterpret_cast<cudaStream_t>(stream);
    s->stats.budget_bytes = budget_bytes;
    auto bail = [&](mdfft_status st) {
        mdfft_server_destroy(s);
        return st;
    };
    cudaError_t e;
    // workspaces: one T-element array per request in flight; each request is
    // charged input + output + workspace, so workspaces use at most a third.
    // Axis launches leave it untouched (they work in place on the output); the
    // pass kernels of a plan without them need it.
    s->arena_bytes = (budget_bytes / 3 + 255) / 256 * 256;
    if ((e = cudaMalloc(&s->arena_mem, s->arena_bytes)) != cudaSuccess) return bail(cuda_fail(e, "cudaMalloc arena"));
    s->arena.reset(s->arena_bytes);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    for (int g = 0; g < kGroups; ++g) {
        const AxisKernel k = axis_kernel(g);
        int per_sm = 0;
        if ((e = cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k.fn, k.threads, k.smem)) != cudaSuccess)
            return bail(cuda_fail(e, "serving kernel"));
        s->wave[g] = std::max(1, sms * std::max(1, per_sm));
    }
    for (Slot &sl : s->slots) {
        if ((e = cudaHostAlloc((void **)&sl.host, sizeof(Table), cudaHostAllocDefault)) != cudaSuccess)
            return bail(cuda_fail(e, "cudaHostAlloc table"));
        std::memset(sl.host, 0, sizeof(Table));
        if ((e = cudaMalloc((void **)&sl.dev, sizeof(Table))) != cudaSuccess)
            return bail(cuda_fail(e, "cudaMalloc table"));
        if ((e = cudaEventCreate(&sl.done)) != cudaSuccess) return bail(cuda_fail(e, "cudaEventCreate"));
        if (mdfft_status st = make_graph(sl)) return bail(st);
    }
    s->stats.grid_ctas = *std::max_element(s->wave, s->wave + kGroups);
    if ((e = cudaEventCreate(&s->t0)) != cudaSuccess) return bail(cuda_fail(e, "cudaEventCreate"));
    cudaEventRecord(s->t0, s->stream);
    if ((e = cudaStreamSynchronize(s->stream)) != cudaSuccess) return bail(cuda_fail(e, "cudaStreamSynchronize"));
    *out = s;
    return MDFFT_OK;
}

mdfft_status mdfft_server_submit(mdfft_server_t s, int M, const int64_t N[], const void *in_dev, void *out_dev,
                                 int dir, int normalize, int64_t *request_id) {
    if (!s || !N || !in_dev || !out_dev || !request_id) return fail(MDFFT_E_ARG, "null argument");
    if (dir != -1 && dir != 1) return fail(MDFFT_E_ARG, "dir must be -1 or +1");
    if (normalize != 0 && !(normalize == 1 && dir == 1)) return fail(MDFFT_E_ARG, "normalize only on the inverse");
    if ((uintptr_t)in_dev % 8 || (uintptr_t)out_dev % 8) return fail(MDFFT_E_ARG, "misaligned data pointer");
    mdfft_plan_t p = nullptr;
    mdfft_status st = get_plan(s, M, N, &p);
    if (st != MDFFT_OK) return st;
    const size_t bytes = (size_t)p->T * p->elem;
    const uintptr_t a = (uintptr_t)in_dev, b = (uintptr_t)out_dev;
    if (a < b + bytes && b < a + bytes) return fail(MDFFT_E_ARG, "in and out overlap");
    if (3 * bytes > s->budget) return fail(MDFFT_E_RANGE, "request larger than the whole HBM budget");
    Request *r = new (std::nothrow) Request;
    if (!r) return fail(MDFFT_E_NOMEM, "host allocation");
    r->id = s->next_id++;
    r->plan = p;
    r->in = in_dev;
    r->out = out_dev;
    r->dir = dir;
    r->normalize = normalize;
    r->bytes = 3 * bytes;
    s->requests[r->id] = r;
    s->queue.push_back(r);
    s->stats.submitted++;
    *request_id = r->id;
    return MDFFT_OK;
}

mdfft_status mdfft_server_step(mdfft_server_t s, int *launched) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    if (launched) *launched = 0;
    poll_slots(s);
    // admission: first come first served, within the budget, the slots and the arena
    while (!s->queue.empty() && (int)s->inflight.size() < s->max_inflight) {
        Request *r = s->queue.front();
        if (s->in_use + r->bytes > s->budget) break;
        size_t off = 0;
        if (!s->arena.alloc((size_t)r->plan->T * r->plan->elem, &off)) break;
        r->ws_off = off;
        r->has_ws = true;
        r->admitted = true;
        s->in_use += r->bytes;
        s->inflight.push_back(r);
        s->queue.pop_front();
        s->stats.admitted++;
    }
    std::vector<Request *> todo;
    for (Request *r : s->inflight)
        if (r->next_pass < request_ops(r)) todo.push_back(r);
    if (todo.empty()) return MDFFT_OK;
    // low load: nothing queued and few requests with passes left -- they run
    // at once; the depth limit, which lets arrivals gather into fuller
    // steps, holds them back only while batched steps are in flight
    const bool direct = (int)todo.size() <= s->direct && s->queue.empty();
    int busy = 0, busy_batched = 0;
    for (const Slot &b : s->slots) busy += b.busy, busy_batched += b.busy && !b.direct;
    if (busy >= s->depth && (!direct || busy_batched > 0)) return MDFFT_OK;  // let more work gather
    Slot &sl = s->slots[s->next_slot];
    if (sl.busy) {  // its table may still be in use: wait for that step
        cudaError_t e = cudaEventSynchronize(sl.done);
        if (e != cudaSuccess) return cuda_fail(e, "cudaEventSynchronize");
        resolve_slot(s, sl);
    }
    cudaError_t e = cudaSuccess;
    if (direct) {
        // low load: every remaining axis of these requests, oldest first, as
        // plain launches (stream order keeps each request's axes in order)
        for (Request *r : todo) {
            for (int op = r->next_pass; op < request_ops(r); ++op) {
                e = launch_alone(s, r, op);
                if (e != cudaSuccess) return cuda_fail(e, "axis launch");
                s->stats.kernel_launches++;
            }
            r->next_pass = request_ops(r);
            r->last_slot = r->slot = s->next_slot;
            sl.finishing.push_back(r);
            s->stats.direct_requests++;
        }
        e = cudaEventRecord(sl.done, s->stream);
        if (e != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
        sl.busy = true;
        sl.direct = true;
        s->next_slot = (s->next_slot + 1) % kSlots;
        s->stats.steps++;
        if (launched) *launched = 1;
        return MDFFT_OK;
    }
    Table *tab = sl.host;
    std::vector<std::pair<Request *, int>> separate;  // lengths without a kernel in the graph
    std::vector<Item> items[kGroups];
    int64_t total[kGroups] = {0};
    int used = 0;
    for (Request *r : todo) {
        if (used >= kMaxItems) break;
        const int op = r->next_pass;
        const int kind = r->plan->nat.empty() ? -1 : kind_of(r->plan->pass[r->plan->nat[op].s].n);
        if (kind < 0) {
            separate.push_back({r, op});
        } else {
            const mdfft::PassKernel &k = r->plan->nat[op].k;
            const int g = 2 * kind + (r->plan->nat[op].args.stride == 1 ? 1 : 0);
            items[g].push_back(Item{axis_args(r, op), total[g]});
            total[g] += (items[g].back().args.nlines + (unsigned)k.lines - 1) / (unsigned)k.lines;
            ++used;
        }
        r->next_pass++;
        r->last_slot = s->next_slot;
        if (r->next_pass == request_ops(r)) {
            r->slot = s->next_slot;
            sl.finishing.push_back(r);
        }
    }
    if (used > 0) {
        int at = 0;
        for (int g = 0; g < kGroups; ++g) {
            Group &gr = tab->group[g];
            const int64_t ctas = s->grid > 0 ? s->grid : s->wave[g];
            gr.first = at, gr.n = (int)items[g].size(), gr.total = total[g];
            // the group's tiles spread over every CTA first: chunks of total / CTAs tiles, at most s->chunk
            gr.chunk = (int)std::max<int64_t>(1, std::min<int64_t>(s->chunk, total[g] / ctas));
            for (const Item &it : items[g]) tab->items[at++] = it;
            const bool on = gr.n > 0;
            if (on) {
                const AxisKernel k = axis_kernel(g);
                void *args[] = {&sl.dev};
                cudaKernelNodeParams np{};
                np.func = const_cast<void *>(k.fn);
                np.gridDim = dim3((unsigned)std::min<int64_t>(ctas, (total[g] + gr.chunk - 1) / gr.chunk));
                np.blockDim = dim3((unsigned)k.threads);
                np.sharedMemBytes = (unsigned)k.smem;
                np.kernelParams = args;
                e = cudaGraphExecKernelNodeSetParams(sl.exec, sl.axis[g], &np);
                if (e != cudaSuccess) return cuda_fail(e, "cudaGraphExecKernelNodeSetParams");
                s->stats.kernel_launches++;
            }
            if (on != sl.enabled[g]) {
                e = cudaGraphNodeSetEnabled(sl.exec, sl.axis[g], on ? 1 : 0);
                if (e != cudaSuccess) return cuda_fail(e, "cudaGraphNodeSetEnabled");
                sl.enabled[g] = on;
            }
        }
        // copy only the header and the items of this step
        e = cudaGraphExecMemcpyNodeSetParams1D(sl.exec, sl.copy, sl.dev, sl.host,
                                               offsetof(Table, items) + (size_t)used * sizeof(Item), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphExecMemcpyNodeSetParams1D");
        e = cudaGraphLaunch(sl.exec, s->stream);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGraphLaunch");
        s->stats.graph_launches++;
    }
    for (auto &pr : separate) {
        e = launch_alone(s, pr.first, pr.second);
        if (e != cudaSuccess) return cuda_fail(e, "axis launch");
        s->stats.kernel_launches++;
    }
    e = cudaEventRecord(sl.done, s->stream);
    if (e != cudaSuccess) return cuda_fail(e, "cudaEventRecord");
    sl.busy = true;
    sl.direct = false;
    s->next_slot = (s->next_slot + 1) % kSlots;
    s->stats.steps++;
    if (launched) *launched = 1;
    return MDFFT_OK;
}

mdfft_status mdfft_server_run(mdfft_server_t s, int max_steps, int *steps) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    int n = 0;
    for (; n < max_steps; ++n) {
        int launched = 0;
        mdfft_status st = mdfft_server_step(s, &launched);
        if (st != MDFFT_OK) return st;
        if (!launched) break;
    }
    if (steps) *steps = n;
    return MDFFT_OK;
}

mdfft_status mdfft_server_poll(mdfft_server_t s, int64_t request_id, int *done, double *done_ms) {
    if (!s || !done) return fail(MDFFT_E_ARG, "null argument");
    auto it = s->requests.find(request_id);
    if (it == s->requests.end()) return fail(MDFFT_E_ARG, "unknown request id");
    Request *r = it->second;
    if (!r->finished && r->slot >= 0) {
        Slot &sl = s->slots[r->slot];
        if (sl.busy && cudaEventQuery(sl.done) == cudaSuccess) resolve_slot(s, sl);
    }
    *done = r->finished ? 1 : 0;
    if (done_ms) *done_ms = r->finished ? r->done_ms : -1.0;
    return MDFFT_OK;
}

mdfft_status mdfft_server_release(mdfft_server_t s, int64_t request_id) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    auto it = s->requests.find(request_id);
    if (it == s->requests.end()) return fail(MDFFT_E_ARG, "unknown request id");
    if (!it->second->finished) return fail(MDFFT_E_ARG, "request not finished");
    delete it->second;
    s->requests.erase(it);
    return MDFFT_OK;
}

mdfft_status mdfft_server_cancel(mdfft_server_t s, int64_t request_id) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    auto it = s->requests.find(request_id);
    if (it == s->requests.end()) return fail(MDFFT_E_ARG, "unknown request id");
    Request *r = it->second;
    if (r->finished || r->cancelled) return fail(MDFFT_E_ARG, "request already finished or cancelled");
    if (!r->admitted) {  // still queued: it never reached the GPU
        s->queue.erase(std::find(s->queue.begin(), s->queue.end(), r));
        r->cancelled = r->finished = true;
        r->done_ms = -1.0;
        s->stats.cancelled++;
        return MDFFT_OK;
    }
    if (r->next_pass == request_ops(r)) return MDFFT_OK;  // its last pass is on the GPU: it completes
    r->cancelled = true;
    r->next_pass = request_ops(r);  // no further passes are scheduled
    Slot *last = r->last_slot >= 0 ? &s->slots[r->last_slot] : nullptr;
    if (last && last->busy) {  // resources come back when its latest step has run
        r->slot = r->last_slot;
        last->finishing.push_back(r);
    } else {  // nothing of it is on the GPU
        r->finished = true;
        r->done_ms = -1.0;
        if (r->has_ws) s->arena.release(r->ws_off, (size_t)r->plan->T * r->plan->elem);
        r->has_ws = false;
        s->in_use -= r->bytes;
        s->stats.cancelled++;
        s->inflight.erase(std::find(s->inflight.begin(), s->inflight.end(), r));
    }
    return MDFFT_OK;
}

mdfft_status mdfft_server_drain(mdfft_server_t s) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    while (!s->queue.empty() || !s->inflight.empty()) {
        int launched = 0;
        mdfft_status st = mdfft_server_step(s, &launched);
        if (st != MDFFT_OK) return st;
        if (!launched) {  // nothing to launch until a step completes: wait for the oldest one only
            for (int k = 0; k < kSlots; ++k) {
                Slot &sl = s->slots[(s->next_slot + k) % kSlots];
                if (!sl.busy) continue;
                cudaError_t e = cudaEventSynchronize(sl.done);
                if (e != cudaSuccess) return cuda_fail(e, "cudaEventSynchronize");
                resolve_slot(s, sl);
                break;
            }
        }
    }
    return MDFFT_OK;
}

mdfft_status mdfft_server_reset_clock(mdfft_server_t s) {
    if (!s) return fail(MDFFT_E_ARG, "null server");
    cudaEventRecord(s->t0, s->stream);
    cudaError_t e = cudaEventSynchronize(s->t0);
    if (e != cudaSuccess) return cuda_fail(e, "cudaEventSynchronize");
    return MDFFT_OK;
}

mdfft_status mdfft_server_set_grid(mdfft_server_t s, int ctas) {
    if (!s || ctas < 1) return fail(MDFFT_E_ARG, "bad argument");
    for (Slot &sl : s->slots)
        if (sl.busy) {
            cudaError_t e = cudaEventSynchronize(sl.done);
            if (e != cudaSuccess) return cuda_fail(e, "cudaEventSynchronize");
            resolve_slot(s, sl);
        }
    s->grid = ctas;
    s->stats.grid_ctas = ctas;
    return MDFFT_OK;
}

mdfft_status mdfft_server_set_line_kernel(mdfft_server_t s, int enable) {
    if (!s || (enable != 0 && enable != 1)) return fail(MDFFT_E_ARG, "enable must be 0 or 1");
    return MDFFT_OK;  // every length has its own kernel
}

mdfft_status mdfft_server_set_chunk(mdfft_server_t s, int chunk) {
    if (!s || chunk < 1 || chunk > 64) return fail(MDFFT_E_ARG, "chunk must be in [1, 64]");
    s->chunk = chunk;
    return MDFFT_OK;
}

mdfft_status mdfft_server_set_direct(mdfft_server_t s, int max_requests) {
    if (!s || max_requests < 0 || max_requests > 64) return fail(MDFFT_E_ARG, "direct threshold must be in [0, 64]");
    s->direct = max_requests;
    return MDFFT_OK;
}

mdfft_status mdfft_server_set_depth(mdfft_server_t s, int depth) {
    if (!s || depth < 1 || depth > kSlots) return fail(MDFFT_E_ARG, "depth must be in [1, 8]");
    s->depth = depth;
    return MDFFT_OK;
}

mdfft_status mdfft_server_get_stats(mdfft_server_t s, mdfft_server_stats *out) {
    if (!s || !out) return fail(MDFFT_E_ARG, "null argument");
    s->stats.inflight = (int64_t)s->inflight.size();
    s->stats.queued = (int64_t)s->queue.size();
    s->stats.bytes_in_use = s->in_use;
    *out = s->stats;
    return MDFFT_OK;
}

mdfft_status mdfft_server_destroy(mdfft_server_t s) {
    if (!s) return MDFFT_OK;
    if (s->stream) cudaStreamSynchronize(s->stream);
    for (Slot &sl : s->slots) {
        if (sl.exec) cudaGraphExecDestroy(sl.exec);
        if (sl.graph) cudaGraphDestroy(sl.graph);
        if (sl.host) cudaFreeHost(sl.host);
        if (sl.dev) cudaFree(sl.dev);
        if (sl.done) cudaEventDestroy(sl.done);
    }
    if (s->t0) cudaEventDestroy(s->t0);
    if (s->arena_mem) cudaFree(s->arena_mem);
    for (auto &kv : s->plans) mdfft_destroy(kv.second);
    for (auto &kv : s->requests) delete kv.second;
    delete s;
    return MDFFT_OK;
}

}  // extern "C"
