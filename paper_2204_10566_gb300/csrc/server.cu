// Request server: continuous batching of many lattices on one GPU.
//
// Requests (flag field, flow parameters, step count, storage precision) are
// queued by lbm_server_submit; host worker threads build each request's
// sparse index while the GPU is busy.  lbm_server_tick admits ready requests
// into resident slots by exact device footprint against the budget, then
// advances every resident lattice by up to steps_per_tick steps with one
// captured CUDA graph, whose one kernel takes all steps of the tick: a
// cooperative launch with a barrier over the grid between steps, whose warps
// walk the inlet/outlet nodes and the fluid tiles of all resident lattices of
// both precisions.  The lattice of a warp's item is found by binary search in
// a per-tick table that the graph copies to the device first.  The table
// changes every tick, the graph never does.  Each cell is updated by the same
// device code as lbm_step, so a lattice's result does not depend on what else
// is resident.  A tick of very many cell updates goes in several launches, and
// a device that refuses the cooperative launch takes the steps in a launch each.
#include <cuda_runtime.h>

#include <algorithm>
#include <condition_variable>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "lbm_device.cuh"

namespace lbm {

// FP16S scale of a descriptor (api.cu): 0 selects the default 4096, any
// other value must be a positive power of two; returns 0 when invalid.
float resolve_fp16_scale(float s);

// A context's step arguments in the tile view (api.cu): every fluid tile and
// every inlet/outlet node, whichever fluid kernel its own steps run.
void ctx_tile_step_args(lbm_ctx *c, StepArgs *out);

constexpr int MAX_SLOTS = LBM_SERVER_MAX_SLOTS;
// Cell updates one launch takes at most, about a quarter of a second at the
// 18.6 G a second of twelve lattices of 2.2 M cells: a tick of more (large
// lattices, many steps) goes in several launches, so that the GPU is not one
// kernel's for long.  LBM_LAUNCH_UPDATES sets another number, for tests.
constexpr int64_t LAUNCH_UPDATES = (int64_t)1 << 32;

struct alignas(16) DomainEntry {
    StepArgs a;        // state at the start of the tick: fin is the current buffer
    int64_t t_base;    // steps done before the tick
    int32_t steps;     // steps this lattice takes in the tick
    int32_t precision; // LBM_FP32 or LBM_FP16S
    int32_t tile_begin, node_begin;  // its first tile item and its first node item (32 nodes) in the tick's list
};

struct alignas(16) TickTable {
    int32_t n_domains, n_tiles, n_nodes, steps;  // steps: the most any lattice takes
    DomainEntry d[MAX_SLOTS];
};

// Words after the health flags (one per domain): the tick's status, then the
// two barrier words.
constexpr int STATUS_WORD = MAX_SLOTS, BARRIER_WORDS = MAX_SLOTS + 8, FLAG_WORDS = MAX_SLOTS + 16;

// Lattice of an item: the last entry whose first item is <= item.
template <bool NODES>
__device__ __forceinline__ int find_domain(const DomainEntry *d, int n, int item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if ((NODES ? d[mid].node_begin : d[mid].tile_begin) <= item)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// Health check of an item on its lattice's last step of the tick (STEP_REDUCE:
// record_cell sets hv[5] for a non-finite density or velocity): one atomic
// per warp that saw one.
__device__ __forceinline__ void flag_non_finite(const StepArgs &a, double bad) {
    if (!(a.flags & STEP_REDUCE)) return;  // uniform over the warp
    if (__any_sync(0xffffffffu, bad != 0.0) && (threadIdx.x & 31) == 0) atomicOr(a.status, 1u);
}

// The arguments come by value: what an item uses of them is read from shared
// memory once, not again after every store that might have changed it.
template <int P, int AX>
__device__ __forceinline__ void serve_nodes(const StepArgs a, int i, int lane) {
    double hv[6] = {0, 0, 0, 0, 0, 0};
    const int k = 32 * i + lane;
    if (k < a.nbnodes) boundary_node<P, RATE_ONE, false, AX, true>(a, k, hv);
    flag_non_finite(a, hv[5]);
}

template <int P, int AX>
__device__ __forceinline__ void serve_tile(const StepArgs a, const TileRec &rec, int lane) {
    double hv[6] = {0, 0, 0, 0, 0, 0};
    tile_update<P, AX, true, false, true>(a, rec, lane, nullptr, hv);
    flag_non_finite(a, hv[5]);
}

// Calls fn<P, AX> for the lattice of an entry.
#define SERVE_DISPATCH(e, fn, ...)                                                         \
    do {                                                                                   \
        if ((e).precision == LBM_FP32) {                                                   \
            if ((e).a.row_axis == 2) fn<1, 2>((e).a, __VA_ARGS__);                         \
            else fn<1, 0>((e).a, __VA_ARGS__);                                             \
        } else {                                                                           \
            if ((e).a.row_axis == 2) fn<2, 2>((e).a, __VA_ARGS__);                         \
            else fn<2, 0>((e).a, __VA_ARGS__);                                             \
        }                                                                                  \
    } while (0)

// Steps k0 .. k0 + count - 1 of a tick, as far as its lattices go: several in a
// cooperative launch, or one (no barrier then) in an ordinary launch.
// Before, a step was four launches in turn (fluid and
// nodes of each precision) whose blocks copied a lattice's arguments to
// shared memory for every 128 cells; here the table stays in shared memory,
// and a warp looks up the lattice and the record of its next tile while it
// updates one.  What then bounds it is the instruction cache: FP32 and FP16S
// lattices in admission order and the fast tiles' own path took 166 us a step
// for twelve lattices of 2.2 M cells (no_instruction half of the stalls),
// each precision in one go and the line sink alone 118 us, the four launches
// 136 us; one lattice of 67 000 cells 17 -> 10 us.  5 blocks per SM: 4 take 2 %
// and 6 take 8 % longer on the burst of the measured mix.
#ifndef LBM_SERVE_BLOCKS
#define LBM_SERVE_BLOCKS 5
#endif
__global__ void __launch_bounds__(STEP_THREADS, LBM_SERVE_BLOCKS) k_serve(const TickTable *tab, int k0, int count,
                                                                        int32_t *barrier, uint32_t *status, int polls) {
    extern __shared__ __align__(16) char serve_smem[];
    DomainEntry *dom = reinterpret_cast<DomainEntry *>(serve_smem);
    const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    const int n = tab->n_domains, tiles = tab->n_tiles, nodes = tab->n_nodes, end = min(k0 + count, tab->steps);
    for (int w = threadIdx.x; w < n * (int)(sizeof(DomainEntry) / 16); w += STEP_THREADS)
        reinterpret_cast<int4 *>(dom)[w] = reinterpret_cast<const int4 *>(tab->d)[w];
    const int first = warp * (int)gridDim.x + (int)blockIdx.x, stride = (int)gridDim.x * (STEP_THREADS / 32);
    for (int k = k0; k < end; ++k) {
        __syncthreads();
        if ((int)threadIdx.x < n) {  // the step's buffers, number and check flag
            DomainEntry &e = dom[threadIdx.x];
            if (k > k0 || (k0 & 1)) {
                const void *t = e.a.fin;
                e.a.fin = e.a.fout;
                e.a.fout = const_cast<void *>(t);
            }
            e.a.t_new = e.t_base + k + 1;
            e.a.flags = k == e.steps - 1 ? STEP_REDUCE : 0;
        }
        __syncthreads();
        int i = first;
        for (; i < nodes; i += stride) {
            const DomainEntry &e = dom[find_domain<true>(dom, n, i)];
            if (k < e.steps) SERVE_DISPATCH(e, serve_nodes, i - e.node_begin, lane);  // uniform over the warp
        }
        i -= nodes;
        // the next tile's lattice and record are looked up while a tile is updated
        int d_next = 0;
        TileRec next;
        if (i < tiles) {
            d_next = find_domain<false>(dom, n, i);
            next = TileRec(dom[d_next].a.tiles, i - dom[d_next].tile_begin);
        }
        for (; i < tiles; i += stride) {
            const DomainEntry &e = dom[d_next];
            const TileRec rec = next;
            if (i + stride < tiles) {
                d_next = find_domain<false>(dom, n, i + stride);
                next = TileRec(dom[d_next].a.tiles, i + stride - dom[d_next].tile_begin);
            }
            if (k < e.steps) SERVE_DISPATCH(e, serve_tile, rec, lane);
        }
        if (k + 1 < end && !grid_barrier(barrier, k - k0 + 1, status, polls)) break;
    }
    // the last block to leave clears the words for the next tick
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(barrier + 1, 1) == (int)gridDim.x - 1) {
        barrier[0] = 0;
        barrier[1] = 0;
    }
}

}  // namespace lbm

using namespace lbm;

namespace {

struct Request {
    int64_t id = 0;
    lbm_request req{};
    std::vector<uint8_t> flags;
    int state = LBM_REQ_QUEUED;
    lbm_status fail_status = LBM_OK;  // why a FAILED request failed
    int64_t steps_done = 0;
    bool cancel = false;
    // built by a worker thread (guarded by the server mutex)
    bool index_ready = false;
    std::string index_error;
    HostIndex idx;
    int64_t footprint = 0;
    int64_t n_active = -1;
    // resident state
    lbm_ctx *ctx = nullptr;
    // result
    std::vector<double> rho, u;
};

int storage_size(int precision) { return precision == LBM_FP32 ? 4 : 2; }

}  // namespace

struct lbm_server {
    lbm_server_desc desc{};
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    std::string err;
    std::map<int64_t, std::unique_ptr<Request>> reqs;
    std::deque<int64_t> queue;      // submitted, not yet admitted (submission order)
    std::vector<int64_t> resident;  // admitted, running
    int64_t next_id = 1;
    int64_t in_use = 0, peak = 0;
    double cell_updates = 0, ticks = 0, graph_launches = 0, graph_captures = 0, finished = 0;
    // worker threads building indexes
    std::vector<std::thread> workers;
    std::mutex mu;
    std::condition_variable cv;
    std::deque<Request *> build_queue;
    bool stop = false;
    // device tables and the tick graph
    TickTable *h_tab = nullptr, *d_tab = nullptr;
    // health flags, one word per domain: cleared at the start of every tick,
    // raised by the check step, copied back at its end; then the tick's status
    // and the kernel's barrier words
    uint32_t *d_flags = nullptr, *h_flags = nullptr;
    cudaGraphExec_t exec = nullptr;
    int grid = 0, resident_blocks = 0, smem = 0, polls = 0;  // of the tick's kernel
    int64_t launch_updates = LAUNCH_UPDATES;
    bool together = false;              // several steps in a cooperative launch; else a launch each
};

namespace {

lbm_status sfail(lbm_server *s, lbm_status st, const std::string &m) {
    if (s) s->err = m;
    return st;
}

// Device bytes a request holds while resident: the context's buffers (the
// readback of its moments is staged in one of them).
int64_t request_footprint(const lbm_request &q, const HostIndex &idx) {
    lbm_desc d{};
    d.nx = q.nx;
    d.ny = q.ny;
    d.nz = q.nz;
    d.periodic = q.periodic;
    d.precision = q.precision;
    return ctx_footprint(d, idx);
}

// The checks of lbm_server_submit that need no index (host only).  *active
// receives the request's active cell count.
lbm_status check_request(const lbm_request *q, int64_t budget_bytes, int64_t *active, const char **why) {
    *active = 0;
    auto bad = [why](lbm_status st, const char *m) {
        *why = m;
        return st;
    };
    if (!q || !q->flags) return bad(LBM_ERR_ARG, "NULL request or flags");
    if (q->precision != LBM_FP32 && q->precision != LBM_FP16S)
        return bad(LBM_ERR_ARG, "the server runs FP32 and FP16S lattices");
    if (q->steps < 1 || q->nx < 1 || q->ny < 1 || q->nz < 1 || (q->periodic & ~7))
        return bad(LBM_ERR_ARG, "bad lattice size, periodicity or step count");
    const lbm_params &p = q->params;
    if (p.omega3 != 1.0 || p.omega4 != 1.0 || p.omega5 != 1.0 || p.omega6 != 1.0)
        return bad(LBM_ERR_ARG, "the server runs the default ghost rates only");
    if (resolve_fp16_scale(q->fp16_scale) == 0.0f)
        return bad(LBM_ERR_ARG, "the FP16 scale must be 0 (default) or a power of two");
    if (lbm_params_check(&p, nullptr, nullptr, why) != LBM_OK) return LBM_ERR_ARG;  // lbm_set_params' checks
    const int64_t ncell = (int64_t)q->nx * q->ny * q->nz;
    int64_t n = 0;
    for (int64_t b = 0; b < ncell; ++b) n += q->flags[b] != LBM_SOLID;
    *active = n;
    // every active cell has a slot: a lattice this large can never get 32-bit offsets
    if (n > MAX_SLOTS_32)
        return bad(LBM_ERR_ARG, "the lattice has more active cells than the server's 32-bit population "
                                "offsets address (2^32 / 27 slots); run it with lbm_step");
    if (2 * 27 * n * storage_size(q->precision) > budget_bytes)
        return bad(LBM_ERR_OOM, "the lattice can never fit the server's memory budget");
    *why = "";
    return LBM_OK;
}

void worker_loop(lbm_server *s) {
    for (;;) {
        Request *r = nullptr;
        {
            std::unique_lock<std::mutex> lk(s->mu);
            s->cv.wait(lk, [&] { return s->stop || !s->build_queue.empty(); });
            if (s->stop) return;
            r = s->build_queue.front();
            s->build_queue.pop_front();
        }
        const TraceRange trace("lbm_server: index build");
        HostIndex idx;
        const lbm_request &q = r->req;
        // the multi-lattice kernels address populations with 32-bit offsets
        std::string e = build_index(r->flags.data(), q.nx, q.ny, q.nz, q.periodic, idx, MAX_SLOTS_32);
        const int64_t fp = e.empty() ? request_footprint(q, idx) : 0;
        {
            std::lock_guard<std::mutex> lk(s->mu);
            r->index_error = e;
            r->footprint = fp;
            r->n_active = e.empty() ? idx.n_active : 0;
            r->idx = std::move(idx);
            r->index_ready = true;
        }
    }
}

// Grid and shared memory of the tick's kernel: the blocks resident at once.
cudaError_t serve_grid(lbm_server *s) {
    s->smem = s->desc.max_slots * (int)sizeof(DomainEntry);
    int per_sm = 0, sms = 0, coop = 0;
    cudaError_t e = cudaFuncSetAttribute(k_serve, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         MAX_SLOTS * (int)sizeof(DomainEntry));
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_serve, STEP_THREADS, s->smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, s->desc.device);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, s->desc.device);
    if (e == cudaSuccess && per_sm < 1) e = cudaErrorNotSupported;
    s->together = coop != 0;
    s->resident_blocks = per_sm * sms;
    s->grid = cooperative_blocks(s->resident_blocks);
    return e;
}

// The tick's work on the stream: table copy, cleared health flags, the kernel
// for `steps` steps, at most `each` of them in a launch, flags back.
cudaError_t enqueue_tick(lbm_server *s, int steps, int each) {
    const TickTable *tab = s->d_tab;
    int32_t *barrier = reinterpret_cast<int32_t *>(s->d_flags) + BARRIER_WORDS;
    uint32_t *status = s->d_flags + STATUS_WORD;
    cudaError_t e = cudaMemcpyAsync(s->d_tab, s->h_tab, sizeof(TickTable), cudaMemcpyHostToDevice, s->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(s->d_flags, 0, (STATUS_WORD + 1) * sizeof(uint32_t), s->stream);
    for (int k0 = 0; k0 < steps && e == cudaSuccess; k0 += each) {
        if (each > 1) {
            void *params[6] = {&tab, &k0, &each, &barrier, &status, &s->polls};
            e = cudaLaunchCooperativeKernel((const void *)k_serve, dim3((unsigned)s->grid), dim3(STEP_THREADS), params,
                                            (size_t)s->smem, s->stream);
            if (k0 > 0 && launch_refused(e)) e = cudaErrorLaunchFailure;  // not to be begun again
        } else {  // no barrier
            k_serve<<<(unsigned)s->grid, STEP_THREADS, (size_t)s->smem, s->stream>>>(tab, k0, 1, barrier, status, s->polls);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(s->h_flags, s->d_flags, (STATUS_WORD + 1) * sizeof(uint32_t), cudaMemcpyDeviceToHost, s->stream);
    return e;
}

// Capture the tick in a graph.
cudaError_t capture_tick(lbm_server *s) {
    cudaGraph_t g = nullptr;
    cudaError_t e = cudaStreamBeginCapture(s->stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return e;
    const cudaError_t work = enqueue_tick(s, s->desc.steps_per_tick, s->desc.steps_per_tick);
    e = cudaStreamEndCapture(s->stream, &g);
    if (work != cudaSuccess) e = work;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&s->exec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        s->exec = nullptr;
        return e;
    }
    s->graph_captures += 1;
    return e;
}

// One tick of `cells` cells: the captured graph (all steps in one launch), or,
// past LAUNCH_UPDATES or where the device does not take the cooperative
// launch, its steps in several launches.
cudaError_t run_tick(lbm_server *s, int64_t cells) {
    const int steps = s->h_tab->steps;
    if (s->together) {
        const int64_t each = std::max<int64_t>(1, s->launch_updates / std::max<int64_t>(1, cells));
        cudaError_t e = cudaSuccess;
        if (each < steps) {
            e = enqueue_tick(s, steps, (int)each);
        } else {
            if (!s->exec) e = capture_tick(s);
            if (e == cudaSuccess) e = cudaGraphLaunch(s->exec, s->stream);
            if (e == cudaSuccess) s->graph_launches += 1;
        }
        if (!launch_refused(e)) return e;
        cudaGetLastError();
        s->together = false;
        s->grid = s->resident_blocks;
    }
    return enqueue_tick(s, steps, 1);
}

// The copied flags and the host index are needed only until admission.
void drop_inputs(Request *r) {
    std::vector<uint8_t>().swap(r->flags);
    r->req.flags = nullptr;
    r->idx = HostIndex();
}

void release(lbm_server *s, Request *r) {
    if (r->ctx) {
        lbm_destroy(r->ctx);
        r->ctx = nullptr;
        s->in_use -= r->footprint;
    }
}

lbm_status admit(lbm_server *s, Request *r) {
    lbm_desc d{};
    d.nx = r->req.nx;
    d.ny = r->req.ny;
    d.nz = r->req.nz;
    d.periodic = r->req.periodic;
    d.precision = r->req.precision;
    d.fp16_scale = r->req.fp16_scale;
    d.device = s->desc.device;
    d.stream = s->stream;
    d.allocator = s->desc.allocator;
    lbm_ctx *c = nullptr;
    lbm_status st = lbm_create(&d, &c);
    if (st == LBM_OK) st = ctx_install_index(c, std::move(r->idx), true);
    if (st == LBM_OK) st = lbm_set_params(c, &r->req.params);
    const double u0[3] = {0.0, 0.0, 0.0};
    if (st == LBM_OK) st = lbm_init_equilibrium(c, 1.0, u0);
    if (st != LBM_OK) {
        r->index_error = c ? lbm_last_error(c) : "context creation failed";
        if (c) lbm_destroy(c);
        drop_inputs(r);
        r->state = LBM_REQ_FAILED;
        r->fail_status = st;
        return st;
    }
    r->ctx = c;
    drop_inputs(r);
    r->state = LBM_REQ_RUNNING;
    s->in_use += r->footprint;
    s->peak = std::max(s->peak, s->in_use);
    return LBM_OK;
}

}  // namespace

extern "C" {

lbm_status lbm_server_create(const lbm_server_desc *desc, lbm_server **out) {
    if (!desc || !out) return LBM_ERR_ARG;
    *out = nullptr;
    if (desc->budget_bytes <= 0 || desc->max_slots < 1 || desc->max_slots > MAX_SLOTS) return LBM_ERR_ARG;
    if (desc->steps_per_tick < 2 || desc->steps_per_tick > 1024 || (desc->steps_per_tick & 1)) return LBM_ERR_ARG;
    if ((desc->allocator.alloc == nullptr) != (desc->allocator.free == nullptr)) return LBM_ERR_ARG;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        cudaGetLastError();
        return LBM_ERR_CUDA;
    }
    if (desc->device < 0 || desc->device >= ndev) return LBM_ERR_ARG;
    std::unique_ptr<lbm_server> s(new lbm_server());
    s->desc = *desc;
    s->polls = barrier_polls();
    if (const char *updates = std::getenv("LBM_LAUNCH_UPDATES")) s->launch_updates = std::max(1ll, std::atoll(updates));
    cudaSetDevice(desc->device);
    // on a failure below, free what was made so far (no worker runs yet)
    auto undo = [&](lbm_status st) {
        if (s->h_tab) cudaFreeHost(s->h_tab);
        if (s->d_tab) cudaFree(s->d_tab);
        if (s->h_flags) cudaFreeHost(s->h_flags);
        if (s->d_flags) cudaFree(s->d_flags);
        if (s->own_stream) cudaStreamDestroy(s->stream);
        cudaGetLastError();
        return st;
    };
    s->stream = static_cast<cudaStream_t>(desc->stream);
    if (!s->stream) {  // graphs cannot be captured on the legacy default stream
        if (cudaStreamCreateWithFlags(&s->stream, cudaStreamNonBlocking) != cudaSuccess) return undo(LBM_ERR_CUDA);
        s->own_stream = true;
    }
    if (cudaMallocHost(&s->h_tab, sizeof(TickTable)) != cudaSuccess) {
        s->h_tab = nullptr;
        return undo(LBM_ERR_CUDA);
    }
    memset(s->h_tab, 0, sizeof(TickTable));
    // the table and the flags are part of the server, not of any lattice: not from the allocator
    if (cudaMalloc(&s->d_tab, sizeof(TickTable)) != cudaSuccess) {
        s->d_tab = nullptr;
        return undo(LBM_ERR_OOM);
    }
    if (cudaMallocHost(&s->h_flags, FLAG_WORDS * sizeof(uint32_t)) != cudaSuccess) {
        s->h_flags = nullptr;
        return undo(LBM_ERR_CUDA);
    }
    memset(s->h_flags, 0, FLAG_WORDS * sizeof(uint32_t));
    if (cudaMalloc(&s->d_flags, FLAG_WORDS * sizeof(uint32_t)) != cudaSuccess) {
        s->d_flags = nullptr;
        return undo(LBM_ERR_OOM);
    }
    if (cudaMemset(s->d_flags, 0, FLAG_WORDS * sizeof(uint32_t)) != cudaSuccess || serve_grid(s.get()) != cudaSuccess)
        return undo(LBM_ERR_CUDA);
    lbm_server *raw = s.get();
    // Index building is host work that is independent per request: a few
    // threads keep admission fed when many small requests arrive at once.
    const unsigned hw = std::thread::hardware_concurrency();
    const int nworkers = (int)std::max(1u, std::min(4u, hw > 1 ? hw - 1 : 1u));
    for (int k = 0; k < nworkers; ++k) s->workers.emplace_back(worker_loop, raw);
    *out = s.release();
    return LBM_OK;
}

lbm_status lbm_server_destroy(lbm_server *s) {
    if (!s) return LBM_OK;
    {
        std::lock_guard<std::mutex> lk(s->mu);
        s->stop = true;
    }
    s->cv.notify_all();
    for (auto &w : s->workers)
        if (w.joinable()) w.join();
    cudaSetDevice(s->desc.device);
    cudaStreamSynchronize(s->stream);
    for (auto &kv : s->reqs) release(s, kv.second.get());
    if (s->exec) cudaGraphExecDestroy(s->exec);
    if (s->h_tab) cudaFreeHost(s->h_tab);
    if (s->d_tab) cudaFree(s->d_tab);
    if (s->h_flags) cudaFreeHost(s->h_flags);
    if (s->d_flags) cudaFree(s->d_flags);
    if (s->own_stream) cudaStreamDestroy(s->stream);
    delete s;
    return LBM_OK;
}

const char *lbm_server_last_error(const lbm_server *s) { return s ? s->err.c_str() : "null server"; }

lbm_status lbm_server_submit(lbm_server *s, const lbm_request *q, int64_t *id) {
    if (!s) return LBM_ERR_ARG;
    if (!id) return sfail(s, LBM_ERR_ARG, "NULL id");
    int64_t active = 0;
    const char *why = "";
    const lbm_status st = check_request(q, s->desc.budget_bytes, &active, &why);
    if (st != LBM_OK) return sfail(s, st, why);
    const int64_t ncell = (int64_t)q->nx * q->ny * q->nz;
    std::unique_ptr<Request> r(new Request());
    r->id = s->next_id++;
    r->req = *q;
    r->flags.assign(q->flags, q->flags + ncell);
    r->req.flags = r->flags.data();
    Request *raw = r.get();
    s->reqs[r->id] = std::move(r);
    s->queue.push_back(raw->id);
    {
        std::lock_guard<std::mutex> lk(s->mu);
        s->build_queue.push_back(raw);
    }
    s->cv.notify_one();
    *id = raw->id;
    return LBM_OK;
}

lbm_status lbm_server_tick(lbm_server *s, int32_t *running, int32_t *queued) {
    const TraceRange trace("lbm_server_tick");
    if (!s) return LBM_ERR_ARG;
    cudaSetDevice(s->desc.device);
    // retire cancelled lattices
    for (size_t k = 0; k < s->resident.size();) {
        Request *r = s->reqs[s->resident[k]].get();
        if (r->cancel) {
            release(s, r);
            r->state = LBM_REQ_CANCELLED;
            s->resident.erase(s->resident.begin() + k);
        } else {
            ++k;
        }
    }
    // admit requests in submission order (the worker threads may finish the
    // indexes out of order); a request that does not fit the memory left is
    // passed over for later ones that do (first fit)
    for (auto it = s->queue.begin(); it != s->queue.end();) {
        Request *r = s->reqs[*it].get();
        bool ready;
        {
            std::lock_guard<std::mutex> lk(s->mu);
            ready = r->index_ready;
        }
        if (r->cancel) {
            if (ready) {  // the worker is done with it
                r->state = LBM_REQ_CANCELLED;
                drop_inputs(r);
                it = s->queue.erase(it);
            } else {
                ++it;
            }
            continue;
        }
        if (!ready) break;  // admission keeps submission order: wait for this index
        if (!r->index_error.empty() || r->footprint > s->desc.budget_bytes) {
            r->state = LBM_REQ_FAILED;
            r->fail_status = r->index_error.empty() ? LBM_ERR_OOM : LBM_ERR_ARG;
            drop_inputs(r);
            if (r->index_error.empty()) r->index_error = "footprint exceeds the memory budget";
            it = s->queue.erase(it);
            continue;
        }
        if ((int)s->resident.size() >= s->desc.max_slots) break;
        if (s->in_use + r->footprint > s->desc.budget_bytes) {
            ++it;
            continue;
        }
        if (admit(s, r) == LBM_OK) s->resident.push_back(r->id);
        it = s->queue.erase(it);
    }
    if (running) *running = (int32_t)s->resident.size();
    if (queued) *queued = (int32_t)s->queue.size();
    if (s->resident.empty()) return LBM_OK;

    // the tick's table
    TickTable *tab = s->h_tab;
    tab->n_domains = tab->n_tiles = tab->n_nodes = tab->steps = 0;
    const int K = s->desc.steps_per_tick;
    int64_t cells = 0;
    std::vector<int> steps_now(s->resident.size()), flag_of(s->resident.size());
    // FP32 lattices first, then FP16S: the warps, which walk the list together,
    // then change from one collision's code to the other's once a step
    for (int q = 0; q < 2; ++q)
        for (size_t k = 0; k < s->resident.size(); ++k) {
            Request *r = s->reqs[s->resident[k]].get();
            if ((r->req.precision == LBM_FP16S) != (q == 1)) continue;
            flag_of[k] = tab->n_domains;
            DomainEntry &e = tab->d[tab->n_domains++];
            ctx_tile_step_args(r->ctx, &e.a);
            e.a.status = s->d_flags + flag_of[k];  // the lattice's health flag
            e.t_base = r->steps_done;
            e.steps = (int32_t)std::min<int64_t>(K, r->req.steps - r->steps_done);
            steps_now[k] = e.steps;
            e.precision = r->req.precision;
            e.tile_begin = tab->n_tiles;
            e.node_begin = tab->n_nodes;
            tab->n_tiles += e.a.ntiles;
            tab->n_nodes += (e.a.nbnodes + 31) / 32;
            tab->steps = std::max(tab->steps, e.steps);
            cells += r->n_active;
        }
    cudaError_t e;
    {
        const TraceRange run("lbm_server_tick: graph");
        e = run_tick(s, cells);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s->stream);
    }
    if (e != cudaSuccess) return sfail(s, LBM_ERR_CUDA, std::string("tick: ") + cudaGetErrorString(e));
    if (s->h_flags[STATUS_WORD] & 2u) {  // torn lattices: no request that took part can go on
        for (const int64_t id : s->resident) {
            Request *r = s->reqs[id].get();
            r->state = LBM_REQ_FAILED;
            r->fail_status = LBM_ERR_TIMEOUT;
            r->index_error = "a bounded device-side wait gave up in a tick";
            release(s, r);
        }
        s->resident.clear();
        if (running) *running = 0;
        return sfail(s, LBM_ERR_TIMEOUT, "a bounded device-side wait gave up (tick kernel): its requests failed");
    }
    s->ticks += 1;
    // account, retire finished lattices
    std::vector<int64_t> still;
    for (size_t k = 0; k < s->resident.size(); ++k) {
        Request *r = s->reqs[s->resident[k]].get();
        ctx_advance(r->ctx, steps_now[k]);
        r->steps_done += steps_now[k];
        s->cell_updates += (double)r->n_active * steps_now[k];
        if (s->h_flags[flag_of[k]]) {  // the tick's health check saw a non-finite cell: evict
            r->state = LBM_REQ_FAILED;
            r->fail_status = LBM_ERR_UNSTABLE;
            r->index_error = "non-finite density or velocity found by the health check at step " +
                             std::to_string(r->steps_done);
            release(s, r);
        } else if (r->steps_done >= r->req.steps) {
            r->rho.assign((size_t)r->n_active, 0.0);
            r->u.assign((size_t)r->n_active * 3, 0.0);
            lbm_status st = lbm_get_moments(r->ctx, r->rho.data(), r->u.data(), LBM_LAYOUT_ACTIVE);
            r->state = st == LBM_OK ? LBM_REQ_DONE : LBM_REQ_FAILED;
            r->fail_status = st;
            if (st != LBM_OK) r->index_error = lbm_last_error(r->ctx);
            release(s, r);
            s->finished += 1;
        } else {
            still.push_back(r->id);
        }
    }
    s->resident.swap(still);
    if (running) *running = (int32_t)s->resident.size();
    return LBM_OK;
}

lbm_status lbm_server_poll(lbm_server *s, int64_t id, int32_t *state, int64_t *steps_done) {
    if (!s) return LBM_ERR_ARG;
    auto it = s->reqs.find(id);
    if (it == s->reqs.end()) return sfail(s, LBM_ERR_ARG, "unknown request id");
    if (state) *state = it->second->state;
    if (steps_done) *steps_done = it->second->steps_done;
    return LBM_OK;
}

lbm_status lbm_server_cells(lbm_server *s, int64_t id, int64_t *active_cells) {
    if (!s || !active_cells) return LBM_ERR_ARG;
    auto it = s->reqs.find(id);
    if (it == s->reqs.end()) return sfail(s, LBM_ERR_ARG, "unknown request id");
    std::lock_guard<std::mutex> lk(s->mu);
    if (it->second->n_active < 0) return sfail(s, LBM_ERR_STATE, "index not built yet");
    *active_cells = it->second->n_active;
    return LBM_OK;
}

lbm_status lbm_server_result(lbm_server *s, int64_t id, double *rho, double *u) {
    if (!s) return LBM_ERR_ARG;
    auto it = s->reqs.find(id);
    if (it == s->reqs.end()) return sfail(s, LBM_ERR_ARG, "unknown request id");
    Request *r = it->second.get();
    if (r->state == LBM_REQ_QUEUED || r->state == LBM_REQ_RUNNING)
        return sfail(s, LBM_ERR_STATE, "request not finished");
    // a terminal request is released here, whatever its outcome (the worker
    // threads are done with it: a request only leaves QUEUED once its index
    // is built)
    if (r->state == LBM_REQ_CANCELLED) {
        s->reqs.erase(it);
        return sfail(s, LBM_ERR_STATE, "request was cancelled");
    }
    if (r->state == LBM_REQ_FAILED) {
        const lbm_status st = r->fail_status != LBM_OK ? r->fail_status : LBM_ERR_ARG;
        const std::string msg = "request failed: " + r->index_error;
        s->reqs.erase(it);
        return sfail(s, st, msg);
    }
    if (rho) memcpy(rho, r->rho.data(), r->rho.size() * 8);
    if (u) memcpy(u, r->u.data(), r->u.size() * 8);
    s->reqs.erase(it);
    return LBM_OK;
}

lbm_status lbm_server_cancel(lbm_server *s, int64_t id) {
    if (!s) return LBM_ERR_ARG;
    auto it = s->reqs.find(id);
    if (it == s->reqs.end()) return sfail(s, LBM_ERR_ARG, "unknown request id");
    it->second->cancel = true;
    return LBM_OK;
}

lbm_status lbm_server_info(lbm_server *s, double out[8]) {
    if (!s || !out) return LBM_ERR_ARG;
    out[0] = s->cell_updates;
    out[1] = s->ticks;
    out[2] = (double)s->in_use;
    out[3] = (double)s->peak;
    out[4] = s->graph_launches;
    out[5] = s->graph_captures;
    out[6] = s->finished;
    out[7] = (double)s->queue.size();
    return LBM_OK;
}

lbm_status lbm_server_check_request(const lbm_request *req, int64_t budget_bytes, int64_t out[4],
                                    const char **why) {
    static thread_local std::string msg;
    const char *w = "";
    int64_t active = 0;
    if (out) out[0] = out[1] = out[2] = out[3] = 0;
    lbm_status st = check_request(req, budget_bytes, &active, &w);
    if (st == LBM_OK) {
        HostIndex idx;
        msg = build_index(req->flags, req->nx, req->ny, req->nz, req->periodic, idx, MAX_SLOTS_32);
        if (!msg.empty()) {
            st = LBM_ERR_ARG;
            w = msg.c_str();
        } else {
            const int64_t fp = request_footprint(*req, idx);
            if (out) {
                out[0] = idx.n_active;
                out[1] = idx.nslots;
                out[2] = fp;
                out[3] = (int64_t)idx.bnodes.size();
            }
            if (fp > budget_bytes) {
                st = LBM_ERR_OOM;
                w = "footprint exceeds the memory budget";
            }
        }
    }
    if (why) *why = w;
    return st;
}

}  // extern "C"
