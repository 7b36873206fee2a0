// Batched count that allocates no memory.
//
// Some callers cannot allocate device memory when they want to run a query:
// real-time loops that reserve all of their memory up front, processes that
// run under a fixed memory cap or an allocator that forbids cudaMalloc after
// start-up, and plug-ins whose host framework owns every allocation.
// tm_count_batch_noalloc serves them.  It runs the same persistent multi-query
// count kernel as tm_count_batch, but the kernel's scratch -- the control
// block, the per-query launch records and the task queue for donated subtrees
// -- lives in one fixed, file-scope __device__ array instead of buffers
// obtained from cudaMalloc.  The caller passes the graph, the compiled queries
// and the device array that receives the totals.
//
// The array is g_noalloc_scratch below: TM_NOALLOC_SCRATCH_BYTES bytes, present
// on every GPU that loads this library until the process exits.  It holds at
// most TM_NOALLOC_MAX_QUERIES launch records and TM_NOALLOC_TASKS task slots,
// which one launch uses up as it donates (slots are not reused within it).
// The launch records are staged in a file-scope host buffer (not on the
// caller's stack, which may be small in a plug-in's threads); a mutex guards
// it while the records are copied out.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>

#include "tm_internal.cuh"

namespace tmg {

namespace {

constexpr int NOALLOC_MAX_QUERIES = TM_NOALLOC_MAX_QUERIES;
constexpr uint64_t NOALLOC_TASKS = TM_NOALLOC_TASKS;

// byte layout of the static array
constexpr int PARTS = 2;                 // launches of a call, see below
constexpr size_t CTRL_STRIDE = 512;      // a control block for each
constexpr size_t OFF_CTRL = 0;
constexpr size_t OFF_QDEV = PARTS * CTRL_STRIDE;
constexpr size_t OFF_READY = (OFF_QDEV + NOALLOC_MAX_QUERIES * sizeof(QueryDev) + 255) / 256 * 256;
constexpr size_t OFF_TASKS = (OFF_READY + NOALLOC_TASKS + 255) / 256 * 256;
constexpr size_t NOALLOC_END = OFF_TASKS + NOALLOC_TASKS * sizeof(Task);
static_assert(NOALLOC_END <= TM_NOALLOC_SCRATCH_BYTES, "static scratch layout exceeds its stated size");
static_assert(sizeof(Ctrl) <= CTRL_STRIDE, "control blocks overlap");

// The scratch itself.  In host code this name is only a host-side stand-in
// for the symbol; its device address comes from cudaGetSymbolAddress below.
static __device__ __align__(256) unsigned char g_noalloc_scratch[TM_NOALLOC_SCRATCH_BYTES];

// Host staging of the control blocks and launch records (about 60 KB).
struct Stage {
    struct {
        Ctrl c;
        unsigned char pad[CTRL_STRIDE - sizeof(Ctrl)];
    } ctrl[PARTS];
    QueryDev q[NOALLOC_MAX_QUERIES];
};
Stage g_stage;
std::mutex g_stage_mu;

// What a call reads back of each control block.
struct Outcome {
    unsigned long long q_reserve, q_head;
    int pad, idle;
    unsigned err, donated;
};
static_assert(offsetof(Ctrl, err) - offsetof(Ctrl, q_reserve) == offsetof(Outcome, err) &&
              offsetof(Ctrl, donated) - offsetof(Ctrl, q_reserve) == offsetof(Outcome, donated), "control block layout");

constexpr int MAX_DEVICES = 64;
std::mutex g_setup_mu;
unsigned char* g_scratch_dev[MAX_DEVICES] = {nullptr};

// Once per device, with that device current: the array's device address.
tm_status scratch_address(int device, unsigned char** out) {
    if (device < 0 || device >= MAX_DEVICES) {
        set_error("device index beyond the no-alloc set-up table");
        return TM_E_INVALID;
    }
    std::lock_guard<std::mutex> lk(g_setup_mu);
    if (!g_scratch_dev[device]) {
        void* p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(g_noalloc_scratch)");
        g_scratch_dev[device] = (unsigned char*)p;
    }
    *out = g_scratch_dev[device];
    return TM_OK;
}

}  // namespace

}  // namespace tmg

using namespace tmg;

extern "C" tm_status tm_count_batch_noalloc(tm_graph* g, tm_query* const* qs, int nq, void* stream,
                                            uint64_t* totals_dev) {
    if (!g || !qs || !totals_dev) { set_error("null argument"); return TM_E_INVALID; }
    if (nq < 1 || nq > NOALLOC_MAX_QUERIES) {
        set_error("tm_count_batch_noalloc: nq must be in [1, " + std::to_string(NOALLOC_MAX_QUERIES) +
                  "], the capacity of its static scratch");
        return TM_E_INVALID;
    }
    TM_ENTER(g->device);
    cudaStream_t st = (cudaStream_t)stream;
    unsigned char* base = nullptr;
    tm_status s = scratch_address(g->device, &base);
    if (s != TM_OK) return s;
    const uint64_t m = (uint64_t)g->v.m;
    for (int j = 0; j < nq; ++j)
        if (!qs[j] || query_graph(qs[j]) != g) { set_error("null or mismatched query in batch"); return TM_E_INVALID; }
    // Every call reuses the array: clear the caller's totals, then rewrite the
    // control block and the launch records and clear the task-ready flags.
    InFlight call(st, &g->unsettled);
    TM_CUDA(cudaMemsetAsync(totals_dev, 0, (size_t)nq * sizeof(uint64_t), st));
    if (m == 0) return cudaStreamSynchronize(st) == cudaSuccess ? TM_OK : cuda_fail(cudaGetLastError(), "sync");
    // Queries with look-ahead or long frames in a launch of their own: their instances run all of a launch at their
    // registers, shared memory and frames, and without pairs (two 4-edge paths over half-day windows on 10M
    // edges 66 ms, with a chorded 4-cycle in their launch 127).
    struct Part {
        int first, count, warp_smem, warps;
        unsigned feat;
        uint64_t chunks;
    } part[PARTS];
    {
        std::lock_guard<std::mutex> lk(g_stage_mu);
        memset(g_stage.ctrl, 0, sizeof g_stage.ctrl);
        int at = 0;
        for (int p = 0; p < PARTS; ++p) {
            Part& pt = part[p];
            pt = Part{at, 0, 16, 1, 0u, 0};
            for (int j = 0; j < nq && at < nq; ++j) {
                QueryDev& qd = g_stage.q[at];
                memset(&qd, 0, sizeof(QueryDev));
                query_plan(qs[j], &qd.plan);
                if (launch_part(plan_features(qd.plan)) != p) continue;
                qd.root_begin = 0;
                qd.root_end = m;
                qd.plan.tune.chunk_roots = effective_chunk(g, qd.plan, m * (uint64_t)nq);
                qd.n_chunks = n_chunks(m, qd.plan.tune.chunk_roots);
                qd.chunk_base = pt.chunks;
                pt.chunks += qd.n_chunks;
                qd.total = (unsigned long long*)totals_dev + j;
                pt.warp_smem = std::max(pt.warp_smem, qd.plan.warp_smem);
                pt.warps = std::max(pt.warps, qd.plan.tune.warps_per_block);
                pt.feat |= plan_features(qd.plan);
                ++at;
            }
            pt.count = at - pt.first;
            g_stage.ctrl[p].c.total_chunks = pt.chunks;
        }
        // pageable source: the copy has left this buffer when the call returns
        TM_CUDA(cudaMemcpyAsync(base + OFF_CTRL, &g_stage, OFF_QDEV + (size_t)nq * sizeof(QueryDev),
                                cudaMemcpyHostToDevice, st));
    }
    for (int p = 0; p < PARTS; ++p) {
        const Part& pt = part[p];
        if (pt.count == 0) continue;
        TM_CUDA(cudaMemsetAsync(base + OFF_READY, 0, NOALLOC_TASKS, st));
        Scratch view;                       // points into the static array; never freed
        view.device = g->device;
        view.head = (char*)(base + OFF_CTRL + p * CTRL_STRIDE);
        view.qcap = NOALLOC_MAX_QUERIES;
        view.tasks = (Task*)(base + OFF_TASKS);
        view.ready = base + OFF_READY;
        view.task_cap = NOALLOC_TASKS;
        s = launch_search(g, MODE_COUNT, (const QueryDev*)(base + OFF_QDEV) + pt.first, pt.count, pt.warp_smem, pt.warps,
                          pt.feat, &view, st,
                          launch_blocks(g, search_launch_cfg(g, MODE_COUNT, pt.warp_smem, pt.warps, pt.feat), pt.chunks));
        if (s != TM_OK) return s;
    }
    Outcome done[PARTS];                // of a launch not made: as staged, nothing
    TM_CUDA(cudaMemcpy2DAsync(done, sizeof(Outcome), base + OFF_CTRL + offsetof(Ctrl, q_reserve), CTRL_STRIDE, sizeof(Outcome), PARTS,
                              cudaMemcpyDeviceToHost, st));
    TM_CUDA(cudaStreamSynchronize(st));
    call.settle();
    note_search_stats((uint64_t)done[0].donated + done[1].donated, done[0].q_reserve + done[1].q_reserve);
    if (done[0].err || done[1].err) { set_error("a bounded device wait timed out"); return TM_E_TIMEOUT; }
    return TM_OK;
}
