// Internal declarations shared by the library's translation units.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/tm.h"

namespace tmg {

// ------------------------------------------------------------------ errors

void set_error(const std::string& msg);

// Kernels this library has launched (all entry points, all threads).
void note_launches(uint64_t n);
tm_status cuda_fail(cudaError_t e, const char* what);

// Every device and pinned-host allocation of the library goes through these,
// so that tm_inject_alloc_failure can make one of them fail like an
// out-of-memory device (cudaErrorMemoryAllocation, nothing allocated).
// dev_malloc returns memory of the library's pool on the current device, ready for any stream; dev_free takes it
// back.  The pool keeps up to POOL_KEEP (or a running server's budget, if that is more) beyond dev_malloc's
// memory in use; pool_give_back returns what is above that, which the driver otherwise does at the
// next synchronisation.  `settled`: nothing in flight uses the memory any more, else the free waits for the
// device first: cudaFree does not wait for the users of pool memory.
constexpr uint64_t POOL_KEEP = 4ull << 30;
cudaError_t dev_malloc(void** p, size_t bytes);
void dev_free(void* p, int device, bool settled);
cudaError_t dev_malloc_async(void** p, size_t bytes, cudaStream_t st);
void pool_give_back(int device);
void pool_budget(int device, uint64_t bytes, bool running);
cudaError_t host_alloc_pinned(void** p, size_t bytes);

// Select the device and drop any error another library left on this thread,
// so that only this call's own CUDA errors are reported.
#define TM_ENTER(dev)                                         \
    do {                                                      \
        cudaGetLastError();                                   \
        TM_CUDA(cudaSetDevice(dev));                          \
    } while (0)

#define TM_CUDA(call)                                         \
    do {                                                      \
        cudaError_t _e = (call);                              \
        if (_e != cudaSuccess) return tmg::cuda_fail(_e, #call); \
    } while (0)

// ------------------------------------------------------------ device graph

// Device-resident temporal graph (paper Section 2.2): the chronological edge
// list plus out- and in-adjacency in time order, stored column-wise so that a
// binary search touches only the time column and a window scan reads
// contiguous (t, neighbour) runs.
struct GraphView {
    int64_t n, m;
    const int32_t* src;       // by edge id
    const int32_t* dst;
    const int64_t* t;
    const uint8_t* elabel;    // nullable
    const uint8_t* nlabel;    // nullable
    const uint32_t* off[2];   // [0] out, [1] in : n+1 list offsets
    const int64_t* at[2];     // list entry time
    const int32_t* anbr[2];   // list entry neighbour (dst for out, src for in)
    const int32_t* aeid[2];   // list entry edge id
    // successor index, by edge id e = (u, v, t): first position with time > t in
    // out(u), in(v), out(v), in(u).  Each word is {x: absolute position in the
    // list columns, y: time of that entry minus t, saturated at SUCC_FAR, or
    // SUCC_END when the list has no later entry}, so one load both starts a
    // window and, for most windows, proves it empty.  Edge e's word is nxt[kind][2 * e]: the
    // two words found in out-list order (out(u), in(u)) lie side by side, and so do the two found in
    // in-list order, since each pair is written at once to an edge from anywhere.
    const uint2* nxt[4];
    // the same, indexed by list position for the common continuations: [0] out-list
    // entry -> next later in that out-list, [1] out-list entry -> out(its neighbour),
    // [2] in-list entry -> next later in that in-list, [3] in-list entry -> in(its neighbour)
    const uint2* pnx[4];
    // root filter, by edge id: the gaps of the edge's four successor words as gap_code()
    // bytes (byte succ_byte(kind)), rounded down, so that one load tells for four lists
    // whether they have an entry soon enough
    const uint32_t* rcode;
    // out-lists again, ordered by (neighbour, time) within each node (offsets off[0]):
    // the edges u -> v form one contiguous, time-ordered range
    const int32_t* pnbr;
    const int64_t* pt;
    const int32_t* peid;
};

constexpr uint32_t SUCC_END = 0xFFFFFFFFu;   // successor word: no later entry in the list
constexpr uint32_t SUCC_FAR = 0xFFFFFFFEu;   // successor word: time gap >= this

enum SuccKind : int8_t { NX_OUT_SRC = 0, NX_IN_DST = 1, NX_OUT_DST = 2, NX_IN_SRC = 3, NX_NONE = -1 };

// A time gap as a 7-bit floating code (5 bits of exponent, 2 of mantissa, rounded down): larger gaps never
// have smaller codes.  GAP_CODE_END (SUCC_END) is above the code of any gap.
constexpr uint32_t GAP_CODE_END = 127;
__host__ __device__ inline uint32_t gap_code(uint32_t gap) {
    if (gap == SUCC_END) return GAP_CODE_END;
    if (gap < 4u) return gap;
#ifdef __CUDA_ARCH__
    const uint32_t e = 31u - (uint32_t)__clz((int)gap);
#else
    const uint32_t e = 31u - (uint32_t)__builtin_clz(gap);
#endif
    return (e - 1u) << 2 | (gap >> (e - 2u) & 3u);
}
// Byte of rcode that holds a list's code.
__host__ __device__ constexpr int succ_byte(int kind) { return kind; }

struct TuneKey {
    uint64_t shape;     // motif structure hash
    int dbucket;        // floor(log2(delta + 1))
    bool operator==(const TuneKey& o) const { return shape == o.shape && dbucket == o.dbucket; }
};
// A tuned setting: `automatic` keeps the chunk size that follows the input (see effective_chunk).
struct Tuned {
    tm_tuning tune;
    bool automatic;
};
struct TuneKeyHash {
    size_t operator()(const TuneKey& k) const { return (size_t)(k.shape * 1315423911ULL + (uint64_t)k.dbucket); }
};

}  // namespace tmg

struct tm_graph {
    int device = 0;
    std::atomic<int> unsettled{0};   // calls on this graph that are running, or ended without having waited for their work
    tmg::GraphView v{};
    std::vector<void*> allocs;     // device buffers owned by the graph
    char* slab = nullptr;          // the graph's columns, carved from one allocation
    size_t slab_used = 0, slab_cap = 0;
    int32_t* perm = nullptr;       // device: edge id -> input index
    uint64_t device_bytes = 0;
    uint32_t longest_list = 0;     // of any node, in either direction (an upper bound where long_frames(m) is false)
    int num_sms = 0;
    std::mutex tune_mu;
    std::unordered_map<tmg::TuneKey, tmg::Tuned, tmg::TuneKeyHash> tuned;
    // serving: device ms one request of a (shape, delta bucket, flavour) takes,
    // learnt from timed launches and shared by every server of this graph
    std::mutex cost_mu;
    std::unordered_map<uint64_t, double> serve_cost_ms;
};

namespace tmg {

// A call that puts work on a stream: until it has waited for that work, what the work
// uses (the graph's columns, a query's scratch) is not settled.  A call that ends early, on
// an error, waits too: its caller may free, or use on another stream, whatever the work still reads.
class InFlight {
    cudaStream_t st;
    std::atomic<int>*a, *b;

public:
    InFlight(cudaStream_t s, std::atomic<int>* x, std::atomic<int>* y = nullptr) : st(s), a(x), b(y) {
        a->fetch_add(1);
        if (b) b->fetch_add(1);
    }
    InFlight(InFlight&& o) noexcept : st(o.st), a(o.a), b(o.b) { o.a = o.b = nullptr; }
    InFlight(const InFlight&) = delete;
    ~InFlight() { wait(); }
    // the work has been waited for
    void settle() {
        if (a) a->fetch_sub(1);
        if (b) b->fetch_sub(1);
        a = b = nullptr;
    }
    // Wait for it here.  What could not be waited for stays unsettled.
    void wait() {
        if (!a) return;
        if (cudaStreamSynchronize(st) == cudaSuccess) settle();
        else cudaGetLastError();
        a = b = nullptr;
    }
};

// --------------------------------------------------------------- the plan

enum LevelKind : int8_t { EXT_OUT = 0, EXT_IN = 1, CLOSE = 2, FREE = 3 };

// How one search level binds motif edge i (paper Section 5.1.2 "minfo"):
// which mapped node supplies the candidate list, which mapped nodes a new
// node must differ from, and the constraints checked on a candidate.
constexpr int TM_MAX_LOOK = 3;

struct LevelPlan {
    int8_t kind;       // LevelKind
    int8_t a;          // EXT_OUT: slot of x_i; EXT_IN: slot of y_i; CLOSE: slot of x_i
    int8_t b;          // CLOSE: slot of y_i
    int8_t nb;         // slots bound before this level
    int16_t elabel;    // -1 = any
    int16_t nl0;       // label of the (first) new node, -1 = any
    int16_t nl1;       // FREE: label of the second new node (y_i)
    int8_t nx_a;       // SuccKind giving the window start of the list used by EXT / CLOSE(out) levels
    int8_t nx_b;       // SuccKind for the in-list option of a CLOSE level
    uint8_t anti_mask; // anti-edges whose nodes and attached edge are all bound once edge i is
    uint8_t n_look;    // later motif edges (after i+1) whose two nodes are first both bound by edge i
    int8_t look_u[TM_MAX_LOOK];  // their endpoint slots: an edge look_u -> look_v must exist in
    int8_t look_v[TM_MAX_LOOK];  // (t_i, t_root + delta], else no match extends this partial match
    int8_t fx, fdir;         // candidate filter (Hot::FILT): new nodes must be in bound slot fx's list of direction fdir
    int8_t fnx;              // SuccKind giving the start of that list's window, after edge i - 1
    uint32_t hot;            // the fields every step needs, packed (see Hot)
    int32_t frame_off;       // byte offset of this level's frame in a warp's shared block (count)
    int32_t frame_off_fill;  // same, enumerate-fill layout (frames also carry edge ids)
    int32_t anti_row_off;    // byte offset of the anti-edge time rows within this level's frame
    int32_t anti_row_off_fill;
    int32_t filt_off;        // byte offset of the candidate filter within this level's frame
    int32_t filt_off_fill;
    int64_t gap;             // t_i - t_{i-1} bound (INT64_MAX = none)
};

// LevelPlan::hot.  One 4-byte load per level change tells a step what kind of
// level it is on, which slots it reads and which optional checks apply; the
// rest of the plan is read only by the checks that need it.
struct Hot {
    static constexpr uint32_t ELABEL = 1u << 18, NLABEL = 1u << 19, ANTI = 1u << 20, LOOK = 1u << 21, GAP = 1u << 22;
    // the level's look-ahead on its new node is filtered first (see CandidateFilter)
    static constexpr uint32_t FILT = 1u << 23;
    // level k - 2, when the last two edges extend by new nodes from one list, without labels,
    // gaps, anti-edges or look-ahead: their pairs are counted from the window itself
    static constexpr uint32_t PAIRS = 1u << 24;
    static uint32_t pack(const LevelPlan& lp) {
        return (uint32_t)lp.kind | (uint32_t)(lp.a & 7) << 2 | (uint32_t)(lp.b & 7) << 5 | (uint32_t)lp.nb << 8 |
               (uint32_t)(lp.nx_a + 1) << 12 | (uint32_t)(lp.nx_b + 1) << 15 | (lp.elabel >= 0 ? ELABEL : 0u) |
               (lp.nl0 >= 0 || lp.nl1 >= 0 ? NLABEL : 0u) | (lp.anti_mask ? ANTI : 0u) | (lp.n_look ? LOOK : 0u) |
               (lp.gap != INT64_MAX ? GAP : 0u) | (lp.n_look && lp.kind <= EXT_IN ? FILT : 0u);
    }
    __host__ __device__ static int kind(uint32_t h) { return (int)(h & 3u); }
    __host__ __device__ static int a(uint32_t h) { return (int)(h >> 2 & 7u); }
    __host__ __device__ static int b(uint32_t h) { return (int)(h >> 5 & 7u); }
    __host__ __device__ static int nb(uint32_t h) { return (int)(h >> 8 & 15u); }
    __host__ __device__ static int nx_a(uint32_t h) { return (int)(h >> 12 & 7u) - 1; }
    __host__ __device__ static int nx_b(uint32_t h) { return (int)(h >> 15 & 7u) - 1; }
};

// One temporal anti-edge (paper Section 2.1, Section 5.4.3), checked at the
// level where its two nodes and its attached edge are all bound.
struct AntiPlan {
    int8_t xs, ys;     // slots of the absent edge's endpoints
    int8_t edge;       // attached motif edge i
    int8_t same_pair;  // the attached edge joins the same two nodes (exclude it)
    int32_t pad;
    int64_t delta;     // window [t(e_i), t(e_i) + delta]
};

// Parents per frame (at most two per lane).  A level is descended into once its
// frame holds cap - 32 parents, so one more 32-wide step of its parent level
// always fits.  Count frames hold 48 (descend at 16): the smaller shared
// memory footprint leaves more of each SM's unified L1 / shared memory to L1;
// fill frames carry edge ids and keep 64 (descend at 32).
constexpr int FCAP_COUNT = 48;
// Counts with look-ahead: the signatures leave shared memory for 12 warps per SM at 48, for 16 at 40, which
// is worth more than fuller child frames (chorded 4-cycle on 100M edges 41.5 -> 34.2 ms; plain
// motifs lose: 4-path over 15 h windows 19.9 -> 21.2 ms).  A launch with look-ahead also runs plans without
// it, laid out for 48: their frames have room to spare.
constexpr int FCAP_LOOK = 40;
constexpr int FCAP_FILL = 64;

struct Plan {
    int32_t k, n_nodes;
    int64_t delta;
    int16_t elabel0, nl_x0, nl_y0, pad0;
    int32_t warp_smem;             // bytes of shared memory a warp needs (count)
    int32_t warp_smem_fill;        // same, enumerate fill
    tm_tuning tune;
    uint64_t shape_hash;
    int32_t n_anti;
    uint8_t anti_mask0;            // anti-edges checked when the root binds edge 0
    uint8_t auto_chunk;            // 1: tune.chunk_roots is the default and may shrink on small inputs
    uint8_t long_frames;           // see FEAT_LONG
    uint8_t pad1;
    uint32_t root_codes;           // lists a match rooted at an edge must continue in: the largest gap allowed, as
                                   // bytes laid out like GraphView::rcode (GAP_CODE_END: the list is not needed)
    AntiPlan anti[TM_MAX_ANTI];
    LevelPlan lv[TM_MAX_EDGES];    // lv[i] for i = 1..k-1 (lv[0]: only the look-ahead of the root)
};

// Code a plan needs beyond plain search: anti-edge checks, look-ahead checks; or can use: pairs.
// FEAT_LONG: the windows of a frame may add up to more than 32 bits hold, and the frame then begins in parts. In
// instances of its own: in all of them the code made plain searches 5 to 7% slower (64-query batch 11.9 -> 12.8 ms).
constexpr unsigned FEAT_ANTI = 1u, FEAT_LOOK = 2u, FEAT_PAIRS = 4u, FEAT_LONG = 64u;
inline unsigned plan_features(const Plan& p) {
    unsigned f = (p.n_anti > 0 ? FEAT_ANTI : 0u) | (p.long_frames ? FEAT_LONG : 0u);
    for (int i = 0; i < TM_MAX_EDGES; ++i)
        f |= (p.lv[i].n_look ? FEAT_LOOK : 0u) | (p.lv[i].hot & Hot::PAIRS ? FEAT_PAIRS : 0u);
    return f;
}

// Launches that take queries of any kind (served batches, the call without allocation) keep two sorts apart: 1 for
// queries with look-ahead or long frames, whose instances cost the others more than a launch.
inline int launch_part(unsigned feat) { return feat & (FEAT_LOOK | FEAT_LONG) ? 1 : 0; }

// Frame field offsets (bytes, relative to frame start), CAP entries each.
//   tprev i64, tend - tprev u32 (0xFFFFFFFF when it does not fit: t_root + delta is
//   then rebuilt from the root edge), beg u32 (bits 31/30: list kind), len u32, root u32,
//   node[nb] i32, eid[i] i32 (enumerate only), anti_t[n_anti] i64 (motifs with
//   anti-edges: time of each anti-edge's attached edge once bound)
template <int CAP>
struct FrameLayout {
    static constexpr int TPREV = 0;
    static constexpr int TEND = TPREV + 8 * CAP;
    static constexpr int BEG = TEND + 4 * CAP;
    static constexpr int LEN = BEG + 4 * CAP;
    static constexpr int ROOT = LEN + 4 * CAP;
    static constexpr int NODE = ROOT + 4 * CAP;
};
// A frame's candidate filter (levels with Hot::FILT, after the anti-edge rows).  The
// list windows the signatures are built from are needed until the frame is begun, the
// pending candidates only after, so the two share their bytes.
struct CandidateFilter {
    static constexpr int WORDS = 16;               // signature words per parent
    static constexpr int PEND = 96;                // up to 31 pending candidates and the 64 of a filter step
    static constexpr int BEG = 0, LEN = 256;       // u32 per parent: window of the list the signature covers
    static constexpr int POS = 0, PAR = 4 * PEND;  // u32 list position, u8 parent of each pending candidate
    static constexpr int SIG = 512;                // WORDS words per parent
    static constexpr int bytes(int cap) { return SIG + 4 * WORDS * cap; }
};
static_assert(4 * FCAP_FILL <= 256 && CandidateFilter::PAR + CandidateFilter::PEND <= CandidateFilter::SIG,
              "candidate filter rows overlap");

// Count frames (no edge ids) or fill frames (edge ids of the bound edges).
inline int frame_bytes(int nb, int level, bool with_eids, int cap_count, int n_anti = 0, bool filter = false) {
    const int cap = with_eids ? FCAP_FILL : cap_count;
    return FrameLayout<FCAP_FILL>::NODE / FCAP_FILL * cap + 4 * cap * (nb + (with_eids ? level : 0)) + 8 * cap * n_anti +
           (filter ? CandidateFilter::bytes(cap) : 0);
}
// A warp's shared block starts with its root buffer: up to 31 roots left over
// and the 128 of one scan step.
constexpr int ROOT_BUF_BYTES = 160 * 4;

tm_status build_plan(const tm_graph* g, const tm_motif* m, Plan* out);
uint64_t plan_shape_hash(const tm_motif* m);

// --------------------------------------------------------- device scratch

// Donated search task: one partial match (its mapped nodes, times and window).
struct Task {
    int16_t query;
    int16_t level;
    uint32_t beg;        // bit 31: in-list
    uint32_t len;
    uint32_t root;
    int64_t tprev;
    int64_t tend;
    int32_t node[TM_MAX_NODES];
};
static_assert(sizeof(Task) == 64, "task is one 64-byte record");

// Per-launch control block.  The root-chunk cursor is claimed by every warp
// many times per launch; the queue and idle counters are polled by waiting
// warps: they sit on separate 128-byte lines so polling never delays claims.
struct Ctrl {
    unsigned long long total_chunks; // root chunks of all queries of the launch
    unsigned long long pad0[15];
    unsigned long long next_chunk;   // root-chunk cursor (own line)
    unsigned long long pad1[15];
    unsigned long long q_reserve;    // task slots reserved by donors
    unsigned long long q_head;       // next task slot to pop (read together with q_reserve)
    int pad3;
    int idle;                        // blocks with a warp waiting for tasks
    unsigned int err;                // 0 or TM_E_TIMEOUT
    unsigned int donated;            // tasks donated (diagnostic)
    unsigned long long done_chunks;  // root chunks whose whole subtree has been searched
    unsigned long long done_tasks;   // task slots run (or found void)
    unsigned long long pad2[10];
};
static_assert(sizeof(Ctrl) == 384, "control block is three 128-byte lines");

// Enumeration chunk buffer of a query with nch root chunks: nch + 1 per-chunk
// match counts (scanned in place into row offsets by the caller), then the
// number of chunks holding a match whose rows start below the cap, and those
// chunks' ids (uint32, in no particular order; written by list_chunks after
// the scan).  The fill pass searches only the listed chunks.  The count pass
// needs the counts and the list length zeroed: the first (nch + 2) * 8 bytes.
inline size_t chunk_buf_bytes(uint64_t nch) { return (size_t)(nch + 2) * 8 + (size_t)nch * 4; }

struct QueryDev {                    // one query of a launch
    Plan plan;
    uint64_t root_begin, root_end;
    uint64_t n_chunks;
    uint64_t chunk_base;             // first global chunk index of this query
    unsigned long long* total;       // device counter
    unsigned long long* per_root;    // nullable (indexed by root - root_begin)
    unsigned long long* chunk_cnt;   // nullable (enumerate count pass): chunk buffer, counts + list
    const unsigned long long* chunk_off;  // enumerate fill: chunk buffer, offsets + list
    int32_t* match_out;              // enumerate fill
    uint64_t cap;
    unsigned long long* work;        // nullable: tm_work counters (2 + 2*TM_MAX_EDGES + 1)
};

// Device memory a launch uses beyond its inputs and outputs, plus the pinned
// host staging it is initialised from.  Layout of `head` (device) and `stage`
// (pinned host): one Ctrl, then nq QueryDev records.
struct Scratch {
    int device = 0;
    char* head = nullptr;            // device: Ctrl + QueryDev[qcap]
    char* stage = nullptr;           // pinned host mirror of head
    int qcap = 0;
    Task* tasks = nullptr;
    uint8_t* ready = nullptr;
    uint64_t task_cap = 0;
    unsigned long long* counters = nullptr;   // device: totals, work counters
    unsigned long long* counters_host = nullptr;  // pinned mirror
    uint64_t counters_len = 0;
    unsigned long long* chunk_cnt = nullptr;  // device: enumerate per-chunk counts / offsets
    uint64_t chunk_cap = 0;
    void* scan_tmp = nullptr;
    size_t scan_tmp_bytes = 0;
    Ctrl* ctrl() const { return (Ctrl*)head; }
    QueryDev* qdev() const { return (QueryDev*)(head + sizeof(Ctrl)); }
    Ctrl* ctrl_stage() const { return (Ctrl*)stage; }
    QueryDev* qdev_stage() const { return (QueryDev*)(stage + sizeof(Ctrl)); }
    size_t head_bytes(int nq) const { return sizeof(Ctrl) + (size_t)nq * sizeof(QueryDev); }
};

void drop_batches(const tm_graph* g);

// Record the donation counters of a finished count-mode launch for
// tm_last_search_stats (per calling thread).
void note_search_stats(uint64_t donated, uint64_t reserved);

// The query's plan with the graph's cached tuning for its shape applied.
void query_plan(tm_query* q, Plan* out);

// The graph a query was compiled for, and the motif it was compiled from.
const tm_graph* query_graph(const tm_query* q);
const tm_motif* query_motif(const tm_query* q);

// Turn a chunk buffer's counts into row offsets and, where cap > 0, list the chunks the fill pass must search:
// none when the count launch, whose control block is `counted`, gave up.
tm_status chunk_offsets(unsigned long long* chunk_buf, uint64_t nch, uint64_t cap, const Ctrl* counted, void* scan_tmp,
                        int num_sms, cudaStream_t st);

tm_status scratch_reserve(Scratch* s, int device, int nq, uint64_t counters_len, uint64_t chunks,
                          uint64_t task_cap);
void scratch_free(Scratch* s, bool settled);

enum Mode { MODE_COUNT = 0, MODE_FILL = 1 };

struct LaunchCfg {
    const void* fn;      // kernel instance
    int warps_per_block;
    int grid;
    int smem_bytes;      // per block
};

// Queries that share one persistent launch.  A launch has one frame size and
// one block size for all its warps, so a query with large frames (a deep motif)
// would lower the occupancy of every other query of the launch; queries whose
// own launch shape allows the same resident blocks per SM go together instead.
struct LaunchGroup {
    int first, count;    // positions in the grouped order
    int warp_smem;       // frame bytes per warp (largest of the group)
    int warps;           // warps per block
    unsigned feat;       // union of the group's plan features
    int grid;            // blocks
};
// Groups of nq plans for `mode`, query j having nch[j] root chunks; order[i] =
// index of the query at grouped position i.
std::vector<LaunchGroup> occupancy_groups(const tm_graph* g, Mode mode, const Plan* const* plans,
                                          const uint64_t* nch, int nq, int* order);

// Launch the persistent search over nq queries (qdev already on the device).
// Ctrl (incl. total_chunks) and qdev must already be initialised on the stream.
// `feat` selects the kernel instance: the union of plan_features() over the
// nq queries (an instance without a feature a query needs gives wrong counts).
tm_status launch_search(const tm_graph* g, Mode mode, const QueryDev* qdev_dev, int nq,
                        int max_warp_smem, int warps_per_block, unsigned feat,
                        const Scratch* s, cudaStream_t st, int grid_override = 0, bool stats = false);

// Whether a frame's windows, none longer than that, may need FEAT_LONG.
bool long_frames(uint64_t longest_window);
int launch_blocks(const tm_graph* g, const LaunchCfg& c, uint64_t total_chunks);
int effective_chunk(const tm_graph* g, const Plan& p, uint64_t roots);
uint64_t n_chunks(uint64_t roots, int chunk_roots);
LaunchCfg search_launch_cfg(const tm_graph* g, Mode mode, int max_warp_smem, int warps_per_block, unsigned feat,
                            bool stats = false);

// ------------------------------------------------------------- primitives

// Exclusive prefix sum of n uint64 values (in place allowed).  Needs
// scan_temp_bytes(n) bytes of device temp.
size_t scan_temp_bytes(uint64_t n);
tm_status exclusive_scan_u64(const unsigned long long* in, unsigned long long* out, uint64_t n,
                             void* temp, cudaStream_t st);

// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of the key
// (K: uint32_t or uint64_t).  keys_in / vals_in are read only (vals_in may be null:
// the values are then 0 .. n-1); keys[] and vals[] are two buffers each, of which
// number *which holds the result.
template <typename K>
tm_status radix_sort_pairs(const K* keys_in, const uint32_t* vals_in, K* const keys[2], uint32_t* const vals[2],
                           uint64_t n, int bits, void* temp, size_t temp_bytes, cudaStream_t st, int* which);
size_t radix_temp_bytes(uint64_t n);

}  // namespace tmg
