// Persistent warp-cooperative temporal motif search (sm_103a).
//
// The search is the chronological depth-first search of the paper's
// Algorithm 1 (Section 2.2), rooted at every edge, with the per-level plan of
// Section 5.1.2 deciding where candidates come from and which mapped nodes a
// new node must differ from.  The GPU organisation is our own:
//
//  * Roots are filtered before anything else of them is read, since most edges
//    have no later edge in the window at one of their nodes: one byte per list
//    (its successor gap, rounded down) decides, four lists of a root in one word, four
//    roots per lane, 128 per step.  The survivors are buffered and taken 32 at a
//    time, so the searches that start a window run on full warps.  (10M-edge
//    power-law graph, 1 h windows: the cycles' roots fall to the tenth whose
//    source is answered within the window.)  With the 8-byte successor words
//    read instead, 64 roots per step, and every warp claiming for itself: 1/61 of
//    10M edges 107 -> 83 us a call, labelled 5-path on 20M edges 450 -> 348 us.
//  * A warp owns a stack of FRAMES, one per motif edge i >= 1.  Frame i holds
//    up to 48 (count; 40 with look-ahead) or 64 (fill) partial matches of i edges ("parents"), each with its candidate
//    window for edge i: the entries of one time-ordered adjacency list with
//    t in (t_prev, min(t_root + delta, t_prev + gap_{i-1})], located by a
//    binary search for the lower end and a galloping search for the upper end
//    (the cached candidate range of Section 5.1.1 is the window itself).  When
//    the list belongs to an endpoint of the edge just bound, the lower end is
//    the graph's successor word for that edge instead, read together with the
//    candidate; its time gap proves most windows empty without further loads.
//  * The windows of a frame are flattened: lane j of a 32-wide step takes the
//    j-th remaining candidate across all parents, so lanes stay busy even when
//    every individual window is short.  Where each window starts in the flattened
//    order is computed once, when the frame is begun; a step then finds its lanes'
//    parents with two ballots and one reduction.  Survivors of a step (structure, label
//    and injectivity checks) are compacted with __ballot_sync into the child
//    frame, which is drained once it holds cap - 32 parents (16 in count
//    frames of 48, 32 in fill frames of 64) or its parent frame is exhausted.
//    Processing frames in order keeps the emitted matches in
//    lexicographic order of edge ids (used by enumeration).
//  * The last motif edge is never expanded.  Counting it, when it extends by a
//    new node, is a loop of its own that reads only the neighbour column and lets each lane
//    count; other last edges count __popc(ballot) of the survivors.  Per-root / per-chunk
//    counts take one atomic per group of lanes with one parent or root.
//  * Load balance (sub-tree-level parallelism, Section 5.2): root edges are
//    claimed in chunks from an atomic cursor; when warps sit idle, a warp at a
//    shallow level donates the upper half of its remaining candidate range to
//    a device task queue (count mode only), and idle warps pop those tasks.
//    The launch ends when all claimed chunks and all donated tasks are reported
//    done.  A launch has no more warps than chunks, and one idle warp per block polls
//    for work: 5,472 warps going through the same lines cost a small launch 50 us.
//    Every device-side wait is bounded by a global-timer deadline.
//    All of it together, against one 32-root batch per claim, prefix sums rebuilt in every step
//    and every warp polling: 20k-edge 3-cycle 192 -> 110 us per call, 1/61 of
//    10M edges 202 -> 109 us, four queries' counts and rows on 10M edges
//    4.76 -> 2.96 ms, 4-edge path over 15 h windows 47 -> 40 ms.
//  * Look-ahead on chords (our addition): when an edge binds the last node of
//    a later motif edge whose node pair no earlier motif edge joins, some
//    graph edge must join their images later in the root's window; the
//    pair-ordered out-list answers that with two searches, and partial
//    matches without one are dropped before their subtrees are searched.
//    Before those searches, candidates go through a signature of the chord's
//    list window, one per parent.
//  * Enumeration is two launches of this kernel: a count launch leaves
//    per-chunk match counts, a device scan turns them into row offsets,
//    list_chunks_kernel lists the chunks holding a match below the cap, and a fill
//    launch searches only the listed chunks again, each writing its rows in
//    lexicographic order from its offset.
//  * The kernel is instantiated per mode (count, enumeration fill), with or
//    without work counters, and per feature set (anti-edges, look-ahead, last
//    edges counted as pairs, frames that may begin in parts), so a plain motif runs code holding none: registers
//    and instruction cache are short (the pair code alone, in the plain instance,
//    made a 4-edge path 22% slower).  The plain instance was 95 KB of code and warps
//    waited for instructions a third of the time on 4-cycles: one call site for each large part and
//    no unrolling of short loops made it 81 KB, the 64-query batch 11.3 -> 10.2 ms and four
//    queries' counts and rows 1.70 -> 1.53 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <unordered_map>

#include "tm_internal.cuh"

namespace tmg {

namespace {

constexpr unsigned FULL = 0xffffffffu;
// read the next level's successor words together with each candidate
constexpr bool PREFETCH = true;
constexpr uint32_t INLIST = 0x80000000u;    // window in an in-list
constexpr uint32_t PAIRLIST = 0x40000000u;  // window in the (neighbour, time)-ordered out-list
constexpr uint32_t POSMASK = 0x3FFFFFFFu;
constexpr unsigned long long NO_CHUNK = ~0ull;
constexpr uint32_t NEVER = 0xFFFFFFFFu;      // prefix entry past a frame's last parent
constexpr uint32_t SPAN_FAR = 0xFFFFFFFFu;   // frame window end: recompute from the root
// Candidates a frame is searched through at a time: positions in its flattened order, a step's overshoot
// included, stay below LATER.  One window always fits (n_edges < 2^30 - 1).
constexpr uint32_t LATER = 0x80000000u;      // prefix entry: a window not begun yet, the other bits its length
#ifndef TMG_FRAME_MAX        // (the tests build one with small parts, for graphs of fewer edges than that)
#define TMG_FRAME_MAX (LATER - 256u)
#endif
constexpr uint32_t FRAME_MAX = TMG_FRAME_MAX;
constexpr uint32_t MORE = 0x100u;            // in a frame's number of parents: it has windows not begun yet
constexpr uint32_t PAIRS_MAX = 256;          // longest window whose last two edges are counted as pairs
constexpr uint32_t PAIR_MIN_DEG = 1024;     // closing lookups on shorter lists scan the time window
constexpr uint32_t PAIR_MIN_WINDOW = 768;   // ... and so do windows shorter than this
#ifndef TMG_WAIT_NS          // (a shorter one in a test's build)
#define TMG_WAIT_NS (20ull * 1000 * 1000 * 1000)
#endif
constexpr uint64_t WAIT_NS = TMG_WAIT_NS;                     // idle-wait deadline
constexpr uint64_t READY_NS = 2ull * 1000 * 1000 * 1000;      // publish-wait deadline

__device__ __forceinline__ int64_t sat_add(int64_t a, int64_t b) {
    return (b > 0 && a > INT64_MAX - b) ? INT64_MAX : a + b;
}

__device__ __forceinline__ uint64_t now_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// first index in [lo, hi) with t[idx] > x
__device__ __forceinline__ uint32_t upper_bound_t(const int64_t* __restrict__ t, uint32_t lo, uint32_t hi, int64_t x) {
#pragma unroll 1
    while (lo < hi) {
        uint32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(t + mid) <= x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// first index in [beg, hi) with t[idx] > lim, searching outward from beg
__device__ __forceinline__ uint32_t gallop_end(const int64_t* __restrict__ t, uint32_t beg, uint32_t hi, int64_t lim) {
    uint32_t a = beg, b = hi, step = 1;
#pragma unroll 1
    while (true) {
        uint32_t probe = a + step - 1;
        if (probe >= hi) { b = hi; break; }
        if (__ldg(t + probe) > lim) { b = probe; break; }
        a = probe + 1;
        step <<= 1;
    }
    return upper_bound_t(t, a, b, lim);
}

// End of a time window that starts at beg: the first index in [beg, hi) with
// t[idx] > lim (galloping from beg: O(log of the window length)).
__device__ __forceinline__ uint32_t window_end(const int64_t* __restrict__ t, uint32_t beg, uint32_t hi, int64_t lim) {
    return gallop_end(t, beg, hi, lim);
}

__device__ __forceinline__ uint32_t ceil_log2p1(uint32_t x) { return 32 - __clz(x); }  // ceil(log2(x+1))

// first index in [lo, hi) with a[idx] >= x
__device__ __forceinline__ uint32_t lower_bound_i32(const int32_t* __restrict__ a, uint32_t lo, uint32_t hi, int32_t x) {
#pragma unroll 1
    while (lo < hi) {
        uint32_t mid = lo + ((hi - lo) >> 1);
        if (__ldg(a + mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Edges u -> v with time in [t0, t1], counted from u's pair-ordered out-list.
__device__ __forceinline__ uint32_t pair_count(const GraphView& g, int32_t u, int32_t v, int64_t t0, int64_t t1) {
    uint32_t u0 = __ldg(g.off[0] + u), u1 = __ldg(g.off[0] + u + 1);
    uint32_t ps = lower_bound_i32(g.pnbr, u0, u1, v);
    uint32_t pe = lower_bound_i32(g.pnbr, ps, u1, v + 1);
    if (ps == pe) return 0u;
    uint32_t a = upper_bound_t(g.pt, ps, pe, t0 - 1);   // first time >= t0 (t0 >= 0)
    uint32_t b = upper_bound_t(g.pt, a, pe, t1);
    return b - a;
}

// Whether some edge u -> v has a time in (t0, t1]: u's pair-ordered out-list
// holds the u -> v edges as one time-ordered run (binary search on the
// neighbour, then a galloping search past t0 inside the run).
__device__ __forceinline__ bool pair_after(const GraphView& g, int32_t u, int32_t v, int64_t t0, int64_t t1) {
    if (t1 <= t0) return false;
    const uint32_t u1 = __ldg(g.off[0] + u + 1);
    uint32_t a = lower_bound_i32(g.pnbr, __ldg(g.off[0] + u), u1, v), hi = u1, step = 1;
#pragma unroll 1
    while (true) {
        const uint32_t probe = a + step - 1;
        if (probe >= u1) break;                       // hi stays at the list end
        if (__ldg(g.pnbr + probe) != v || __ldg(g.pt + probe) > t0) { hi = probe; break; }
        a = probe + 1;
        step <<= 1;
    }
#pragma unroll 1
    while (a < hi) {
        const uint32_t mid = a + ((hi - a) >> 1);
        if (__ldg(g.pnbr + mid) == v && __ldg(g.pt + mid) <= t0) a = mid + 1; else hi = mid;
    }
    return a < u1 && __ldg(g.pnbr + a) == v && __ldg(g.pt + a) <= t1;
}

// ------------------------------------------------------------ frame access

// The block's dynamic shared memory: each warp's frames, back to back.
extern __shared__ __align__(16) char smem[];

template <int CAP>
struct FrameT {
    using L = FrameLayout<CAP>;
    uint32_t o;      // byte offset in smem
    __device__ int64_t& tprev(int s) const { return ((int64_t*)(smem + o + L::TPREV))[s]; }
    // window end t_root + delta, as its distance from tprev (SPAN_FAR: too far to hold)
    __device__ uint32_t& tspan(int s) const { return ((uint32_t*)(smem + o + L::TEND))[s]; }
    __device__ uint32_t& beg(int s) const { return ((uint32_t*)(smem + o + L::BEG))[s]; }
    __device__ uint32_t& len(int s) const { return ((uint32_t*)(smem + o + L::LEN))[s]; }
    // once begin_frame has run, the same row holds where each window starts in the flattened order
    __device__ uint32_t& pre(int s) const { return ((uint32_t*)(smem + o + L::LEN))[s]; }
    __device__ uint2& pre2(int lane) const { return ((uint2*)(smem + o + L::LEN))[lane]; }
    __device__ uint32_t& root(int s) const { return ((uint32_t*)(smem + o + L::ROOT))[s]; }
    __device__ int32_t& node(int j, int s) const { return ((int32_t*)(smem + o + L::NODE))[j * CAP + s]; }
    // eids follow the nb node rows
    __device__ int32_t& eid(int nb, int j, int s) const { return ((int32_t*)(smem + o + L::NODE))[(nb + j) * CAP + s]; }
    // anti-edge attached-edge times, at byte offset `row_off` of the frame
    __device__ int64_t& anti_t(int row_off, int a, int s) const { return ((int64_t*)(smem + o + row_off))[a * CAP + s]; }
};

// ------------------------------------------------------------ per-warp state

// work counters, laid out like tm_work
constexpr int W_ROOTS = 0, W_NODES = 1, W_ENTRIES = 1 + TM_MAX_EDGES, W_PROBE = 1 + 2 * TM_MAX_EDGES,
              W_MATCH = 2 + 2 * TM_MAX_EDGES, W_LEN = 3 + 2 * TM_MAX_EDGES;

struct Acc {             // per-warp accumulators for the current query
    unsigned long long total;      // per lane
    unsigned long long w[W_LEN];   // stats launches; lane-0 values except W_PROBE (per lane)
};

// What the warps of a block share.  One global atomic claims chunks for all of them, and one
// reports what they finished: returning atomics on one address take 1.9 ns each
// on a GB300 however they are spread, so 5,472 warps claiming, reporting and going
// idle one by one took 56 us without any search (200k edges, a query without a single window;
// 10M edges: 103 us); per block they take 31 (58) us.
struct Block {
    int lock;                     // guards cn, left, grow, claimed_at, ended
    int ended;                    // no chunks are left to claim
    unsigned long long cn;        // claimed chunks nobody took yet: cn .. cn + left
    uint32_t left, grow;
    uint32_t claimed_at;          // clock at the last claim
    int poller, finished;         // see wait_for_work()
    unsigned unreported;          // finished chunks not added to done_chunks yet
    int arrived;                  // warps that have left the search, of a launch of one query,
    unsigned long long total;     // ... and their matches
};

template <int MODE, bool STATS, int FEAT>
struct Search {
    static constexpr bool ANTI = (FEAT & FEAT_ANTI) != 0;   // anti-edge checks compiled in
    static constexpr bool LOOK = (FEAT & FEAT_LOOK) != 0;   // look-ahead checks compiled in
    static constexpr bool FILTER = LOOK && !STATS;          // ... with their candidate filter
    static constexpr bool PAIRS = (FEAT & FEAT_PAIRS) != 0;   // last two edges as pairs
    static constexpr bool LONG = (FEAT & FEAT_LONG) != 0;     // frames may begin in parts
    static constexpr int CAP = MODE == MODE_FILL ? FCAP_FILL : LOOK ? FCAP_LOOK : FCAP_COUNT;   // parents per frame
    static constexpr uint32_t DESCEND = CAP - 32;   // a child frame this full is drained next
    using Frame = FrameT<CAP>;
    const GraphView& g;
    const QueryDev* __restrict__ qs;
    Ctrl* ctrl;
    Task* tasks;
    uint8_t* ready;
    uint64_t task_cap;
    uint32_t wbase;           // this warp's shared block (byte offset in smem)
    int lane;
    // current query
    int qi;
    const QueryDev* q;
    int k;
    // cursors of the suspended levels: lane j holds level j's next candidate and total
    uint32_t myOff, myT, myNp, myPend;
    uint32_t np1;             // parents in frame 1 (warp-uniform)
    uint32_t nbuf;            // roots in the root buffer (warp-uniform)
    Acc acc;
    // enumerate fill
    unsigned long long out_base, out_local;
    unsigned polls;           // donation checks (warp-uniform)
    uint32_t claimed;         // root chunks this warp has taken (warp-uniform)
    Block* blk;

    __device__ Search(const GraphView& g_, const QueryDev* qs_, Ctrl* c, Task* t, uint8_t* r, uint64_t cap, uint32_t wb,
                      Block* b)
        : g(g_), qs(qs_), ctrl(c), tasks(t), ready(r), task_cap(cap), wbase(wb), blk(b) {
        lane = threadIdx.x & 31;
        qi = -1; q = nullptr; k = 0;
        myOff = myT = myNp = myPend = 0;
        np1 = nbuf = 0;
        acc.total = 0;
        if (STATS) for (int i = 0; i < W_LEN; ++i) acc.w[i] = 0;
        out_base = out_local = 0;
        polls = 0;
        claimed = 0;
    }

    // The window end t_root + delta of entry s of frame f (4 bytes per entry
    // instead of 8: rebuilt from the root edge's time when too far from tprev).
    __device__ int64_t tend_of(Frame f, int s) const {
        const uint32_t sp = f.tspan(s);
        return sp != SPAN_FAR ? f.tprev(s) + (int64_t)sp : sat_add(__ldg(g.t + f.root(s)), q->plan.delta);
    }
    __device__ static void set_tend(Frame f, int s, int64_t tprev, int64_t tend) {
        const uint64_t d = (uint64_t)(tend - tprev);   // tprev <= tend
        f.tspan(s) = d < (uint64_t)SPAN_FAR ? (uint32_t)d : SPAN_FAR;
    }

    __device__ Frame frame(int i) const {
        return Frame{wbase + (uint32_t)__ldg(MODE == MODE_FILL ? &q->plan.lv[i].frame_off_fill : &q->plan.lv[i].frame_off)};
    }

    __device__ int anti_off(int i) const {
        return MODE == MODE_FILL ? q->plan.lv[i].anti_row_off_fill : q->plan.lv[i].anti_row_off;
    }

    __device__ uint32_t hot(int i) const { return __ldg(&q->plan.lv[i].hot); }

    // Anti-edges in `mask` (Section 2.1): true when none of them has an edge in
    // its window.  Slots of the candidate's partial match are the parent's
    // slots [0, nb) plus n0, n1; times: edge `lvl` is the candidate (ct), edge
    // lvl-1 is the parent's tprev, older attached edges come from anti rows.
    __device__ bool anti_clear(unsigned mask, int lvl, Frame pf, int ps, int nb, int32_t n0, int32_t n1, int64_t ct,
                               int64_t tprev, int prow) const {
        const Plan& pl = q->plan;
        auto slot = [&](int s) -> int32_t { return s < nb ? pf.node(s, ps) : (s == nb ? n0 : n1); };
        for (int a = 0; a < pl.n_anti; ++a) {
            if (!(mask & (1u << a))) continue;
            const AntiPlan& ap = pl.anti[a];
            int64_t ti = ap.edge == lvl ? ct : (ap.edge == lvl - 1 ? tprev : pf.anti_t(prow, a, ps));
            uint32_t c = pair_count(g, slot(ap.xs), slot(ap.ys), ti, sat_add(ti, ap.delta));
            if (c > (uint32_t)ap.same_pair) return false;
        }
        return true;
    }

    // Look-ahead of level `lp` for a partial match whose slots are the
    // parent's [0, nb) plus n0, n1, just extended by an edge at time ct:
    // false when a later motif edge between bound nodes has no graph edge left
    // in (ct, tend].
    __device__ bool look_ok(const LevelPlan& lp, Frame pf, int ps, int nb, int32_t n0, int32_t n1, int64_t ct,
                            int64_t tend) const {
        auto slot = [&](int s) -> int32_t { return s < nb ? pf.node(s, ps) : (s == nb ? n0 : n1); };
        for (int l = 0; l < lp.n_look; ++l)
            if (!pair_after(g, slot(lp.look_u[l]), slot(lp.look_v[l]), ct, tend)) return false;
        return true;
    }

    __device__ void flush() {
        if (q == nullptr) return;
        for (int d = 16; d > 0; d >>= 1) acc.total += __shfl_down_sync(FULL, acc.total, d);
        if (lane == 0 && acc.total) atomicAdd(q->total, acc.total);
        if (STATS) {
            for (int i = 0; i < W_LEN; ++i) {
                unsigned long long v = acc.w[i];
                for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(FULL, v, d);
                if (lane == 0 && v && q->work) atomicAdd(q->work + i, v);
                acc.w[i] = 0;
            }
        }
        acc.total = 0;
    }

    __device__ void use_query(int j) {
        if (j == qi) return;
        flush();
        qi = j;
        q = qs + j;
        k = q->plan.k;
    }

    // Window for motif edge `lv_i` of a (child) partial match whose slots are
    // parent slots [0, nb) of frame `pf` at index `ps`, plus new nodes n0, n1
    // at slots nb, nb+1; prev_e is the edge just bound (time tprev).  The
    // window's lower end comes from the successor index when the list belongs
    // to an endpoint of prev_e, else from a binary search; the upper end from
    // a galloping search.  Returns len; beg gets bit 31 for in-lists.
    // The edge just bound sits at position cpos of list cdir (0 out-list, 1 in-list,
    // 2 the edge list itself, 3 a pair-ordered list); prev_e is its edge id when
    // already loaded, else -1.  Successor-index lookups read the position-indexed
    // copy when it covers the continuation, else the edge-indexed one.
    __device__ uint2 successor(int nx, int cdir, uint32_t cpos, int32_t prev_e) const {
        if (cdir == 0 && nx == NX_OUT_SRC) return __ldg(g.pnx[0] + cpos);
        if (cdir == 0 && nx == NX_OUT_DST) return __ldg(g.pnx[1] + cpos);
        if (cdir == 1 && nx == NX_IN_DST) return __ldg(g.pnx[2] + cpos);
        if (cdir == 1 && nx == NX_IN_SRC) return __ldg(g.pnx[3] + cpos);
        return __ldg(g.nxt[nx] + 2u * (uint32_t)edge_at(cdir, cpos, prev_e));
    }
    // True when successor() is one load (no edge id needed first).
    __device__ static bool successor_direct(int nx, int cdir) {
        if (cdir == 2) return true;
        if (cdir == 0) return nx == NX_OUT_SRC || nx == NX_OUT_DST;
        if (cdir == 1) return nx == NX_IN_DST || nx == NX_IN_SRC;
        return false;
    }
    // Successor words of the lists level `ln` draws its window from, after a
    // candidate edge at position cpos of list cdir, read ahead together with
    // the candidate: only those that take one load.  y == 0 means "not read".
    __device__ void next_words(uint32_t hn, int cdir, uint32_t cpos, uint2& wa, uint2& wb) const {
        wa = make_uint2(0u, 0u);
        wb = make_uint2(0u, 0u);
        const int na = Hot::nx_a(hn), nb = Hot::nx_b(hn);
        if (na >= 0 && successor_direct(na, cdir)) wa = successor(na, cdir, cpos, -1);
        if (Hot::kind(hn) == CLOSE && nb >= 0 && successor_direct(nb, cdir)) wb = successor(nb, cdir, cpos, -1);
    }
    // True when a list whose successor word is w has no entry in (tprev, lim].
    __device__ static bool word_shows_empty(uint2 w, uint64_t span) {
        return w.y == SUCC_END || (uint64_t)w.y > span;
    }
    __device__ int32_t edge_at(int cdir, uint32_t cpos, int32_t prev_e) const {
        if (prev_e >= 0) return prev_e;
        if (cdir == 0 || cdir == 1) return __ldg(g.aeid[cdir] + cpos);
        if (cdir == 3) return __ldg(g.peid + cpos);
        return (int32_t)cpos;
    }

    __device__ uint32_t locate(int lv_i, uint32_t h, Frame pf, int ps, int nb, int32_t n0, int32_t n1, int32_t prev_e,
                               int cdir, uint32_t cpos, int64_t tprev, int64_t tend, uint32_t& beg_out,
                               uint2 wa, uint2 wb) {
        auto slot = [&](int s) -> int32_t { return s < nb ? pf.node(s, ps) : (s == nb ? n0 : n1); };
        int64_t lim = tend;
        if (h & Hot::GAP) lim = min(tend, sat_add(tprev, q->plan.lv[lv_i].gap));
        beg_out = 0;
        if (!STATS && lim <= tprev) return 0;
        const uint64_t span = (uint64_t)(lim - tprev);
        // words read ahead: an empty list empties the window (a closing
        // window is drawn from either of two lists)
        if (!STATS && (word_shows_empty(wa, span) || word_shows_empty(wb, span))) return 0;
        const int64_t* tarr;
        uint32_t b, hi, flag = 0, in = 0;
        const int kind = Hot::kind(h);
        if (kind == FREE) {
            tarr = g.t;
            hi = (uint32_t)g.m;
            b = gallop_end(tarr, (uint32_t)edge_at(cdir, cpos, prev_e) + 1u, hi, tprev);
            if (STATS) acc.w[W_PROBE] += ceil_log2p1(hi);
        } else {
            int dir, nx;
            uint32_t lo;
            if (kind == CLOSE) {
                // the shorter of out(phi(x_i)) and in(phi(y_i))
                int32_t u = slot(Hot::a(h)), w = slot(Hot::b(h));
                uint32_t u0 = __ldg(g.off[0] + u), u1 = __ldg(g.off[0] + u + 1);
                uint32_t w0 = __ldg(g.off[1] + w), w1 = __ldg(g.off[1] + w + 1);
                if (u1 - u0 <= w1 - w0) { dir = 0; lo = u0; hi = u1; nx = Hot::nx_a(h); }
                else { dir = 1; lo = w0; hi = w1; nx = Hot::nx_b(h); }
                if (!STATS && hi - lo >= PAIR_MIN_DEG) {
                    // a long list: if its time window is long too, take the u -> w
                    // edges straight from u's pair-ordered out-list instead of
                    // scanning the window for one neighbour
                    const int64_t* ta = g.at[dir];
                    uint32_t b0;
                    if (nx >= 0) {
                        const uint2 pw = dir ? wb : wa;
                        const uint2 w = pw.y ? pw : successor(nx, cdir, cpos, prev_e);
                        if (word_shows_empty(w, span)) return 0;
                        b0 = w.x;
                    } else {
                        b0 = upper_bound_t(ta, lo, hi, tprev);
                    }
                    uint32_t e0 = (b0 < hi) ? window_end(ta, b0, hi, lim) : b0;
                    if (e0 - b0 < PAIR_MIN_WINDOW) {
                        beg_out = b0 | (dir ? INLIST : 0u);
                        return e0 - b0;
                    }
                    uint32_t ps = lower_bound_i32(g.pnbr, u0, u1, w);
                    uint32_t pe = lower_bound_i32(g.pnbr, ps, u1, w + 1);
                    uint32_t pb = upper_bound_t(g.pt, ps, pe, tprev);
                    uint32_t pz = (pb < pe) ? window_end(g.pt, pb, pe, lim) : pb;
                    beg_out = pb | PAIRLIST;
                    return pz - pb;
                }
            } else {
                dir = kind == EXT_IN ? 1 : 0;
                int32_t v = slot(Hot::a(h));
                nx = Hot::nx_a(h);
                hi = __ldg(g.off[dir] + v + 1);
                lo = (nx >= 0 && !STATS) ? 0u : __ldg(g.off[dir] + v);
            }
            tarr = g.at[dir];
            flag = dir ? INLIST : 0u;
            if (nx >= 0) {
                const uint2 pw = (kind == CLOSE && dir) ? wb : wa;
                const uint2 w = pw.y ? pw : successor(nx, cdir, cpos, prev_e);
                if (!STATS && word_shows_empty(w, span)) return 0;
                b = w.x;
                // the word says that the first entry is in the window: the search for its end starts behind it
                // (64-query batch 9.8 -> 9.5 ms, 4-path over 15 h windows 20.1 -> 19.8)
                in = !STATS && w.y < SUCC_FAR ? 1u : 0u;
            } else {
                b = upper_bound_t(tarr, lo, hi, tprev);
            }
            if (STATS) acc.w[W_PROBE] += ceil_log2p1(hi - lo);
        }
        uint32_t e = (b < hi) ? window_end(tarr, b + in, hi, lim) : b;
        beg_out = b | flag;
        return e - b;
    }

    // Start frame i, which holds np parents: its window lengths become their
    // exclusive prefix (the flattened position each window starts at; entries past
    // np never start), computed once per frame.  Returns the flattened total.  Windows of a frame may add
    // up to more than 32 bits hold (a few dozen roots of a long delta, each followed by a FREE
    // edge, on 100M edges): a frame with one that long begins its first parents only (LONG instances).
    __device__ uint32_t begin_frame(Frame f, uint32_t& np) const {
        if (LONG) {
            bool lng = lane < np && f.len(lane) > FRAME_MAX / CAP;
            if (lane + 32u < np) lng = lng || f.len(lane + 32) > FRAME_MAX / CAP;
            if (__any_sync(FULL, lng)) return begin_part(f, np);
        }
        return begin_row(&f.pre2(0), np);
    }

    // Start as many of frame f's np windows as FRAME_MAX holds, at least one with entries; np becomes the number
    // of parents up to there, with MORE if others are left.  Those keep their lengths, marked LATER, which no
    // flattened position reaches.
    __device__ uint32_t begin_part(Frame f, uint32_t& np) const {
        const uint32_t a = 2u * lane;
        uint2 l = make_uint2(0u, 0u);
        if (a < (uint32_t)CAP) l = f.pre2(lane);
        if (a >= np) l.x = 0u;
        if (a + 1u >= np) l.y = 0u;
        uint32_t inc = min(l.x + l.y, FRAME_MAX + 1u);      // sums saturate there
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, inc, d);
            if (lane >= d) inc = min(inc + u, FRAME_MAX + 1u);
        }
        uint32_t at = __shfl_up_sync(FULL, inc, 1);
        if (lane == 0) at = 0u;
        const uint32_t mid = min(at + l.x, FRAME_MAX + 1u);
        const bool fx = a < np && mid <= FRAME_MAX, fy = a + 1u < np && inc <= FRAME_MAX;
        const uint32_t taken = __popc(__ballot_sync(FULL, fx)) + __popc(__ballot_sync(FULL, fy));
        const uint32_t tot = __reduce_max_sync(FULL, fy ? inc : fx ? mid : 0u);
        if (a < (uint32_t)CAP)
            f.pre2(lane) = make_uint2(fx ? at : a < np ? l.x | LATER : NEVER, fy ? mid : a + 1u < np ? l.y | LATER : NEVER);
        __syncwarp();
        if (taken < np) np = taken | MORE;
        return tot;
    }

    // Start the windows that begin_part() left: the parents before them stay, with empty windows.
    __device__ uint32_t begin_rest(Frame f, uint32_t& np) const {
        uint2 v = make_uint2(NEVER, NEVER);
        if (2 * lane < CAP) v = f.pre2(lane);
        np = __popc(__ballot_sync(FULL, v.x != NEVER)) + __popc(__ballot_sync(FULL, v.y != NEVER));
        if (2 * lane < CAP) f.pre2(lane) = make_uint2(v.x & LATER ? v.x & ~LATER : 0u, v.y & LATER ? v.y & ~LATER : 0u);
        __syncwarp();
        return begin_part(f, np);
    }

    __device__ static bool pair_level(uint32_t h) { return PAIRS && (h & Hot::PAIRS); }

    // Whether a frame, not begun yet, has only windows that count_pairs() takes.
    __device__ bool short_windows(Frame f, uint32_t np) const {
        bool longer = lane < np && f.len(lane) > PAIRS_MAX;
        if (lane + 32u < np) longer = longer || f.len(lane + 32) > PAIRS_MAX;
        return !__any_sync(FULL, longer);
    }

    __device__ uint32_t begin_row(uint2* row, uint32_t np) const {
        const uint32_t a = 2u * lane;
        uint32_t tot = 0;
        uint2 l = make_uint2(0u, 0u);
        if (a < (uint32_t)CAP) l = row[lane];
        if (a >= np) l.x = 0u;
        if (a + 1u >= np) l.y = 0u;
        const uint32_t s = l.x + l.y;
        uint32_t inc = s;
        for (int d = 1; d < 32; d <<= 1) {
            uint32_t u = __shfl_up_sync(FULL, inc, d);
            if (lane >= d) inc += u;
        }
        tot = __shfl_sync(FULL, inc, 31);
        const uint32_t pa = inc - s;
        if (a < (uint32_t)CAP) row[lane] = make_uint2(a < np ? pa : NEVER, a + 1u < np ? pa + l.x : NEVER);
        __syncwarp();
        return tot;
    }

    // Parent whose window holds flattened position x (warp-uniform); empty windows of a
    // begun frame come before all others, so it is the last one starting at or before x.
    __device__ static int parent_of(uint2 pr, uint32_t x) {
        return __popc(__ballot_sync(FULL, pr.x <= x)) + __popc(__ballot_sync(FULL, pr.y <= x)) - 1;
    }

    // This lane's parent for the 32-wide step at off: the parent holding off plus
    // the windows that start in (off, off + lane].  starts: bit j = a window starts at off + j.
    __device__ int lane_parent(uint2 pr, uint32_t off, unsigned& starts) const {
        const int p0 = parent_of(pr, off);
        unsigned mk = 0;
        const uint32_t da = pr.x - off, db = pr.y - off;   // a start at or before off wraps or is 0: masked out
        if (da - 1u < 31u) mk |= 1u << da;
        if (db - 1u < 31u) mk |= 1u << db;
        starts = __reduce_or_sync(FULL, mk);
        return p0 + __popc(starts & ((2u << lane) - 1u));
    }

    // ---------------------------------------------------- candidate filter
    //
    // A level whose look-ahead joins its new node to a bound node x keeps, per
    // parent, a 512-bit signature (two bits per entry) of x's list in (tprev, tend]:
    // a candidate whose two bits are not both set has no such edge.  The filter reads the
    // neighbour column only; what passes is collected in order and goes through step() 32 at
    // a time, so the exact check's dependent searches run on full warps.  Without
    // it every candidate paid those searches (a hub's list: ~20 loads each): the chorded
    // 4-cycle on 100M hub-skewed edges 222 -> 53 ms, with 80 registers 48.  (256 bits and at most 8 list
    // entries per candidate: 49 ms against 42; 512-entry lists: no more.)

    __device__ uint32_t filt(Frame f, int i) const {
        return f.o + (uint32_t)__ldg(MODE == MODE_FILL ? &q->plan.lv[i].filt_off_fill : &q->plan.lv[i].filt_off);
    }
    __device__ static uint32_t& filt_u32(uint32_t area, int row, int s) { return ((uint32_t*)(smem + area + row))[s]; }
    __device__ static uint32_t* filt_sig(uint32_t area, int s) {
        return (uint32_t*)(smem + area + CandidateFilter::SIG) + CandidateFilter::WORDS * s;
    }
    __device__ static uint32_t filt_hash(int32_t x) { return (uint32_t)x * 2654435761u; }   // bits 31-23 and 22-14

    // Window of x's list for the filter of level i, for a partial match as in locate() with a
    // level-i window of clen candidates; 0 when no candidate can pass.  A long list window saturates
    // its signature, and one much longer than the candidates' costs more to read than
    // their searches (32 entries a search): those parents pass everything (beg = NEVER).
    __device__ uint32_t filt_window(int i, Frame pf, int ps, int nb, int32_t n0, int32_t n1, int32_t prev_e, int cdir,
                                    uint32_t cpos, int64_t tprev, int64_t tend, uint32_t clen, uint32_t& beg) const {
        const LevelPlan& lp = q->plan.lv[i];
        const int fx = lp.fx, dir = lp.fdir, nx = lp.fnx;
        const int32_t x = fx < nb ? pf.node(fx, ps) : (fx == nb ? n0 : n1);
        const int64_t* ta = g.at[dir];
        const uint32_t hi = __ldg(g.off[dir] + x + 1);
        uint32_t b;
        if (nx >= 0 && cdir >= 0) {
            const uint2 w = successor(nx, cdir, cpos, prev_e);
            if (word_shows_empty(w, (uint64_t)(tend - tprev))) return 0u;
            b = w.x;
        } else {
            b = upper_bound_t(ta, __ldg(g.off[dir] + x), hi, tprev);
            if (b >= hi || __ldg(ta + b) > tend) return 0u;
        }
        const uint32_t most = 32u * min(clen, 8u);
        const uint32_t e = window_end(ta, b, min(hi, b + most + 1u), tend);
        beg = b;
        if (e - b <= most) return e - b;
        beg = NEVER;
        return 1u;
    }

    // The signatures of frame f's np parents.
    __device__ void build_filter(Frame f, int i, uint32_t np) const {
        const uint32_t area = filt(f, i);
        for (uint32_t s = lane; s < np; s += 32u) {
            const uint32_t v = filt_u32(area, CandidateFilter::BEG, s) == NEVER ? FULL : 0u;
            uint4* sig = (uint4*)filt_sig(area, s);
            sig[0] = sig[1] = sig[2] = sig[3] = make_uint4(v, v, v, v);
        }
        uint2* row = (uint2*)(smem + area + CandidateFilter::LEN);
        const uint32_t tot = begin_row(row, np);
        const uint2 pr = 2 * lane < CAP ? row[lane] : make_uint2(NEVER, NEVER);
        const int32_t* __restrict__ nbr = g.anbr[q->plan.lv[i].fdir];
        for (uint32_t off = 0; off < tot; off += 32u) {
            unsigned starts;
            const int p = lane_parent(pr, off, starts);
            if (off + lane < tot) {
                const uint32_t b = filt_u32(area, CandidateFilter::BEG, p);
                if (b != NEVER) {
                    const uint32_t h = filt_hash(__ldg(nbr + b + (off + lane - filt_u32(area, CandidateFilter::LEN, p))));
                    uint32_t* sig = filt_sig(area, p);
                    atomicOr(sig + (h >> 28), 1u << (h >> 23 & 31u));
                    atomicOr(sig + (h >> 19 & 15u), 1u << (h >> 14 & 31u));
                }
            }
        }
        __syncwarp();
    }

    // Filter candidates [off, off + 64) of frame f's tot; those that pass join the
    // pend pending ones.  Returns their new number.
    __device__ uint32_t filter_step(int i, uint32_t h, Frame f, uint32_t off, uint32_t tot, uint32_t pend) const {
        const uint32_t area = filt(f, i);
        const int32_t* __restrict__ nbr = g.anbr[Hot::kind(h) == EXT_IN ? 1 : 0];
        const uint2 pr = 2 * lane < CAP ? f.pre2(lane) : make_uint2(NEVER, NEVER);
        unsigned starts;
        uint32_t pos[2];
        int32_t x[2];
        int p[2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t idx = off + 32u * j + lane;
            p[j] = lane_parent(pr, off + 32u * j, starts);
            if (idx >= tot) { p[j] = -1; continue; }
            pos[j] = (f.beg(p[j]) & POSMASK) + (idx - f.pre(p[j]));
            x[j] = __ldg(nbr + pos[j]);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            bool pass = p[j] >= 0;
            if (pass) {
                const uint32_t hx = filt_hash(x[j]);
                const uint32_t* sig = filt_sig(area, p[j]);
                pass = (sig[hx >> 28] >> (hx >> 23 & 31u) & sig[hx >> 19 & 15u] >> (hx >> 14 & 31u) & 1u) != 0u;
            }
            const unsigned b = __ballot_sync(FULL, pass);
            if (pass) {
                const uint32_t at = pend + __popc(b & ((1u << lane) - 1u));
                filt_u32(area, CandidateFilter::POS, at) = pos[j];
                ((uint8_t*)(smem + area + CandidateFilter::PAR))[at] = (uint8_t)p[j];
            }
            pend += __popc(b);
        }
        __syncwarp();
        return pend;
    }

    // Take the first 32 of frame f's pend pending candidates: this lane's position, and its
    // parent or -1.  The rest move up.
    __device__ int pop_pending(int i, Frame f, uint32_t pend, uint32_t& pos) const {
        const uint32_t area = filt(f, i);
        uint8_t* par = (uint8_t*)(smem + area + CandidateFilter::PAR);
        uint32_t ps[3];
        int pp[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const uint32_t a = 32u * j + lane;
            ps[j] = filt_u32(area, CandidateFilter::POS, a);
            pp[j] = par[a];
        }
        __syncwarp();
#pragma unroll
        for (int j = 1; j < 3; ++j) {
            filt_u32(area, CandidateFilter::POS, 32 * (j - 1) + lane) = ps[j];
            par[32 * (j - 1) + lane] = (uint8_t)pp[j];
        }
        __syncwarp();
        pos = ps[0];
        return lane < pend ? pp[0] : -1;
    }

    // Emit survivors of the last level (or of the root level when k == 1).
    __device__ void emit(bool ok, uint32_t root, Frame pf, int ps, int nb, int32_t last_eid) {
        unsigned bal = __ballot_sync(FULL, ok);
        if (!bal) return;
        unsigned cnt = __popc(bal);
        if (MODE == MODE_COUNT) {
            if (lane == 0) acc.total += cnt;
            if (STATS && lane == 0) acc.w[W_MATCH] += cnt;
            if (q->per_root && ok) {
                unsigned grp = __match_any_sync(bal, root);
                if (lane == __ffs(grp) - 1) atomicAdd(q->per_root + (root - q->root_begin), (unsigned long long)__popc(grp));
            }
            if (q->chunk_cnt && ok) {
                uint32_t c = (uint32_t)((root - q->root_begin) / (uint32_t)q->plan.tune.chunk_roots);
                unsigned grp = __match_any_sync(bal, c);
                if (lane == __ffs(grp) - 1) atomicAdd(q->chunk_cnt + c, (unsigned long long)__popc(grp));
            }
        } else {
            unsigned rank = __popc(bal & ((1u << lane) - 1u));
            unsigned long long pos = out_base + out_local + rank;
            if (ok && pos < q->cap) {
                int32_t* o = q->match_out + pos * (unsigned long long)k;
                for (int j = 0; j < k - 1; ++j) o[j] = pf.eid(nb, j, ps);
                o[k - 1] = last_eid;
            }
            out_local += cnt;
        }
    }

    // One 32-candidate step of frame f at level i < k - 1 (or of the last level,
    // where survivors are emitted): candidates [off, off + 32) of its tot.  h, hc: packed plans of
    // levels i and i + 1; survivors with a window join child frame c after its cp
    // parents.  On a filtered level the candidates are the first of its pend
    // pending ones.  Returns the child frame's new size.
    __device__ uint32_t step(int i, uint32_t h, uint32_t hc, Frame f, Frame c, uint32_t off, uint32_t tot,
                                          uint32_t cp, uint32_t pend) {
        const int nb = Hot::nb(h), kind = Hot::kind(h);
        uint32_t pos = 0;
        bool act;
        int p;
        if (FILTER && (h & Hot::FILT)) {
            p = pop_pending(i, f, pend, pos);
            act = p >= 0;
            if (!act) p = 0;
        } else {
            const uint2 pr = f.pre2(2 * lane < CAP ? lane : 0);
            unsigned starts;
            const uint32_t idx = off + lane;
            act = idx < tot;
            const int pl_ = lane_parent(2 * lane < CAP ? pr : make_uint2(NEVER, NEVER), off, starts);
            p = act ? pl_ : 0;
            if (act) pos = (f.beg(p) & POSMASK) + (idx - f.pre(p));
        }
        int32_t n0 = -1, n1 = -1, ceid = -1;
        int64_t ct = 0;
        bool ok = act;
        // the candidate's edge id: written by enumeration and read by edge labels;
        // the next level's successor lookup loads it only if it needs it
        const bool need_eid = (MODE == MODE_FILL) || (h & Hot::ELABEL);
        int cdir = 2;
        uint2 wa = make_uint2(0u, 0u), wb = wa;   // next level's successor words, read with the candidate
        if (act) {
            const uint32_t bw = f.beg(p);
            cdir = (bw & PAIRLIST) ? 3 : (kind == FREE ? 2 : ((bw & INLIST) ? 1 : 0));
            if (PREFETCH && !STATS && i < k - 1) next_words(hc, cdir, pos, wa, wb);
            if (bw & PAIRLIST) {
                // closing edge from the pair-ordered list: structure holds by construction
                ct = __ldg(g.pt + pos);
                if (need_eid) ceid = __ldg(g.peid + pos);
            } else if (kind == FREE) {
                ct = __ldg(g.t + pos);
                n0 = __ldg(g.src + pos);
                n1 = __ldg(g.dst + pos);
                ceid = (int32_t)pos;
                ok = n0 != n1;
#pragma unroll 1
                for (int j = 0; j < nb; ++j) {
                    int32_t x = f.node(j, p);
                    ok &= (x != n0) && (x != n1);
                }
                if (h & Hot::NLABEL) {
                    const LevelPlan& lp = q->plan.lv[i];
                    if (lp.nl0 >= 0) ok &= g.nlabel[n0] == (uint8_t)lp.nl0;
                    if (lp.nl1 >= 0) ok &= g.nlabel[n1] == (uint8_t)lp.nl1;
                }
            } else {
                int dir = (bw & INLIST) ? 1 : 0;
                ct = __ldg(g.at[dir] + pos);
                int32_t nbr = __ldg(g.anbr[dir] + pos);
                if (need_eid) ceid = __ldg(g.aeid[dir] + pos);
                if (kind == CLOSE) {
                    ok = nbr == f.node(dir ? Hot::a(h) : Hot::b(h), p);
                } else {
                    n0 = nbr;
#pragma unroll 1
                    for (int j = 0; j < nb; ++j) ok &= f.node(j, p) != nbr;
                    if (h & Hot::NLABEL) ok &= g.nlabel[nbr] == (uint8_t)q->plan.lv[i].nl0;
                }
            }
            if (h & Hot::ELABEL) ok &= g.elabel[ceid] == (uint8_t)q->plan.lv[i].elabel;
            if (ANTI && ok && (h & Hot::ANTI))
                ok = anti_clear(q->plan.lv[i].anti_mask, i, f, p, nb, n0, n1, ct, f.tprev(p), anti_off(i));
            if (LOOK && ok && (h & Hot::LOOK)) ok = look_ok(q->plan.lv[i], f, p, nb, n0, n1, ct, tend_of(f, p));
        }
        uint32_t root = act ? f.root(p) : 0u;
        if (i == k - 1) {
            emit(ok, root, f, p, nb, ceid);
            return 0u;
        }
        // expand survivors into frame i+1
        const int nb_c = Hot::nb(hc);
        uint32_t cbeg = 0, clen = 0, fbeg = 0, flen = 1;
        int64_t tend = 0;
        if (ok) {
            tend = tend_of(f, p);
            clen = locate(i + 1, hc, f, p, nb, n0, n1, ceid, cdir, pos, ct, tend, cbeg, wa, wb);
            if (FILTER && (hc & Hot::FILT) && clen > 0)
                flen = filt_window(i + 1, f, p, nb, n0, n1, ceid, cdir, pos, ct, tend, clen, fbeg);
        }
        if (STATS) {
            unsigned b = __ballot_sync(FULL, ok);
            unsigned long long l = ok ? clen : 0u;
            for (int d = 16; d > 0; d >>= 1) l += __shfl_down_sync(FULL, l, d);
            if (lane == 0) {
                acc.w[W_NODES + (i + 1)] += __popc(b);
                acc.w[W_ENTRIES + (i + 1)] += l;
            }
        }
        bool keep = ok && clen > 0 && flen > 0;
        unsigned kb = __ballot_sync(FULL, keep);
        if (!kb) return cp;
        if (keep) {
            int s = (int)(cp + __popc(kb & ((1u << lane) - 1u)));
#pragma unroll 1
            for (int j = 0; j < nb; ++j) c.node(j, s) = f.node(j, p);
            if (nb_c > nb) c.node(nb, s) = n0;
            if (nb_c > nb + 1) c.node(nb + 1, s) = n1;
            c.tprev(s) = ct;
            set_tend(c, s, ct, tend);
            c.beg(s) = cbeg;
            c.len(s) = clen;
            c.root(s) = root;
            if (FILTER && (hc & Hot::FILT)) {
                filt_u32(filt(c, i + 1), CandidateFilter::BEG, s) = fbeg;
                filt_u32(filt(c, i + 1), CandidateFilter::LEN, s) = flen;
            }
            if (MODE == MODE_FILL) {
                for (int j = 0; j < i; ++j) c.eid(nb_c, j, s) = f.eid(nb, j, p);
                c.eid(nb_c, i, s) = ceid;
            }
            const Plan& pl = q->plan;
            for (int a = 0; ANTI && a < pl.n_anti; ++a) {
                const int e = pl.anti[a].edge;
                if (e == i) c.anti_t(anti_off(i + 1), a, s) = ct;
                else if (e < i) c.anti_t(anti_off(i + 1), a, s) = f.anti_t(anti_off(i), a, p);
            }
        }
        __syncwarp();
        return cp + __popc(kb);
    }

    // Donate the upper half of frame i's remaining candidates [off, tot) as
    // tasks; returns the frame's new total.  np: its parents (shrunk too).
    __device__ uint32_t maybe_donate(int i, Frame f, uint32_t& np, uint32_t off, uint32_t tot) {
        const tm_tuning& tu = q->plan.tune;
        if (i > tu.split_depth || tot - off <= (uint32_t)tu.split_min || (ANTI && q->plan.n_anti)) return tot;
        if ((++polls & 15u) != 1u) return tot;      // look at the idle count every 16th step
        int idle = 0;
        if (lane == 0) idle = *(volatile int*)&ctrl->idle;
        idle = __shfl_sync(FULL, idle, 0);
        if (idle <= 0) return tot;
        uint32_t mid = off + ((tot - off) >> 1);
        mid = (mid + 31u) & ~31u;
        if (mid >= tot || mid <= off) return tot;
        // parent containing mid
        const int p0 = parent_of(2 * lane < CAP ? f.pre2(lane) : make_uint2(NEVER, NEVER), mid);
        const int ntask = (int)(LONG ? np & (MORE - 1u) : np) - p0;
        // a task is one parent's window range: donate only when the tasks carry
        // split_min candidates each on average, else the queue traffic costs
        // more than the work it moves
        if ((tot - mid) < (uint32_t)ntask * (uint32_t)max(tu.split_min, 32)) return tot;
        unsigned long long base = 0;
        if (lane == 0) base = atomicAdd(&ctrl->q_reserve, (unsigned long long)ntask);
        base = __shfl_sync(FULL, base, 0);
        if (base + (unsigned long long)ntask > task_cap) {
            // no room: void the reserved slots that exist and keep the work
            for (int j = lane; j < ntask; j += 32)
                if (base + j < task_cap) *(volatile uint8_t*)&ready[base + j] = 2;
            return tot;
        }
        const int nb = q->plan.lv[i].nb;
        for (int j = lane; j < ntask; j += 32) {
            int p = p0 + j;
            const uint32_t pre = f.pre(p), end = p + 1 < p0 + ntask ? f.pre(p + 1) : tot;
            const uint32_t skip = (p == p0) ? (mid - pre) : 0u;
            Task* t = tasks + base + j;
            t->query = (int16_t)qi;
            t->level = (int16_t)i;
            t->beg = f.beg(p) + skip;
            t->len = end - pre - skip;
            t->tprev = f.tprev(p);
            t->tend = tend_of(f, p);
            t->root = f.root(p);
            for (int s = 0; s < nb; ++s) t->node[s] = f.node(s, p);
        }
        __threadfence();
        for (int j = lane; j < ntask; j += 32) *(volatile uint8_t*)&ready[base + j] = 1;
        __syncwarp();
        if (lane == 0) atomicAdd(&ctrl->donated, (unsigned)ntask);
        np = (LONG ? np & MORE : 0u) | ((uint32_t)p0 + 1u);
        return mid;
    }

    // Of the lanes in v, those after this lane in its window whose entry is later than t and another
    // neighbour than x.  starts: bit j = a window starts at lane j > 0; the lanes are in list order.
    __device__ unsigned later_others(unsigned v, unsigned starts, int64_t t, int32_t x) const {
        const unsigned above = ~((2u << lane) - 1u), next = starts & above;
        unsigned m = v & above & (next ? (next & (0u - next)) - 1u : FULL);
        const int64_t t1 = __shfl_down_sync(FULL, t, 1);
        if (__any_sync(FULL, (m >> lane & 2u) != 0u && t1 == t)) m &= ~__match_any_sync(FULL, (long long)t);
        return m & ~__match_any_sync(FULL, x);
    }

    // The j-th set bit of m (j < popc(m)).
    __device__ static int nth_bit(unsigned m, uint32_t j) {
        int at = 0;
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) {
            const uint32_t low = __popc(m & ((1u << s) - 1u));
            if (j >= low) {
                j -= low;
                m >>= s;
                at += s;
            }
        }
        return at;
    }

    // Write the rows of the pairs (this lane's entry of parent p and edge e, each entry of m), whose first goes
    // to row `at`: 32 rows of the warp's at a time, each lane one.  eo: the edge of the entry a bit of m stands for.
    __device__ void write_pairs(Frame f, int nb, int p, unsigned m, unsigned long long at, int32_t e, int32_t eo) const {
        uint32_t inc = __popc(m);
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, inc, d);
            if (lane >= d) inc += u;
        }
        const uint32_t total = __shfl_sync(FULL, inc, 31);
        for (uint32_t t = 0; t < total; t += 32u) {
            const uint32_t r = min(t + lane, total - 1u);
            int o = 0;                              // the lane whose pair row r is: as many have theirs before it
#pragma unroll
            for (int s = 16; s > 0; s >>= 1)
                if (__shfl_sync(FULL, inc, o + s - 1) <= r) o += s;
            const unsigned mo = __shfl_sync(FULL, m, o);
            const uint32_t j = r - (__shfl_sync(FULL, inc, o) - __popc(mo));
            const unsigned long long pos = __shfl_sync(FULL, at, o) + j;
            const int po = __shfl_sync(FULL, p, o);
            const int32_t ea = __shfl_sync(FULL, e, o), eb = __shfl_sync(FULL, eo, nth_bit(mo, j));
            if (t + lane < total && pos < q->cap) {
                int32_t* row = q->match_out + pos * (unsigned long long)k;
                for (int i = 0; i < k - 2; ++i) row[i] = f.eid(nb, i, po);
                row[k - 2] = ea;
                row[k - 1] = eb;
            }
        }
    }

    // Level k - 2 of a search whose last two edges extend by new nodes from one list (out-stars and
    // the like): the last edge's window is what follows the candidate in its own window, so the
    // pairs are counted (enumeration: written) with ballots, without a frame entry, a window search and another pass
    // per candidate.  A step takes whole windows, as many as fit 32 lanes; a longer window is taken
    // in tiles of 32, each against itself and those after it.  Frames with a window above
    // PAIRS_MAX go the general way, whose subtrees can be donated: tiles cost its square.
    // 8 queries on 200k edges 361 -> 246 us, four queries' counts and rows on 10M edges 2.32 -> 1.87 ms
    // with the count's pairs, 1.73 ms with the rows' too (out-star fill 726 -> 538 us).
    __device__ void pairs_of(uint32_t h, Frame f, uint32_t tot) {
        const int nb = Hot::nb(h), dir = Hot::kind(h) == EXT_IN ? 1 : 0;
        const int32_t* __restrict__ nbr = g.anbr[dir];
        const int64_t* __restrict__ ta = g.at[dir];
        const uint2 pr = 2 * lane < CAP ? f.pre2(lane) : make_uint2(NEVER, NEVER);
        const bool attrib = MODE == MODE_COUNT && (q->per_root || q->chunk_cnt);
        // an entry of parent p's window: false when its neighbour is bound already
        auto entry = [&](bool act, int p, uint32_t pos, int32_t& x, int64_t& t, int32_t& e) -> bool {
            x = -1;
            t = 0;
            e = 0;
            if (!act) return false;
            x = __ldg(nbr + pos);
            t = __ldg(ta + pos);
            if (MODE == MODE_FILL) e = __ldg(g.aeid[dir] + pos);
            bool ok = true;
#pragma unroll 1
            for (int j = 0; j < nb; ++j) ok &= f.node(j, p) != x;
            return ok;
        };
        // a tile's entries [o, o + 32) of a window at b that come after this lane's (t, x) in an earlier tile
        auto after = [&](int p, uint32_t b, uint32_t o, uint32_t len, int64_t t, int32_t x, int32_t& eo) -> unsigned {
            int32_t xo;
            int64_t to;
            unsigned v = __ballot_sync(FULL, entry(o + lane < len, p, b + o + lane, xo, to, eo));
            const int64_t t_last = __shfl_sync(FULL, t, 31);
            const bool tie = __shfl_sync(FULL, to, 0) == t_last;
#pragma unroll 2
            for (int j = 0; j < 32; ++j) {
                unsigned same = __shfl_sync(FULL, xo, j) == x ? 1u : 0u;
                if (tie) same |= __shfl_sync(FULL, to, j) == t ? 1u : 0u;
                v &= ~(same << j);
            }
            return v;
        };
        // rows of the lanes' c pairs each start here (and the next ones after them)
        auto place = [&](uint32_t c) -> unsigned long long {
            uint32_t inc = c;
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t u = __shfl_up_sync(FULL, inc, d);
                if (lane >= d) inc += u;
            }
            const unsigned long long at = out_base + out_local + inc - c;
            out_local += __shfl_sync(FULL, inc, 31);
            return at;
        };
        unsigned long long sum = 0;
        uint32_t off = 0;
        while (off < tot) {
            unsigned starts;
            int p = lane_parent(pr, off, starts);
            uint32_t n = min(tot - off, 32u);      // entries of whole windows in this step
            if (off + 32u < tot && !__any_sync(FULL, pr.x == off + 32u || pr.y == off + 32u)) n = starts ? 31u - __clz(starts) : 0u;
            int32_t x, e;
            int64_t t;
            if (n > 0u) {
                if (lane >= n) p = 0;
                const bool ok = entry(lane < n, p, (f.beg(p) & POSMASK) + (off + lane - f.pre(p)), x, t, e);
                unsigned m = later_others(__ballot_sync(FULL, ok), starts, t, x);
                if (!ok) m = 0;
                const uint32_t c = __popc(m);
                if (MODE == MODE_FILL) write_pairs(f, nb, p, m, place(c), e, e);
                sum += c;
                if (attrib) attribute_lanes(f.root(p), c);
                off += n;
                continue;
            }
            // one window, from off to end
            p = __shfl_sync(FULL, p, 0);
            const uint32_t end = p + 1 < CAP ? min(f.pre(p + 1), tot) : tot, b = f.beg(p) & POSMASK, len = end - off;
            for (uint32_t a = 0; a < len; a += 32u) {
                const bool ok = entry(a + lane < len, p, b + a + lane, x, t, e);
                int32_t eo;
                unsigned m = later_others(__ballot_sync(FULL, ok), 0u, t, x);
                uint32_t c = __popc(m);
                for (uint32_t o = a + 32u; o < len; o += 32u) c += __popc(after(p, b, o, len, t, x, eo));
                if (!ok) m = c = 0;
                if (MODE == MODE_FILL) {
                    unsigned long long at = place(c);
                    write_pairs(f, nb, p, m, at, e, e);
                    at += __popc(m);
                    for (uint32_t o = a + 32u; o < len; o += 32u) {
                        unsigned v = after(p, b, o, len, t, x, eo);
                        if (!ok) v = 0;
                        write_pairs(f, nb, p, v, at, e, eo);
                        at += __popc(v);
                    }
                }
                sum += c;
                if (attrib) attribute_lanes(f.root(p), c);
            }
            off = end;
        }
        if (MODE == MODE_COUNT) acc.total += sum;
    }

    // Add each lane's c matches of its root, lanes in root order (per-root or per-chunk counts asked for).
    __device__ void attribute_lanes(uint32_t root, uint32_t c) const {
        if (!q->per_root) {
            // one chunk for all of them, mostly
            const uint32_t cr = (uint32_t)q->plan.tune.chunk_roots, ch = (root - (uint32_t)q->root_begin) / cr;
            const unsigned with = __ballot_sync(FULL, c > 0u);
            if (!with) return;
            const int l = __ffs(with) - 1;
            const uint32_t first = __shfl_sync(FULL, ch, l);
            if (!__any_sync(FULL, c > 0u && ch != first)) {
                const unsigned all = __reduce_add_sync(FULL, c);
                if (lane == l) atomicAdd(q->chunk_cnt + ch, (unsigned long long)all);
                return;
            }
        }
        if (c) attribute(root, c);
    }

    // The last level of a count-mode search whose last edge extends by one new
    // node without labels or anti-edges: a candidate survives when its neighbour is none of the
    // bound nodes, so only the neighbour column is read and lanes count on their own.
    __device__ void count_ext(int i, uint32_t h, Frame f, uint32_t np, uint32_t tot) {
        const int nb = Hot::nb(h);
        const int32_t* __restrict__ nbr = g.anbr[Hot::kind(h) == EXT_IN ? 1 : 0];
        const uint2 pr = 2 * lane < CAP ? f.pre2(lane) : make_uint2(NEVER, NEVER);
        const bool attrib = q->per_root || q->chunk_cnt;
        uint32_t off = 0;
        unsigned long long cnt = 0;
        while (off < tot) {
            tot = maybe_donate(i, f, np, off, tot);
            unsigned starts;
            const uint32_t idx = off + lane;
            const int pl_ = lane_parent(pr, off, starts);
            bool ok = idx < tot;
            const int p = ok ? pl_ : 0;
            if (ok) {
                const uint32_t pos = (f.beg(p) & POSMASK) + (idx - f.pre(p));
                const int32_t x = __ldg(nbr + pos);
                for (int j = 0; j < nb; ++j) ok &= f.node(j, p) != x;
            }
            cnt += ok;
            if (attrib) {
                // lanes of one parent share a root: its first lane adds for all of them
                const unsigned bal = __ballot_sync(FULL, ok);
                if (bal && (lane == 0 || (starts >> lane & 1u))) {
                    const unsigned later = starts & ~((2u << lane) - 1u);     // starts after this lane
                    const unsigned mine = bal & ~((1u << lane) - 1u) & (later ? (later & (0u - later)) - 1u : FULL);
                    if (mine) attribute(f.root(p), (unsigned long long)__popc(mine));
                }
            }
            off += 32;
        }
        acc.total += cnt;
    }

    // Add n matches to their root's and their chunk's counters (where asked for).
    __device__ void attribute(uint32_t root, unsigned long long n) const {
        const uint64_t r = root - q->root_begin;
        if (q->per_root) atomicAdd(q->per_root + r, n);
        if (q->chunk_cnt) atomicAdd(q->chunk_cnt + (uint32_t)r / (uint32_t)q->plan.tune.chunk_roots, n);
    }

    // Drain frame `base`, holding np parents (and everything below it), to completion.
    // whole: the windows end where the search's do (a donated task's is a part of one).
    __device__ void drain(int base, uint32_t np, bool whole) {
        int lvl = base;
        uint32_t h = hot(lvl), hc = lvl + 1 < k ? hot(lvl + 1) : 0u;
        Frame f = frame(lvl), c = lvl + 1 < k ? frame(lvl + 1) : f;
        bool pairs = pair_level(h) && whole && short_windows(f, np);
        const uint32_t all = np;
        uint32_t off = 0, tot = begin_frame(f, np), nch = 0, pend = 0;
        if (FILTER && (h & Hot::FILT)) build_filter(f, lvl, all);
        while (true) {
            if (MODE == MODE_COUNT && !STATS && lvl == k - 1 && Hot::kind(h) <= EXT_IN &&
                !(h & (Hot::ELABEL | Hot::NLABEL | Hot::ANTI))) {
                count_ext(lvl, h, f, np, tot);
                off = tot;
            } else if (pairs) {
                pairs_of(h, f, tot);
                off = tot;
                pairs = false;
            }
            while (off < tot || (FILTER && pend > 0)) {
                if (MODE == MODE_COUNT && off < tot) tot = maybe_donate(lvl, f, np, off, tot);
                if (FILTER && (h & Hot::FILT)) {
                    for (; pend < 32u && off < tot; off += 64u) pend = filter_step(lvl, h, f, off, tot, pend);
                    if (pend == 0) break;
                    nch = step(lvl, h, hc, f, c, 0u, 0u, nch, pend);
                    pend -= min(pend, 32u);
                } else {
                    nch = step(lvl, h, hc, f, c, off, tot, nch, 0u);
                    off += 32;
                }
                if (nch >= DESCEND) break;
            }
            if (nch > 0) {
                // down into the child frame
                if (lane == lvl) { myOff = off; myT = tot; myNp = np; if (FILTER) myPend = pend; }
                ++lvl;
                np = nch;
                nch = 0;
                h = hc;
                f = c;
                if (lvl + 1 < k) { hc = hot(lvl + 1); c = frame(lvl + 1); }
                off = 0;
                pairs = pair_level(h) && short_windows(f, np);
                const uint32_t all = np;
                tot = begin_frame(f, np);
                if (FILTER) {
                    pend = 0;
                    if (h & Hot::FILT) build_filter(f, lvl, all);
                }
                continue;
            }
            if (LONG && (np & MORE)) {
                off = 0;
                tot = begin_rest(f, np);
                continue;
            }
            if (lvl == base) break;
            // back to the suspended parent frame, whose child frame is empty again
            --lvl;
            hc = h;
            c = f;
            h = hot(lvl);
            f = frame(lvl);
            off = __shfl_sync(FULL, myOff, lvl);
            tot = __shfl_sync(FULL, myT, lvl);
            np = __shfl_sync(FULL, myNp, lvl);
            if (FILTER) pend = __shfl_sync(FULL, myPend, lvl);
        }
    }

    __device__ uint32_t& root_buf(uint32_t j) const { return ((uint32_t*)(smem + wbase))[j]; }

    // Scan 128 root edges from rb (rounded down to a multiple of 4) up to re: those whose
    // gap codes leave them a chance of a match join the root buffer, in order.  A
    // root dies when a list the motif draws a later edge from -- any of the out- and
    // in-lists of its two nodes -- has no entry soon enough; a code says so when it is above
    // the query's byte for that list (both below 128: the subtraction borrows from no neighbour).
    __device__ void scan_roots(uint32_t rb, uint32_t re) {
        const uint32_t base = rb & ~3u, r = base + 4u * lane;
        // the columns are padded past the last edge: no read is out of range
        unsigned alive = 0;
        if (STATS) {
            alive = 15u;
            if (lane == 0) acc.w[W_ROOTS] += min(re, base + 128u) - rb;
        } else if (r < re) {
            const Plan& pl = q->plan;
            const uint32_t most = __ldg(&pl.root_codes) | 0x80808080u;
            const uint4 c = __ldg((const uint4*)(g.rcode + r));
            alive = ((most - c.x) & 0x80808080u) == 0x80808080u ? 1u : 0u;
            alive |= ((most - c.y) & 0x80808080u) == 0x80808080u ? 2u : 0u;
            alive |= ((most - c.z) & 0x80808080u) == 0x80808080u ? 4u : 0u;
            alive |= ((most - c.w) & 0x80808080u) == 0x80808080u ? 8u : 0u;
            if (pl.elabel0 >= 0) {
                const uchar4 l = __ldg((const uchar4*)(g.elabel + r));
                const uint8_t want = (uint8_t)pl.elabel0;
                alive &= (l.x == want ? 1u : 0u) | (l.y == want ? 2u : 0u) | (l.z == want ? 4u : 0u) | (l.w == want ? 8u : 0u);
            }
        }
        if (r < rb) alive &= 15u << (rb - r);             // rb - r < 4: only lane 0's word
        if (r + 4u > re) alive &= r < re ? 15u >> (r + 4u - re) : 0u;
        if (!__any_sync(FULL, alive != 0u)) return;
        const unsigned lt = (1u << lane) - 1u;
        uint32_t at = nbuf;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const unsigned b = __ballot_sync(FULL, alive >> j & 1u);
            at += __popc(b & lt);
            nbuf += __popc(b);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (alive >> j & 1u) root_buf(at++) = r + j;
        __syncwarp();
    }

    // Drop the first n of the buffered roots: 32 of them, or all.
    __device__ void pop_roots(uint32_t n) {
        const uint32_t left = nbuf - n;
        for (uint32_t j = lane; j < left; j += 32u) root_buf(j) = root_buf(32u + j);   // each lane its own slots
        __syncwarp();
        nbuf = left;
    }

    // Level 0 of the search for the first up to 32 buffered roots; those with a
    // window join frame 1 after its np1 parents.
    __device__ void root_batch() {
        const Plan& pl = q->plan;
        const uint32_t hc = k > 1 ? hot(1) : 0u;
        const uint32_t n = min(nbuf, 32u);
        {
            bool ok = lane < n;
            const uint32_t r = ok ? root_buf(lane) : 0u;
            pop_roots(n);
            int32_t s = 0, d = 0;
            int64_t tt = 0;
            uint2 wa = make_uint2(0u, 0u), wb = wa;
            if (ok) {
                if (PREFETCH && !STATS && k > 1) next_words(hc, 2, r, wa, wb);
                s = __ldg(g.src + r);
                d = __ldg(g.dst + r);
                tt = __ldg(g.t + r);
                ok = s != d;
                if (pl.elabel0 >= 0) ok &= g.elabel[r] == (uint8_t)pl.elabel0;
                if (pl.nl_x0 >= 0) ok &= g.nlabel[s] == (uint8_t)pl.nl_x0;
                if (pl.nl_y0 >= 0) ok &= g.nlabel[d] == (uint8_t)pl.nl_y0;
                if (ANTI && ok && pl.anti_mask0)
                    ok = anti_clear(pl.anti_mask0, 0, Frame{wbase}, 0, 0, s, d, tt, tt, 0);
                if (LOOK && ok && pl.lv[0].n_look)
                    ok = look_ok(pl.lv[0], Frame{wbase}, 0, 0, s, d, tt, sat_add(tt, pl.delta));
            }
            if (k == 1) {
                emit(ok, r, Frame{wbase}, 0, 0, (int32_t)r);
                return;
            }
            uint32_t cbeg = 0, clen = 0, fbeg = 0, flen = 1;
            int64_t tend = 0;
            if (ok) {
                tend = sat_add(tt, pl.delta);
                clen = locate(1, hc, Frame{wbase}, 0, 0, s, d, (int32_t)r, 2, (uint32_t)r, tt, tend, cbeg, wa, wb);
                if (FILTER && (hc & Hot::FILT) && clen > 0)
                    flen = filt_window(1, Frame{wbase}, 0, 0, s, d, (int32_t)r, 2, (uint32_t)r, tt, tend, clen, fbeg);
            }
            if (STATS) {
                unsigned b = __ballot_sync(FULL, ok);
                unsigned long long l = ok ? clen : 0u;
                for (int dd = 16; dd > 0; dd >>= 1) l += __shfl_down_sync(FULL, l, dd);
                if (lane == 0) {
                    acc.w[W_NODES + 1] += __popc(b);
                    acc.w[W_ENTRIES + 1] += l;
                }
            }
            bool keep = ok && clen > 0 && flen > 0;
            unsigned kb = __ballot_sync(FULL, keep);
            if (kb) {
                Frame c = frame(1);
                if (keep) {
                    int sl = (int)(np1 + __popc(kb & ((1u << lane) - 1u)));
                    c.node(0, sl) = s;
                    c.node(1, sl) = d;
                    c.tprev(sl) = tt;
                    set_tend(c, sl, tt, tend);
                    c.beg(sl) = cbeg;
                    c.len(sl) = clen;
                    c.root(sl) = (uint32_t)r;
                    if (FILTER && (hc & Hot::FILT)) {
                        filt_u32(filt(c, 1), CandidateFilter::BEG, sl) = fbeg;
                        filt_u32(filt(c, 1), CandidateFilter::LEN, sl) = flen;
                    }
                    if (MODE == MODE_FILL) c.eid(2, 0, sl) = (int32_t)r;
                    for (int a = 0; ANTI && a < pl.n_anti; ++a)
                        if (pl.anti[a].edge == 0) c.anti_t(anti_off(1), a, sl) = tt;
                }
                __syncwarp();
                np1 += __popc(kb);
            }
        }
    }

    // Put the donated task in slot h into its level's frame as the only parent; returns the level.
    __device__ int take_task(unsigned long long h) {
        const Task* t = tasks + h;
        const uint32_t ql = __ldcg((const uint32_t*)t);     // query, level
        use_query((int)(ql & 0xFFFFu));
        const int i = (int)(ql >> 16);
        const int nb = Hot::nb(hot(i));
        Frame f = frame(i);
        if (lane == 0) {
            const int64_t tprev = __ldcg(&t->tprev);
            f.tprev(0) = tprev;
            set_tend(f, 0, tprev, __ldcg(&t->tend));
            f.beg(0) = __ldcg(&t->beg);
            f.len(0) = __ldcg(&t->len);
            f.root(0) = __ldcg(&t->root);
        }
        if (lane < nb) f.node(lane, 0) = __ldcg(&t->node[lane]);
        __syncwarp();
        if (FILTER && (hot(i) & Hot::FILT) && lane == 0) {
            // the edge just bound is not in the task: the list is searched for its time
            const int64_t tprev = f.tprev(0);
            uint32_t fbeg = NEVER;
            const uint32_t flen = filt_window(i, f, 0, nb, -1, -1, -1, -1, 0u, tprev, tend_of(f, 0), f.len(0), fbeg);
            filt_u32(filt(f, i), CandidateFilter::BEG, 0) = flen ? fbeg : NEVER;
            filt_u32(filt(f, i), CandidateFilter::LEN, 0) = max(flen, 1u);
        }
        __syncwarp();
        return i;
    }

    // Global chunk c -> query index (chunks of query j are contiguous).
    __device__ int query_of_chunk(uint64_t c, int nq) const {
        int lo = 0, hi = nq;
        while (hi - lo > 1) {
            int mid = (lo + hi) >> 1;
            if (qs[mid].chunk_base <= c) lo = mid; else hi = mid;
        }
        return lo;
    }

    // Pop a published task; returns its slot, or NO_CHUNK when none is ready.
    __device__ unsigned long long try_pop() {
        int got = 0;
        unsigned long long h = 0;
        if (lane == 0) {
            for (int attempt = 0; attempt < 64 && !got; ++attempt) {
                h = *(volatile unsigned long long*)&ctrl->q_head;
                unsigned long long r = *(volatile unsigned long long*)&ctrl->q_reserve;
                if (h >= min(r, (unsigned long long)task_cap)) break;
                if (atomicCAS(&ctrl->q_head, h, h + 1) != h) continue;
                uint64_t t0 = now_ns();
                uint8_t st = 0;
                while ((st = *(volatile uint8_t*)&ready[h]) == 0) {
                    if (now_ns() - t0 > READY_NS) { atomicMax(&ctrl->err, (unsigned)TM_E_TIMEOUT); break; }
                    __nanosleep(64);
                }
                if (st == 1) got = 1;
                else atomicAdd(&ctrl->done_tasks, 1ULL);   // a void slot holds nothing to run
            }
        }
        got = __shfl_sync(FULL, got, 0);
        if (!got) return NO_CHUNK;
        h = __shfl_sync(FULL, h, 0);
        __threadfence();
        return h;
    }

    __device__ bool queue_empty() const {
        unsigned long long r, h;
        asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(r), "=l"(h) : "l"(&ctrl->q_reserve));
        return h >= min(r, (unsigned long long)task_cap);
    }

    // Nothing is left to run and nothing can be donated any more: every chunk's
    // subtree and every reserved task slot is done.  A donor reserves its slots before it
    // reports its own chunk or task done, so done_tasks catching up with q_reserve
    // after that is final.
    __device__ bool all_done(uint64_t total_chunks) const {
        if (*(volatile unsigned long long*)&ctrl->done_chunks < total_chunks) return false;
        const unsigned long long d = *(volatile unsigned long long*)&ctrl->done_tasks;
        __threadfence();
        const unsigned long long r = *(volatile unsigned long long*)&ctrl->q_reserve;
        return d >= min(r, (unsigned long long)task_cap);
    }

    // Wait for a task (true) or the end of the launch (false).  One warp per block
    // polls the control block at a time, and stands for the block in the idle count; the
    // block's other idle warps watch shared memory: thousands of warps polling one line delayed
    // every claim and donation that goes through it.
    __device__ bool wait_for_work(uint64_t total_chunks) {
        int leave = 0;
        if (lane == 0) {
            const uint64_t t0 = now_ns();
            // a poll is two loads of a line that every block polls: sooner ones only delay each other
            unsigned ns = 512;
            bool polling = false;
            while (true) {
                if (*(volatile int*)&blk->finished) { leave = 1; break; }
                if (!polling && atomicCAS(&blk->poller, 0, 1) == 0) {
                    polling = true;
                    atomicAdd(&ctrl->idle, 1);
                }
                if (polling) {
                    const unsigned n = atomicExch(&blk->unreported, 0u);
                    if (n) {
                        __threadfence();
                        atomicAdd(&ctrl->done_chunks, (unsigned long long)n);
                    }
                    if (!queue_empty()) break;
                    if (all_done(total_chunks)) { *(volatile int*)&blk->finished = 1; leave = 1; break; }
                }
                if (now_ns() - t0 > WAIT_NS) { leave = 1; break; }
                __nanosleep(ns);
                if (ns < 2048) ns <<= 1;
            }
            if (polling) {
                // also when the block gives up waiting: donors would go on handing out work nobody waits for
                atomicSub(&ctrl->idle, 1);
                atomicExch(&blk->poller, 0);
            }
        }
        return __shfl_sync(FULL, leave, 0) == 0;
    }

    // Take chunks for this warp from the block's, claiming more for the block when it has none: up to
    // `n` of them from `c` on; 0 when the launch has none left.
    __device__ uint32_t take_chunks(uint64_t total_chunks, unsigned long long& c) {
        uint32_t n = 0;
        if (lane == 0) {
            const uint64_t t0 = now_ns();
            bool mine = true;
            while (atomicCAS(&blk->lock, 0, 1) != 0) {
                if (now_ns() - t0 > READY_NS) { atomicMax(&ctrl->err, (unsigned)TM_E_TIMEOUT); mine = false; break; }
                __nanosleep(32);
            }
            if (mine) {
                __threadfence_block();
                volatile Block* b = blk;
                if (b->left == 0u && !b->ended) {
                    const uint32_t warps = blockDim.x >> 5, now = (uint32_t)clock();
                    const unsigned long long seen = b->cn;    // where the cursor stood at the last claim
                    uint32_t grow = MODE == MODE_FILL ? 1u : claim_size(b->grow, now - b->claimed_at, total_chunks - seen, warps);
                    const unsigned long long at = atomicAdd(&ctrl->next_chunk, (unsigned long long)(grow * warps));
                    b->grow = grow;
                    b->claimed_at = now;
                    if (at >= total_chunks) {
                        b->ended = 1;
                    } else {
                        b->cn = at;
                        b->left = (uint32_t)min((unsigned long long)(grow * warps), total_chunks - at);
                    }
                }
                n = min(b->left, b->grow);
                c = b->cn;
                b->cn = c + n;
                b->left = b->left - n;
                __threadfence_block();
                atomicExch(&blk->lock, 0);
            }
        }
        c = __shfl_sync(FULL, c, 0);
        return __shfl_sync(FULL, n, 0);
    }

    // Find the next frame to drain, in order: roots collected in frame 1 (root
    // chunks are claimed and scanned until it is full enough or must be emptied), then
    // donated tasks, until the launch has no work left.  One loop with one drain,
    // so the search's code exists once per kernel.
    __device__ void run(int nq, uint64_t total_chunks) {
        uint32_t rb = 0, re = 0;                  // roots left of the current chunks
        unsigned long long cn = 0;                // chunks taken and not scanned yet: cn .. cn + left
        uint32_t left = 0;
        bool scanning = true, switching = false, ending = false, ran_task = false;
        while (true) {
            int base = 1;
            uint32_t np = 0;
            bool is_task = false;
            if (scanning) {
                while (np1 < DESCEND) {
                    // once the chunks are scanned, what they left in the root buffer and frame 1
                    // stays for the next ones, except where those belong to another
                    // query or (enumeration) write from another offset
                    const bool empty_out = rb >= re && (MODE == MODE_FILL || switching || ending);
                    if (nbuf >= 32u || (empty_out && nbuf > 0u)) { root_batch(); continue; }
                    if (rb < re) {
                        scan_roots(rb, re);
                        rb = (rb & ~3u) + 128u;
                        continue;
                    }
                    if (empty_out) {
                        if (np1 > 0u) break;
                        if (ending) { scanning = false; break; }
                        switching = false;
                    }
                    if (left == 0u) {
                        left = take_chunks(total_chunks, cn);
                        if (left == 0u) { ending = true; continue; }
                        claimed += left;
                    }
                    if (q == nullptr || cn < q->chunk_base || cn - q->chunk_base >= q->n_chunks) {
                        // nothing of the previous query may be left when switching
                        if (np1 + nbuf > 0u) { switching = true; continue; }
                        use_query(query_of_chunk(cn, nq));
                    }
                    uint64_t lc = cn - q->chunk_base;
                    const uint64_t cr = (uint64_t)q->plan.tune.chunk_roots;
                    uint32_t n = 1;
                    if (MODE == MODE_FILL) {
                        // claim index lc -> the lc-th listed chunk (one holding a match whose
                        // rows start below the cap); past the list's end the rest of this
                        // query is skipped
                        if (lc >= q->chunk_off[q->n_chunks + 1]) {
                            unsigned long long nxt = (qi + 1 < nq) ? qs[qi + 1].chunk_base : total_chunks;
                            if (lane == 0) atomicMax(&ctrl->next_chunk, nxt);
                            left = 0u;
                            continue;
                        }
                        lc = ((const uint32_t*)(q->chunk_off + q->n_chunks + 2))[lc];
                        out_base = q->chunk_off[lc];
                        out_local = 0;
                    } else {
                        n = (uint32_t)min((uint64_t)left, q->n_chunks - lc);
                    }
                    cn += n;
                    left -= n;
                    rb = (uint32_t)(q->root_begin + lc * cr);
                    re = (uint32_t)min(q->root_end, (uint64_t)rb + n * cr);
                }
                np = np1;
                np1 = 0;
                if (np == 0) continue;
            } else {
                if (MODE == MODE_FILL) break;
                report_chunks();
                // a launch of one query that never donates has nothing to wait for; after a task, more of
                // them are likely; before the first, the block's poller looks
                const bool alone = nq == 1 && qs[0].plan.tune.split_depth <= 0;
                if (!alone && !ran_task && !wait_for_work(total_chunks)) break;
                const unsigned long long slot = try_pop();
                ran_task = slot != NO_CHUNK;
                if (!ran_task) {
                    if (alone) break;
                    continue;
                }
                base = take_task(slot);
                np = 1;
                is_task = true;
            }
            drain(base, np, !is_task);
            if (MODE == MODE_COUNT && is_task) {
                __threadfence();      // donations made by this task are reserved before it counts as done
                if (lane == 0) atomicAdd(&ctrl->done_tasks, 1ULL);
            }
        }
        if (STATS || nq != 1) flush(); else leave();
    }

    // The end of a launch of one query: the block's last warp adds the matches of all of them.
    __device__ void leave() {
        for (int d = 16; d > 0; d >>= 1) acc.total += __shfl_down_sync(FULL, acc.total, d);
        if (lane == 0) {
            if (acc.total) atomicAdd(&blk->total, acc.total);
            __threadfence_block();
            if (atomicAdd(&blk->arrived, 1) == (int)(blockDim.x >> 5) - 1) {
                __threadfence_block();
                const unsigned long long all = atomicAdd(&blk->total, 0ULL);
                if (all) atomicAdd(qs[0].total, all);
            }
        }
    }

    // Chunks per warp of a block's next claim.  Chunks without matches are scanned in less than
    // a claim takes, so the size doubles (up to 16) when the last claim of `last` was gone within 16k cycles,
    // about 8 us, and starts over when it was not: roots held by a busy warp wait for it.
    // With `ahead` chunks unclaimed it is at most a quarter of the warp's share.
    __device__ static uint32_t claim_size(uint32_t last, uint32_t cycles, unsigned long long ahead, uint32_t warps) {
        if (cycles > 16384u) return 1u;
        const uint32_t share = (uint32_t)fminf(__fdividef((float)ahead, 4.f * (float)(warps * gridDim.x)), 16.f);
        return max(min(2u * last, share), 1u);
    }

    // Count this warp's chunks as done, once their subtrees (and the slots they donated) are.
    __device__ void report_chunks() {
        if (!claimed) return;
        __threadfence();
        if (lane == 0) atomicAdd(&blk->unreported, claimed);
        claimed = 0;
    }
};

// Registers per thread of an instance.  Plain motifs of up to 4 edges: 64, which is 32 warps per SM (4-path over
// 15 h windows 21.5 ms at 56, 20.0 at 64, 21.3 at 72, 22.1 at 80; at 64 the count still stores 106
// and loads 60 bytes of spills, fills with look-ahead 112 and 106).  Where shared memory allows WIDE_WARPS warps or fewer (5 edges: 28) the registers of the others are
// there to take, and without spills at 80 fewer warps are faster: labelled 5-path on 20M edges
// 344 us at 64, 313 at 72, 265 at 80.  Pairs (8 queries on 200k edges 278, 259, 247 us),
// anti-edges (109, 106, 104) and look-ahead (chorded 4-cycle on 100M edges 52, 49, 48 ms) likewise.
// Plain fills have the widest frames and 64 did best (four queries' counts and rows 1.85 ms, at 72 1.92).
constexpr int search_regs(int mode, bool stats, int feat) {
    feat &= ~(int)FEAT_LONG;
    return stats || feat == 0 || (mode == MODE_FILL && feat != FEAT_PAIRS) ? 64 : 80;
}
constexpr unsigned FEAT_WIDE = 8u;     // a plain count with 80 registers
constexpr int WIDE_WARPS = 28;

template <int MODE, bool STATS, int FEAT>
__global__ void __maxnreg__(search_regs(MODE, STATS, FEAT)) search_kernel(const __grid_constant__ GraphView g,
                                                     const QueryDev* __restrict__ qs, int nq, int warp_smem,
                                                     Ctrl* ctrl, Task* tasks, uint8_t* ready, uint64_t task_cap) {
    __shared__ Block blk;
    if (threadIdx.x == 0) {
        blk = Block{};
        blk.grow = 1;
        blk.claimed_at = (uint32_t)clock();
    }
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    Search<MODE, STATS, FEAT> s(g, qs, ctrl, tasks, ready, task_cap, (uint32_t)(warp * warp_smem), &blk);
    uint64_t chunks = ctrl->total_chunks;
    // a fill of one query ends with its list; of several, each warp finds that out query by query
    if (MODE == MODE_FILL && nq == 1) chunks = min((unsigned long long)chunks, qs[0].chunk_off[qs[0].n_chunks + 1]);
    s.run(nq, chunks);
}

}  // namespace

namespace {

// The chunks of an enumeration that hold a match and whose rows start below
// the cap, from the scanned row offsets: their ids are appended (in no
// particular order) after the offsets and the list length (zeroed by the
// caller), for the fill pass to claim.  A count that gave up (counted->err) has no rows to fill: nothing
// is listed, and the fill ends at once.
__global__ void list_chunks_kernel(unsigned long long* buf, uint64_t nch, uint64_t cap, const Ctrl* __restrict__ counted) {
    if (counted->err) return;
    const unsigned long long* off = buf;
    unsigned long long* n_list = buf + nch + 1;
    uint32_t* list = (uint32_t*)(buf + nch + 2);
    const int lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t base = (uint64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < nch; base += stride) {
        const uint64_t c = base + lane;
        const bool keep = c < nch && off[c + 1] > off[c] && off[c] < cap;
        const unsigned b = __ballot_sync(FULL, keep);
        if (!b) continue;
        unsigned long long at = 0;
        if (lane == 0) at = atomicAdd(n_list, (unsigned long long)__popc(b));
        at = __shfl_sync(FULL, at, 0);
        if (keep) list[at + __popc(b & ((1u << lane) - 1u))] = (uint32_t)c;
    }
}

// Scan and list of a small chunk buffer in one block: a launch each for the scan's two levels and the
// list took 15 us between the passes of a 100 us call.
constexpr int SMALL_THREADS = 1024, SMALL_ITEMS = 4;
constexpr uint64_t SMALL_CHUNKS = 16384;      // four rounds of the block; longer buffers scan faster on many

__global__ void __launch_bounds__(SMALL_THREADS) small_offsets_kernel(unsigned long long* buf, uint32_t nch, uint64_t cap,
                                                                      const Ctrl* __restrict__ counted) {
    __shared__ unsigned long long wsum[SMALL_THREADS / 32];
    __shared__ uint32_t wkeep[SMALL_THREADS / 32];
    uint32_t* list = (uint32_t*)(buf + nch + 2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned long long carry = 0;
    uint32_t listed = 0;
    for (uint32_t base = 0; base <= nch; base += SMALL_THREADS * SMALL_ITEMS) {
        const uint32_t c0 = base + threadIdx.x * SMALL_ITEMS;
        unsigned long long v[SMALL_ITEMS], sum = 0;
#pragma unroll
        for (int j = 0; j < SMALL_ITEMS; ++j) {
            v[j] = c0 + j < nch ? buf[c0 + j] : 0;        // entry nch, past the counts, becomes the total
            sum += v[j];
        }
        unsigned long long inc = sum;
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned long long u = __shfl_up_sync(FULL, inc, d);
            if (lane >= d) inc += u;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        unsigned long long at = carry + inc - sum;
        for (int w = 0; w < SMALL_THREADS / 32; ++w) {
            if (w < warp) at += wsum[w];
            carry += wsum[w];
        }
        uint32_t keep = 0;
#pragma unroll
        for (int j = 0; j < SMALL_ITEMS; ++j) {
            if (c0 + j <= nch) buf[c0 + j] = at;
            if (v[j] > 0 && at < cap) keep |= 1u << j;
            at += v[j];
        }
        uint32_t kin = __popc(keep);
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t u = __shfl_up_sync(FULL, kin, d);
            if (lane >= d) kin += u;
        }
        if (lane == 31) wkeep[warp] = kin;
        __syncthreads();
        uint32_t to = listed + kin - __popc(keep);
        for (int w = 0; w < SMALL_THREADS / 32; ++w) {
            if (w < warp) to += wkeep[w];
            listed += wkeep[w];
        }
#pragma unroll
        for (int j = 0; j < SMALL_ITEMS; ++j)
            if (keep >> j & 1u) list[to++] = c0 + j;
        __syncthreads();
    }
    if (threadIdx.x == 0) buf[nch + 1] = counted->err ? 0u : listed;
}

}  // namespace

tm_status chunk_offsets(unsigned long long* chunk_buf, uint64_t nch, uint64_t cap, const Ctrl* counted, void* scan_tmp,
                        int num_sms, cudaStream_t st) {
    if (nch == 0) return TM_OK;
    if (nch <= SMALL_CHUNKS) {
        small_offsets_kernel<<<1, SMALL_THREADS, 0, st>>>(chunk_buf, (uint32_t)nch, cap, counted);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
        return TM_OK;
    }
    tm_status s = exclusive_scan_u64(chunk_buf, chunk_buf, nch + 1, scan_tmp, st);
    if (s != TM_OK || cap == 0) return s;
    const uint64_t blocks = std::min<uint64_t>((nch + 255) / 256, (uint64_t)num_sms * 8);
    list_chunks_kernel<<<(unsigned)blocks, 256, 0, st>>>(chunk_buf, nch, cap, counted);
    note_launches(1);
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}

bool long_frames(uint64_t longest_window) { return longest_window > FRAME_MAX / FCAP_FILL; }

namespace {
std::mutex g_cfg_mu;
std::unordered_map<uint64_t, int> g_blocks_per_sm;   // (device, kernel, warps, smem) -> resident blocks per SM

// Kernel instances: count and fill for each feature set (anti-edge checks, look-ahead
// checks, long frames), and count with work counters (all features).  A query
// runs the instance holding only the code its plan needs.
template <int MODE>
const void* kernel_for(unsigned feat) {
    if (feat & FEAT_LONG) {
        switch (feat & 3u) {
            case 0: return (const void*)search_kernel<MODE, false, FEAT_LONG>;
            case 1: return (const void*)search_kernel<MODE, false, FEAT_LONG | 1>;
            case 2: return (const void*)search_kernel<MODE, false, FEAT_LONG | 2>;
            default: return (const void*)search_kernel<MODE, false, FEAT_LONG | 3>;
        }
    }
    // pairs are only faster, not needed: beside a query with checks they are searched like any level
    if (feat == FEAT_PAIRS) return (const void*)search_kernel<MODE, false, FEAT_PAIRS>;
    if (MODE == MODE_COUNT && feat == FEAT_WIDE) return (const void*)search_kernel<MODE_COUNT, false, FEAT_WIDE>;
    switch (feat & 3u) {
        case 0: return (const void*)search_kernel<MODE, false, 0>;
        case 1: return (const void*)search_kernel<MODE, false, 1>;
        case 2: return (const void*)search_kernel<MODE, false, 2>;
        default: return (const void*)search_kernel<MODE, false, 3>;
    }
}
const void* kernel_of(Mode mode, bool stats, unsigned feat) {
    if (mode == MODE_FILL) return kernel_for<MODE_FILL>(feat);
    if (stats) return (const void*)search_kernel<MODE_COUNT, true, FEAT_LONG | 3>;
    return kernel_for<MODE_COUNT>(feat);
}

// dynamic shared memory a block may use beside the kernel's few static bytes
constexpr int MAX_DYN_SMEM = 232448 - 128;

// Resident blocks per SM for one launch shape, computed once per shape.
int blocks_per_sm(const tm_graph* g, const void* fn, int kid, int threads, int smem) {
    uint64_t key = ((uint64_t)g->device << 56) | ((uint64_t)kid << 48) | ((uint64_t)threads << 32) | (uint64_t)smem;
    std::lock_guard<std::mutex> lk(g_cfg_mu);
    auto it = g_blocks_per_sm.find(key);
    if (it != g_blocks_per_sm.end()) return it->second;
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, MAX_DYN_SMEM);
    int blocks = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, fn, threads, smem);
    cudaGetLastError();
    if (blocks < 1) blocks = 1;
    g_blocks_per_sm[key] = blocks;
    return blocks;
}
}  // namespace

// Blocks of a launch: the resident grid, less when the root chunks are too few
// to give each of its warps one (at least a block per SM stays to take donated
// subtrees).  Idle warps are not free: claiming, waiting and leaving go
// through a few shared lines.
int launch_blocks(const tm_graph* g, const LaunchCfg& c, uint64_t total_chunks) {
    const uint64_t need = (total_chunks + (uint64_t)c.warps_per_block - 1) / (uint64_t)c.warps_per_block;
    return (int)std::min<uint64_t>((uint64_t)c.grid, std::max<uint64_t>(need, (uint64_t)g->num_sms));
}

// Roots a warp claims at a time, of `roots` in the launch.  Too few of them to
// give each warp of a full grid (about 32 per SM) two chunks: smaller ones, down
// to 8 roots.  There the longest chain of one warp's chunks is the launch's time,
// not the number of claims.  Sizes set by the caller or picked by the tuner are kept.
int effective_chunk(const tm_graph* g, const Plan& p, uint64_t roots) {
    int cr = p.tune.chunk_roots;
    if (p.auto_chunk)
        while (cr > 8 && roots < 64ull * (uint64_t)g->num_sms * (uint64_t)cr) cr >>= 1;
    return cr;
}

LaunchCfg search_launch_cfg(const tm_graph* g, Mode mode, int max_warp_smem, int warps_per_block, unsigned feat,
                            bool stats) {
    LaunchCfg c;
    c.warps_per_block = std::max(1, std::min(16, warps_per_block));
    // keep the block's frames within the shared memory a block may use
    while (c.warps_per_block > 1 && max_warp_smem * c.warps_per_block > MAX_DYN_SMEM) c.warps_per_block--;
    c.smem_bytes = max_warp_smem * c.warps_per_block;
    feat &= 7u | FEAT_LONG;
    // 228 KB per SM, of which a block takes 1 KB beside its own
    if (feat == 0 && mode == MODE_COUNT && !stats &&
        228 * 1024 / (c.smem_bytes + (int)sizeof(Block) + 1024) * c.warps_per_block <= WIDE_WARPS)
        feat = FEAT_WIDE;
    c.fn = kernel_of(mode, stats, feat);
    c.grid = blocks_per_sm(g, c.fn, (mode == MODE_FILL ? 32 : 0) + (stats ? 16 : 0) + (int)feat, c.warps_per_block * 32,
                           c.smem_bytes) * g->num_sms;
    return c;
}

tm_status launch_search(const tm_graph* g, Mode mode, const QueryDev* qdev_dev, int nq, int max_warp_smem,
                        int warps_per_block, unsigned feat, const Scratch* s, cudaStream_t st, int grid_override,
                        bool stats) {
    if (mode == MODE_FILL) stats = false;
    // sets the instance's shared-memory limit too (once per launch shape)
    LaunchCfg c = search_launch_cfg(g, mode, max_warp_smem, warps_per_block, feat, stats);
    const int grid = grid_override > 0 ? std::min(grid_override, c.grid) : c.grid;
    GraphView v = g->v;
    Ctrl* ctrl = s->ctrl();
    Task* tasks = s->tasks;
    uint8_t* ready = s->ready;
    uint64_t cap = s->task_cap;
    void* args[] = {&v, (void*)&qdev_dev, &nq, &max_warp_smem, &ctrl, &tasks, &ready, &cap};
    TM_CUDA(cudaLaunchKernel(c.fn, dim3(grid), dim3(c.warps_per_block * 32), args, (size_t)c.smem_bytes, st));
    note_launches(1);
    return TM_OK;
}

}  // namespace tmg
