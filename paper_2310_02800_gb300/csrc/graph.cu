// Graph ingest (paper Section 4.2 data loader, Section 2.2 layout), on the GPU:
//   1. validate times and find their range, and validate node ids (host lists: the ids are
//      copied and checked while the times are sorted)
//   2. stable radix sort by time with the input index as payload -> edge ids
//      (skipped when the input is already in time order)
//   3. gather the edge columns into edge-id order, and the same as records
//   4. per direction: stable radix sort of (endpoint, edge id) -> lists in time
//      order and their offsets; gather (t, neighbour) columns for the lists.
//   5. out-lists re-ordered by (neighbour, time): closing-edge lookups
//   6. successor index: per edge, the first later position in its four lists; root filter
#include <cuda_runtime.h>
#include <sys/mman.h>
#include <unistd.h>

#include <algorithm>

#include "tm_internal.cuh"

namespace tmg {

namespace {

struct Check {
    unsigned long long tmin, tmax;
    unsigned long long bad;       // count of negative times
    unsigned long long descents;  // count of t[i] > t[i+1]
    unsigned long long bad_nodes; // not 0: some id is out of range
};

__global__ void check_times_kernel(const int64_t* __restrict__ t, int64_t m, Check* out) {
    unsigned long long tmin = ~0ULL, tmax = 0, bad = 0, desc = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t ti = t[i];
        if (ti < 0) bad++;
        unsigned long long u = (unsigned long long)(ti < 0 ? 0 : ti);
        tmin = min(tmin, u);
        tmax = max(tmax, u);
        if (i + 1 < m && t[i + 1] < ti) desc++;
    }
    for (int d = 16; d > 0; d >>= 1) {
        tmin = min(tmin, __shfl_down_sync(0xffffffffu, tmin, d));
        tmax = max(tmax, __shfl_down_sync(0xffffffffu, tmax, d));
        bad += __shfl_down_sync(0xffffffffu, bad, d);
        desc += __shfl_down_sync(0xffffffffu, desc, d);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMin(&out->tmin, tmin);
        atomicMax(&out->tmax, tmax);
        if (bad) atomicAdd(&out->bad, bad);
        if (desc) atomicAdd(&out->descents, desc);
    }
}

// Also packs the two endpoints of an edge side by side, for the gather into time order.
__global__ void check_nodes_kernel(const int32_t* __restrict__ src, const int32_t* __restrict__ dst, int64_t m, int64_t n,
                                   Check* out, int2* __restrict__ ends) {
    bool bad = false;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t s = src[i], d = dst[i];
        bad = bad || s < 0 || s >= n || d < 0 || d >= n;
        ends[i] = make_int2(s, d);
    }
    if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicAdd(&out->bad_nodes, 1ULL);
}

template <typename K>
__global__ void time_keys_kernel(const int64_t* __restrict__ t, int64_t m, unsigned long long tmin,
                                 K* __restrict__ keys) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x)
        keys[i] = (K)((uint64_t)t[i] - tmin);
}

// Elements a thread of the gather kernels takes at a time: their loads are all
// issued before the first is used, since each is a sector from anywhere in the column.
constexpr int GATHER = 4;

// An edge as one 16-byte record, for the gathers into list order: one sector per entry, where
// the time and the endpoint columns are two.
struct __align__(16) EdgeRec {
    int64_t t;
    int32_t src, dst;
};

// Edge columns in edge-id order, and the same as records.  The sorted keys are the times; without them
// (keys null) the input is in time order already and perm is null too.
template <typename K>
__global__ void gather_edges_kernel(const uint32_t* __restrict__ perm, const K* __restrict__ keys,
                                    unsigned long long tmin, int64_t m, const int2* __restrict__ ends,
                                    const int64_t* __restrict__ t,
                                    const uint8_t* __restrict__ el, int32_t* __restrict__ src_o,
                                    int32_t* __restrict__ dst_o, int64_t* __restrict__ t_o, uint8_t* __restrict__ el_o,
                                    int32_t* __restrict__ perm_o, EdgeRec* __restrict__ rec_o) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t e0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e0 < m; e0 += GATHER * stride) {
        uint32_t i[GATHER];
        int2 n[GATHER];
        int64_t tt[GATHER];
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t e = e0 + j * stride;
            i[j] = e >= m ? 0u : perm ? perm[e] : (uint32_t)e;
        }
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t e = e0 + j * stride;
            n[j] = ends[i[j]];
            tt[j] = e >= m ? 0 : keys ? (int64_t)((unsigned long long)keys[e] + tmin) : t[e];
        }
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t e = e0 + j * stride;
            if (e >= m) break;
            src_o[e] = n[j].x;
            dst_o[e] = n[j].y;
            t_o[e] = tt[j];
            if (el) el_o[e] = el[i[j]];
            rec_o[e] = EdgeRec{tt[j], n[j].x, n[j].y};
            perm_o[e] = (int32_t)i[j];
        }
    }
}

// List offsets from the list's sorted node column: off[v] = first entry of a
// node >= v.  (A binary search per node, neighbouring threads on neighbouring nodes:
// a degree histogram by atomics took 190 and 280 us for 10M edges, this 20.)
__global__ void offsets_kernel(const uint32_t* __restrict__ nodes, int64_t m, int64_t n1, uint32_t* __restrict__ off) {
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n1; v += (int64_t)gridDim.x * blockDim.x) {
        uint32_t lo = 0, hi = (uint32_t)m;
        while (lo < hi) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if ((int64_t)nodes[mid] < v) lo = mid + 1; else hi = mid;
        }
        off[v] = lo;
    }
}

__global__ void longest_list_kernel(const uint32_t* __restrict__ off0, const uint32_t* __restrict__ off1, int64_t n,
                                    uint32_t* __restrict__ longest) {
    uint32_t most = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x)
        most = max(most, max(off0[v + 1] - off0[v], off1[v + 1] - off1[v]));
    most = __reduce_max_sync(0xffffffffu, most);
    if ((threadIdx.x & 31) == 0) atomicMax(longest, most);
}

// List columns (time, other endpoint, edge id) from the list's edge ids.  Bound by its
// random sectors: 10M edges took 180 us from the time and endpoint columns, 158 from records.
template <bool IN>
__global__ void list_columns_kernel(const uint32_t* __restrict__ eids, int64_t m, const EdgeRec* __restrict__ rec,
                                    int64_t* __restrict__ at, int32_t* __restrict__ anbr, int32_t* __restrict__ aeid) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < m; i0 += GATHER * stride) {
        uint32_t e[GATHER];
        int4 r[GATHER];
#pragma unroll
        for (int j = 0; j < GATHER; ++j) e[j] = i0 + j * stride < m ? eids[i0 + j * stride] : 0u;
#pragma unroll
        for (int j = 0; j < GATHER; ++j) r[j] = __ldg((const int4*)(rec + e[j]));
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t i = i0 + j * stride;
            if (i >= m) break;
            at[i] = (int64_t)((uint64_t)(uint32_t)r[j].x | (uint64_t)(uint32_t)r[j].y << 32);
            anbr[i] = IN ? r[j].z : r[j].w;
            aeid[i] = (int32_t)e[j];
        }
    }
}

// Successor index by list position (see GraphView::pnx), the two words that
// were found in the other direction's order: position i's edge's word.
__global__ void successor_by_position_kernel(int64_t m, const int32_t* __restrict__ aeid_out,
                                             const int32_t* __restrict__ aeid_in, const uint2* __restrict__ so_dst,
                                             const uint2* __restrict__ si_src, uint2* __restrict__ p_out_dst,
                                             uint2* __restrict__ p_in_src) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < m; i0 += GATHER * stride) {
        int32_t eo[GATHER], ei[GATHER];
        uint2 wo[GATHER], wi[GATHER];
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t i = i0 + j * stride;
            eo[j] = i < m ? aeid_out[i] : 0;
            ei[j] = i < m ? aeid_in[i] : 0;
        }
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            wo[j] = so_dst[2u * (uint32_t)eo[j]];
            wi[j] = si_src[2u * (uint32_t)ei[j]];
        }
#pragma unroll
        for (int j = 0; j < GATHER; ++j) {
            const int64_t i = i0 + j * stride;
            if (i >= m) break;
            p_out_dst[i] = wo[j];
            p_in_src[i] = wi[j];
        }
    }
}

// first index in [lo, hi) with t[idx] > x
__device__ __forceinline__ uint32_t first_later(const int64_t* __restrict__ t, uint32_t lo, uint32_t hi, int64_t x) {
    while (lo < hi) {
        uint32_t mid = lo + ((hi - lo) >> 1);
        if (t[mid] <= x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// first index in [beg, hi) with t[idx] > x, searching outward from beg
__device__ __forceinline__ uint32_t first_later_from(const int64_t* __restrict__ t, uint32_t beg, uint32_t hi,
                                                     int64_t x) {
    uint32_t a = beg, b = hi, step = 1;
    while (true) {
        uint32_t probe = a + step - 1;
        if (probe >= hi) { b = hi; break; }
        if (t[probe] > x) { b = probe; break; }
        a = probe + 1;
        step <<= 1;
    }
    return first_later(t, a, b, x);
}

// Successor word for the first entry of a list [.., hi) at position p that is
// later than time te: {p, gap to its time} (SUCC_END when p == hi).
__device__ __forceinline__ uint2 succ_word(const int64_t* __restrict__ t, uint32_t p, uint32_t hi, int64_t te) {
    if (p >= hi) return make_uint2(p, SUCC_END);
    const uint64_t d = (uint64_t)(t[p] - te);
    return make_uint2(p, d < SUCC_FAR ? (uint32_t)d : SUCC_FAR);
}

// Successor index of one direction's lists, in list order.  Entry i of node v's
// list is edge e at time te: the first later entry of the same list (the search
// starts just past i) and the first later entry of v's list in the other direction,
// each with its time gap.  Both go to the edge in one 16-byte store: 10M edges took 690 us per
// direction when they were two stores to anywhere, 349 as one (reading them back in list order
// takes 352 us instead of 238, from columns twice as wide).  A search level whose candidate list belongs to an endpoint of
// the previous level's edge reads its window start here instead of
// binary-searching the list, and skips the window when the gap already
// exceeds it.  In list order, neighbouring threads search the same node's lists
// around the same times, so the searches stay in L1; by edge id every
// thread of a warp searched another node's list.
__global__ void successor_kernel(int64_t m, const uint32_t* __restrict__ nodes, const int32_t* __restrict__ eid,
                                 const uint32_t* __restrict__ off, const int64_t* __restrict__ at,
                                 const uint32_t* __restrict__ off_x, const int64_t* __restrict__ at_x,
                                 uint2* __restrict__ same_by_pos, uint4* __restrict__ by_edge) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < m; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t v = nodes[i];
        const int32_t e = eid[i];
        const int64_t te = at[i];
        uint32_t hi = off[v + 1];
        const uint2 w = succ_word(at, first_later_from(at, (uint32_t)i + 1u, hi, te), hi, te);
        same_by_pos[i] = w;
        hi = off_x[v + 1];
        const uint2 x = succ_word(at_x, first_later(at_x, off_x[v], hi, te), hi, te);
        by_edge[e] = make_uint4(w.x, w.y, x.x, x.y);
    }
}

// Root filter (see GraphView::rcode) from the four words of each edge.  A streaming pass of its own:
// storing the two bytes of a direction from successor_kernel, whose edges come in list
// order, is a partial sector per edge and cost ten times as much (0.5 ms for 10M edges).
__global__ void root_codes_kernel(int64_t m, const uint4* __restrict__ by_out, const uint4* __restrict__ by_in,
                                  uint32_t* __restrict__ rcode) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint4 o = by_out[e], i = by_in[e];
        rcode[e] = gap_code(o.y) << (8 * succ_byte(NX_OUT_SRC)) | gap_code(o.w) << (8 * succ_byte(NX_IN_SRC)) |
                   gap_code(i.y) << (8 * succ_byte(NX_IN_DST)) | gap_code(i.w) << (8 * succ_byte(NX_OUT_DST));
    }
}

__global__ void widen_kernel(const int32_t* __restrict__ in, int64_t n, int64_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) out[i] = in[i];
}

// Permutations of this many ids are widened on the host: 5,000 take 13 us there and 19 by the device's allocation,
// launch and free, 32,000 19 and 20, 64,000 37 and 21.
constexpr int64_t PERM_HOST = 1 << 15;

// Pages that the caller never touched are slow to fault in from the device (5.7M ids into fresh memory took 11 ms,
// with each page touched first 1.9): have them present, with their contents as they are.
void populate(void* p, size_t bytes) {
    char* const end = (char*)p + bytes;
    const size_t page = (size_t)sysconf(_SC_PAGESIZE);
    char* from = (char*)((uintptr_t)p & ~(uintptr_t)(page - 1));
#ifdef MADV_POPULATE_WRITE
    if (madvise(from, (size_t)(end - from), MADV_POPULATE_WRITE) == 0) return;
#endif
    // (a kernel without it, or memory it does not take) a read-modify-write of a byte of each
    for (char* b = (char*)p; b < end; b += page) __atomic_fetch_or(b, 0, __ATOMIC_RELAXED);
    __atomic_fetch_or(end - 1, 0, __ATOMIC_RELAXED);
}

int bits_for(unsigned long long x) {
    int b = 0;
    while (b < 64 && (x >> b) != 0) ++b;
    return b;
}

struct Pool {  // temporary device allocations, stream-ordered, freed at scope exit
    cudaStream_t st;
    std::vector<void*> ptrs;
    explicit Pool(cudaStream_t s) : st(s) {}
    ~Pool() {
        for (void* p : ptrs) cudaFreeAsync(p, st);
    }
    template <typename T>
    tm_status get(T** out, size_t count) {
        void* p = nullptr;
        if (dev_malloc_async(&p, std::max<size_t>(count * sizeof(T), 16), st) != cudaSuccess) {
            cudaGetLastError();
            set_error("cudaMalloc failed during graph build");
            return TM_E_OOM;
        }
        ptrs.push_back(p);
        *out = (T*)p;
        return TM_OK;
    }
};

// Host edge lists of at least this many edges copy their endpoints on a stream of their own, beside
// the time sort; below, the stream and its events cost what the overlap gives.
constexpr int64_t OVERLAP_MIN = 1 << 19;

// That stream: after what st held when it was opened; st goes on after it once joined.  It is
// drained before the buffers it writes (declared earlier) are freed.
struct Side {
    cudaStream_t st, cs = nullptr;
    cudaEvent_t ev = nullptr;
    explicit Side(cudaStream_t s) : st(s) {}
    tm_status open() {
        TM_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
        TM_CUDA(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        TM_CUDA(cudaEventRecord(ev, st));
        TM_CUDA(cudaStreamWaitEvent(cs, ev, 0));
        return TM_OK;
    }
    tm_status join() {
        TM_CUDA(cudaEventRecord(ev, cs));
        TM_CUDA(cudaStreamWaitEvent(st, ev, 0));
        return TM_OK;
    }
    ~Side() {
        if (cs) {
            cudaStreamSynchronize(cs);
            cudaStreamDestroy(cs);
        }
        if (ev) cudaEventDestroy(ev);
    }
};

// Graph storage is one allocation, carved into 256-byte aligned columns.
constexpr size_t COL_ALIGN = 256;
inline size_t col_bytes(size_t count, size_t elem) {
    return (std::max<size_t>(count * elem, 16) + COL_ALIGN - 1) & ~(COL_ALIGN - 1);
}

// Bytes of every column build() takes with owned(), in the same order.
size_t storage_bytes(int64_t n, int64_t m, bool node_labels, bool edge_labels) {
    size_t b = 0;
    if (node_labels) b += col_bytes(n, 1);
    b += col_bytes(m, 4) * 2 + col_bytes(m, 8) + col_bytes(m, 4);           // src, dst, t, perm
    if (edge_labels) b += col_bytes(m, 1);
    b += 2 * (col_bytes(n + 1, 4) + col_bytes(m, 8) + col_bytes(m, 4) * 2);  // out / in lists
    b += col_bytes(m, 4) + col_bytes(m, 8) + col_bytes(m, 4);               // pair-ordered list
    b += 2 * col_bytes(m, sizeof(uint4)) + 4 * col_bytes(m, sizeof(uint2));   // successor words
    b += col_bytes(m, 4);                                                     // root filter
    return b;
}

tm_status reserve_storage(tm_graph* g, size_t bytes) {
    void* p = nullptr;
    if (dev_malloc(&p, bytes) != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaMalloc failed for graph storage");
        return TM_E_OOM;
    }
    g->allocs.push_back(p);
    g->device_bytes += bytes;
    g->slab = (char*)p;
    g->slab_used = 0;
    g->slab_cap = bytes;
    return TM_OK;
}

template <typename T>
tm_status owned(tm_graph* g, T** out, size_t count) {
    const size_t bytes = col_bytes(count, sizeof(T));
    if (g->slab_used + bytes > g->slab_cap) {
        set_error("graph storage layout does not match the columns built");
        return TM_E_INVALID;
    }
    *out = (T*)(g->slab + g->slab_used);
    g->slab_used += bytes;
    return TM_OK;
}

#define TRY(x)                              \
    do {                                    \
        tm_status _s = (x);                 \
        if (_s != TM_OK) return _s;         \
    } while (0)

int grid_for(int64_t m, int sms) {
    int64_t g = (m + 255) / 256;
    return (int)std::max<int64_t>(1, std::min<int64_t>(g, (int64_t)sms * 16));
}

tm_status build(tm_graph* g, const tm_edges* e, cudaStream_t st) {
    const int64_t m = e->n_edges, n = e->n_nodes;
    const int sms = g->num_sms;
    Pool tmp(st);
    const int32_t *src = e->src, *dst = e->dst;
    const int64_t* t = e->t;
    const uint8_t* el = e->elabel;
    const bool host = !e->on_device && m > 0;
    // host endpoints and labels are copied and checked beside the time sort
    Side side(st);
    const bool overlap = host && m >= OVERLAP_MIN;
    cudaStream_t cs = st;
    int32_t *s2 = nullptr, *d2 = nullptr;
    int2* ends;
    uint8_t* el2 = nullptr;
    TRY(tmp.get(&ends, m));
    if (host) {
        int64_t* t2;
        TRY(tmp.get(&s2, m));
        TRY(tmp.get(&d2, m));
        TRY(tmp.get(&t2, m));
        if (el) TRY(tmp.get(&el2, m));
        TM_CUDA(cudaMemcpyAsync(t2, t, m * 8, cudaMemcpyHostToDevice, st));
        t = t2;
    }
    GraphView& v = g->v;
    v.n = n; v.m = m;
    TRY(reserve_storage(g, storage_bytes(n, m, e->nlabel != nullptr, el != nullptr)));
    // node labels
    if (e->nlabel) {
        uint8_t* nl;
        TRY(owned(g, &nl, n));
        TM_CUDA(cudaMemcpyAsync(nl, e->nlabel, n, e->on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, st));
        v.nlabel = nl;
    }
    // 1. validate
    Check* chk;
    TRY(tmp.get(&chk, 1));
    Check init{~0ULL, 0ULL, 0ULL, 0ULL, 0ULL}, hc;
    TM_CUDA(cudaMemcpyAsync(chk, &init, sizeof(Check), cudaMemcpyHostToDevice, st));
    if (overlap) {
        TRY(side.open());              // ordered after the allocations and the cleared counters
        cs = side.cs;
    }
    if (m > 0) {
        check_times_kernel<<<grid_for(m, sms), 256, 0, st>>>(t, m, chk);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
    }
    // the endpoints, on cs: copied where they come from the host, then checked
    auto endpoints = [&]() -> tm_status {
        if (host) {
            TM_CUDA(cudaMemcpyAsync(s2, src, m * 4, cudaMemcpyHostToDevice, cs));
            TM_CUDA(cudaMemcpyAsync(d2, dst, m * 4, cudaMemcpyHostToDevice, cs));
            if (el) TM_CUDA(cudaMemcpyAsync(el2, el, m, cudaMemcpyHostToDevice, cs));
            src = s2; dst = d2; el = el2;
        }
        if (m > 0) {
            check_nodes_kernel<<<grid_for(m, sms), 256, 0, cs>>>(src, dst, m, n, chk, ends);
            note_launches(1);
            TM_CUDA(cudaGetLastError());
        }
        return TM_OK;
    };
    auto read_check = [&](cudaStream_t on) -> tm_status {
        TM_CUDA(cudaMemcpyAsync(&hc, chk, sizeof(Check), cudaMemcpyDeviceToHost, on));
        TM_CUDA(cudaStreamSynchronize(on));
        if (hc.bad || hc.bad_nodes) {
            set_error("edge endpoint out of [0, n_nodes) or negative timestamp");
            return TM_E_INVALID;
        }
        return TM_OK;
    };
    if (!overlap) TRY(endpoints());
    TRY(read_check(st));
    // 2. time order
    const uint64_t um = (uint64_t)m;
    const int grid = grid_for(m, sms), grid4 = grid_for((m + GATHER - 1) / GATHER, sms);
    uint32_t *ka[2], *kb[2], *va[2], *keys_of[2], *spare[2];
    for (int j = 0; j < 2; ++j) {
        TRY(tmp.get(&ka[j], m));
        TRY(tmp.get(&kb[j], m));
        TRY(tmp.get(&va[j], m));
    }
    size_t rtemp_bytes = radix_temp_bytes(um);
    void* rtemp;
    TRY(tmp.get((char**)&rtemp, rtemp_bytes));
    int32_t *s_o, *d_o, *p_o;
    int64_t* t_o;
    uint8_t* el_o = nullptr;
    TRY(owned(g, &s_o, m));
    TRY(owned(g, &d_o, m));
    TRY(owned(g, &t_o, m));
    TRY(owned(g, &p_o, m));
    if (el) TRY(owned(g, &el_o, m));
    EdgeRec* rec;
    TRY(tmp.get(&rec, m));
    if (m > 0) {
        const int tbits = bits_for(hc.tmax - hc.tmin);
        const bool sorted = hc.descents == 0, narrow = tbits <= 32;
        int w = 0;
        uint64_t* k8[2] = {nullptr, nullptr};
        if (!sorted && narrow) {
            // a time range below 2^32: 4-byte keys
            time_keys_kernel<uint32_t><<<grid, 256, 0, st>>>(t, m, hc.tmin, kb[0]);
            note_launches(1);
            TM_CUDA(cudaGetLastError());
            TRY(radix_sort_pairs<uint32_t>(kb[0], nullptr, ka, va, um, tbits, rtemp, rtemp_bytes, st, &w));
        } else if (!sorted) {
            uint64_t* k0;
            TRY(tmp.get(&k0, m));
            TRY(tmp.get(&k8[0], m));
            TRY(tmp.get(&k8[1], m));
            time_keys_kernel<uint64_t><<<grid, 256, 0, st>>>(t, m, hc.tmin, k0);
            note_launches(1);
            TM_CUDA(cudaGetLastError());
            TRY(radix_sort_pairs<uint64_t>(k0, nullptr, k8, va, um, tbits, rtemp, rtemp_bytes, st, &w));
        }
        if (overlap) {
            TRY(endpoints());
            TRY(read_check(cs));
            TRY(side.join());
        }
        // 3. edge columns in edge-id order
        if (sorted)
            gather_edges_kernel<uint32_t><<<grid4, 256, 0, st>>>(nullptr, nullptr, 0, m, ends, t, el, s_o, d_o, t_o,
                                                                 el_o, p_o, rec);
        else if (narrow)
            gather_edges_kernel<uint32_t><<<grid4, 256, 0, st>>>(va[w], ka[w], hc.tmin, m, ends, t, el, s_o, d_o, t_o,
                                                                 el_o, p_o, rec);
        else
            gather_edges_kernel<uint64_t><<<grid4, 256, 0, st>>>(va[w], k8[w], hc.tmin, m, ends, t, el, s_o, d_o, t_o,
                                                                 el_o, p_o, rec);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
    }
    v.src = s_o; v.dst = d_o; v.t = t_o; v.elabel = el_o;
    g->perm = p_o;
    // 4. adjacency lists: edge ids sorted by endpoint, stably, are in time order per node
    const int nbits = bits_for((unsigned long long)(n > 0 ? n - 1 : 0));
    for (int dir = 0; dir < 2; ++dir) {
        const int32_t* key_node = dir == 0 ? s_o : d_o;
        uint32_t* off;
        int64_t* at;
        int32_t *anbr, *aeid;
        TRY(owned(g, &off, n + 1));
        TRY(owned(g, &at, m));
        TRY(owned(g, &anbr, m));
        TRY(owned(g, &aeid, m));
        uint32_t** nk = dir == 0 ? ka : kb;       // both directions' sorted nodes stay for step 6
        int w = 0;
        TRY(radix_sort_pairs<uint32_t>((const uint32_t*)key_node, nullptr, nk, va, um, nbits, rtemp, rtemp_bytes, st, &w));
        keys_of[dir] = nk[w];
        spare[dir] = nk[w ^ 1];
        offsets_kernel<<<grid_for(n + 1, sms), 256, 0, st>>>(keys_of[dir], m, n + 1, off);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
        if (m > 0) {
            if (dir == 0) list_columns_kernel<false><<<grid4, 256, 0, st>>>(va[w], m, rec, at, anbr, aeid);
            else list_columns_kernel<true><<<grid4, 256, 0, st>>>(va[w], m, rec, at, anbr, aeid);
            note_launches(1);
            TM_CUDA(cudaGetLastError());
        }
        v.off[dir] = off; v.at[dir] = at; v.anbr[dir] = anbr; v.aeid[dir] = aeid;
    }
    g->longest_list = (uint32_t)m;
    if (long_frames(um)) {
        uint32_t* longest;
        TRY(tmp.get(&longest, 1));
        TM_CUDA(cudaMemsetAsync(longest, 0, sizeof *longest, st));
        longest_list_kernel<<<grid_for(n, sms), 256, 0, st>>>(v.off[0], v.off[1], n, longest);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
        TM_CUDA(cudaMemcpyAsync(&g->longest_list, longest, sizeof *longest, cudaMemcpyDeviceToHost, st));
    }
    // 5. pair-ordered out-lists: the in-lists hold the edges by (destination, time) with
    //    their sources beside them, so one more stable sort, by source, gives
    //    (source, destination, time) order
    {
        int32_t *pn, *pe;
        int64_t* ptm;
        TRY(owned(g, &pn, m));
        TRY(owned(g, &ptm, m));
        TRY(owned(g, &pe, m));
        if (m > 0) {
            int w = 0;                            // the sorted sources are not needed
            TRY(radix_sort_pairs<uint32_t>((const uint32_t*)v.anbr[1], (const uint32_t*)v.aeid[1], spare, va, um, nbits,
                                           rtemp, rtemp_bytes, st, &w));
            list_columns_kernel<false><<<grid4, 256, 0, st>>>(va[w], m, rec, ptm, pn, pe);
            note_launches(1);
            TM_CUDA(cudaGetLastError());
        }
        v.pnbr = pn; v.pt = ptm; v.peid = pe;
    }
    // 6. successor index (window starts for lists that touch the previous edge)
    uint4* by_edge[2];                            // by out-list order, by in-list order
    uint2* px[4];
    for (int j = 0; j < 2; ++j) TRY(owned(g, &by_edge[j], m));
    for (int j = 0; j < 4; ++j) TRY(owned(g, &px[j], m));
    uint32_t* codes;
    TRY(owned(g, &codes, m));
    v.nxt[NX_OUT_SRC] = (const uint2*)by_edge[0];
    v.nxt[NX_IN_SRC] = (const uint2*)by_edge[0] + 1;
    v.nxt[NX_IN_DST] = (const uint2*)by_edge[1];
    v.nxt[NX_OUT_DST] = (const uint2*)by_edge[1] + 1;
    if (m > 0) {
        successor_kernel<<<grid, 256, 0, st>>>(m, keys_of[0], v.aeid[0], v.off[0], v.at[0], v.off[1], v.at[1], px[0], by_edge[0]);
        successor_kernel<<<grid, 256, 0, st>>>(m, keys_of[1], v.aeid[1], v.off[1], v.at[1], v.off[0], v.at[0], px[2], by_edge[1]);
        successor_by_position_kernel<<<grid4, 256, 0, st>>>(m, v.aeid[0], v.aeid[1], v.nxt[NX_OUT_DST], v.nxt[NX_IN_SRC],
                                                           px[1], px[3]);
        root_codes_kernel<<<grid, 256, 0, st>>>(m, by_edge[0], by_edge[1], codes);
        note_launches(4);
        TM_CUDA(cudaGetLastError());
    }
    for (int j = 0; j < 4; ++j) v.pnx[j] = px[j];
    v.rcode = codes;
    TM_CUDA(cudaStreamSynchronize(st));
    return TM_OK;
}

}  // namespace

}  // namespace tmg

using namespace tmg;

extern "C" tm_status tm_graph_load(const tm_edges* e, int device, void* stream, tm_graph** out) {
    if (!e || !out) { set_error("null argument"); return TM_E_INVALID; }
    if (e->n_edges < 0 || e->n_nodes < 0 || e->n_edges >= 0x3FFFFFFF || e->n_nodes >= 0x7FFFFFFF) {
        set_error("n_edges / n_nodes out of range");
        return TM_E_INVALID;
    }
    if (e->n_edges > 0 && (!e->src || !e->dst || !e->t || e->n_nodes < 1)) {
        set_error("missing edge columns");
        return TM_E_INVALID;
    }
    int ndev = 0;
    TM_CUDA(cudaGetDeviceCount(&ndev));
    if (device < 0 || device >= ndev) { set_error("bad device"); return TM_E_INVALID; }
    TM_ENTER(device);
    tm_graph* g = new tm_graph();
    g->device = device;
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) { delete g; return cuda_fail(cudaGetLastError(), "props"); }
    g->num_sms = prop.multiProcessorCount;
    InFlight call((cudaStream_t)stream, &g->unsettled);
    tm_status s = build(g, e, (cudaStream_t)stream);
    if (s != TM_OK) {
        call.wait();
        tm_graph_free(g);
        return s;
    }
    call.settle();
    *out = g;
    return TM_OK;
}

extern "C" tm_status tm_graph_free(tm_graph* g) {
    if (!g) return TM_OK;
    cudaSetDevice(g->device);
    drop_batches(g);
    for (void* p : g->allocs) dev_free(p, g->device, g->unsettled == 0);
    pool_give_back(g->device);
    delete g;
    return TM_OK;
}

extern "C" tm_status tm_graph_info(const tm_graph* g, int64_t* n_nodes, int64_t* n_edges, uint64_t* device_bytes) {
    if (!g) { set_error("null graph"); return TM_E_INVALID; }
    if (n_nodes) *n_nodes = g->v.n;
    if (n_edges) *n_edges = g->v.m;
    if (device_bytes) *device_bytes = g->device_bytes;
    return TM_OK;
}

extern "C" tm_status tm_graph_edge_perm(const tm_graph* g, int64_t* out_perm) {
    if (!g || (!out_perm && g->v.m > 0)) { set_error("null argument"); return TM_E_INVALID; }
    if (g->v.m == 0) return TM_OK;
    TM_ENTER(g->device);
    // widened on the device, all of it before any is copied, and copied straight out; up to PERM_HOST ids
    // through the host copy below
    const int64_t m = g->v.m;
    int64_t* wide = nullptr;
    if (m > PERM_HOST && dev_malloc((void**)&wide, (size_t)m * 8) == cudaSuccess) {
        widen_kernel<<<grid_for(m, g->num_sms), 256>>>(g->perm, m, wide);
        note_launches(1);
        cudaError_t e = cudaGetLastError();
        const bool launched = e == cudaSuccess;
        if (launched) {
            populate(out_perm, (size_t)m * 8);
            e = cudaMemcpy(out_perm, wide, (size_t)m * 8, cudaMemcpyDeviceToHost);
        }
        dev_free(wide, g->device, !launched || e == cudaSuccess);
        return e == cudaSuccess ? TM_OK : cuda_fail(e, "edge permutation");
    }
    // few ids, or no device memory to spare
    cudaGetLastError();
    std::vector<int32_t> tmp((size_t)m);
    TM_CUDA(cudaMemcpy(tmp.data(), g->perm, m * 4, cudaMemcpyDeviceToHost));
    for (int64_t i = 0; i < m; ++i) out_perm[i] = tmp[i];
    return TM_OK;
}
