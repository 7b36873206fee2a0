// Device building blocks for graph ingest and enumeration offsets:
// an exclusive prefix sum and a stable LSD radix sort of (key, value) pairs.
#include <cuda_runtime.h>

#include <algorithm>

#include "tm_internal.cuh"

namespace tmg {

// ------------------------------------------------------------------- scan

namespace {
constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        T u = __shfl_up_sync(0xffffffffu, v, d);
        if (lane >= d) v += u;
    }
    return v;
}

// Exclusive scan of one block's thread totals; returns this thread's prefix,
// and the block total in *total.
template <typename T>
__device__ T block_excl_scan(T v, T* total) {
    __shared__ T warp_sum[SCAN_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) warp_sum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < SCAN_THREADS / 32 ? warp_sum[lane] : T(0);
        T wi = warp_incl_scan(w);
        if (lane < SCAN_THREADS / 32) warp_sum[lane] = wi - w;
        if (lane == SCAN_THREADS / 32 - 1) *total = wi;
    }
    __syncthreads();
    T r = warp_sum[warp] + inc - v;
    __syncthreads();
    return r;
}

template <typename T>
__global__ void scan_reduce_kernel(const T* __restrict__ in, uint64_t n, T* __restrict__ partial) {
    __shared__ T red[SCAN_THREADS / 32];
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE;
    T s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        uint64_t i = base + (uint64_t)j * SCAN_THREADS + threadIdx.x;
        if (i < n) s += in[i];
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_down_sync(0xffffffffu, s, d);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        T t = 0;
        for (int w = 0; w < SCAN_THREADS / 32; ++w) t += red[w];
        partial[blockIdx.x] = t;
    }
}

// Block-level exclusive scan of one tile plus the tile's carried-in offset.
template <typename T>
__global__ void scan_down_kernel(const T* in, T* out, uint64_t n, const T* __restrict__ partial_scanned) {
    __shared__ T tile[SCAN_TILE];
    __shared__ T tot;
    uint64_t base = (uint64_t)blockIdx.x * SCAN_TILE;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        int li = j * SCAN_THREADS + threadIdx.x;
        uint64_t i = base + li;
        tile[li] = i < n ? in[i] : T(0);
    }
    __syncthreads();
    T loc[SCAN_ITEMS];
    T s = 0;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        loc[j] = tile[threadIdx.x * SCAN_ITEMS + j];
        s += loc[j];
    }
    T pre = block_excl_scan(s, &tot);
    T carry = partial_scanned ? partial_scanned[blockIdx.x] : T(0);
    pre += carry;
#pragma unroll
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        tile[threadIdx.x * SCAN_ITEMS + j] = pre;
        pre += loc[j];
    }
    __syncthreads();
    for (int j = 0; j < SCAN_ITEMS; ++j) {
        int li = j * SCAN_THREADS + threadIdx.x;
        uint64_t i = base + li;
        if (i < n) out[i] = tile[li];
    }
}

uint64_t ceil_div(uint64_t a, uint64_t b) { return (a + b - 1) / b; }
}  // namespace

size_t scan_temp_bytes(uint64_t n) {
    size_t bytes = 0;
    uint64_t len = n;
    while (len > (uint64_t)SCAN_TILE) {
        len = ceil_div(len, SCAN_TILE);
        bytes += ((len * 8 + 255) / 256) * 256;
    }
    return bytes + 256;
}

template <typename T>
tm_status exclusive_scan(const T* in, T* out, uint64_t n, T* temp, cudaStream_t st) {
    if (n == 0) return TM_OK;
    uint64_t nb = ceil_div(n, SCAN_TILE);
    if (nb == 1) {
        scan_down_kernel<T><<<1, SCAN_THREADS, 0, st>>>(in, out, n, nullptr);
        note_launches(1);
        TM_CUDA(cudaGetLastError());
        return TM_OK;
    }
    T* partial = temp;
    T* rest = (T*)((char*)temp + ((nb * 8 + 255) / 256) * 256);
    scan_reduce_kernel<T><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, n, partial);
    note_launches(1);
    TM_CUDA(cudaGetLastError());
    tm_status s = exclusive_scan(partial, partial, nb, rest, st);
    if (s != TM_OK) return s;
    scan_down_kernel<T><<<(unsigned)nb, SCAN_THREADS, 0, st>>>(in, out, n, partial);
    note_launches(1);
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}

tm_status exclusive_scan_u64(const unsigned long long* in, unsigned long long* out, uint64_t n, void* temp,
                             cudaStream_t st) {
    return exclusive_scan(in, out, n, (unsigned long long*)temp, st);
}

// ------------------------------------------------------------ radix sort
//
// Stable LSD sort of (key, 32-bit value) pairs, up to 8 bits a pass, the key's
// bits spread evenly over the passes (20 bits: 7 + 7 + 6).  A pass counts each
// tile's digits, scans the counts (digit-major) and scatters.  What bounds it
// is how the scatter's writes fall: an element's destination is anywhere, so
// writing from registers touches a 32-byte sector per element.  The scatter therefore
// orders its tile in shared memory first and writes each digit's run with
// consecutive threads: 8,192 elements over 128 digits are runs of 256 bytes.

namespace {
constexpr int RS_BINS = 256;
// threads and elements per thread: small inputs take small tiles, so that their few tiles still cover the SMs
struct RsBig { static constexpr int THREADS = 512, ITEMS = 16; };
struct RsSmall { static constexpr int THREADS = 256, ITEMS = 4; };
constexpr uint64_t RS_SMALL_N = 1u << 20;
inline int rs_tile(uint64_t n) {
    return n <= RS_SMALL_N ? RsSmall::THREADS * RsSmall::ITEMS : RsBig::THREADS * RsBig::ITEMS;
}

template <typename K, int RS_THREADS, int ITEMS>
__global__ void radix_hist_kernel(const K* __restrict__ keys, uint64_t n, int shift, unsigned mask, uint64_t ntiles,
                                  uint32_t* __restrict__ counts) {
    __shared__ unsigned int h[RS_BINS];
    if (threadIdx.x < RS_BINS) h[threadIdx.x] = 0;
    __syncthreads();
    const uint64_t base = (uint64_t)blockIdx.x * (RS_THREADS * ITEMS);
    K key[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint64_t i = base + (uint64_t)j * RS_THREADS + threadIdx.x;
        key[j] = i < n ? keys[i] : K(0);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint64_t i = base + (uint64_t)j * RS_THREADS + threadIdx.x;
        if (i < n) atomicAdd(&h[(unsigned)(key[j] >> shift) & mask], 1u);
    }
    __syncthreads();
    if (threadIdx.x <= mask) counts[(uint64_t)threadIdx.x * ntiles + blockIdx.x] = h[threadIdx.x];
}

// Elements of a tile are ranked in input order: warp w holds the tile's w-th
// part, item by item; one ballot per digit bit ranks equal digits within an item (__match_any_sync
// takes longer the more digits differ: a 7-bit pass over 10M elements 85 us with it, 52 without), the
// warp's running digit counts rank the items, and a scan over the warps ranks the warps.
template <typename K, int RS_THREADS, int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 1024 / RS_THREADS) radix_scatter_kernel(
    const K* __restrict__ kin, const uint32_t* __restrict__ vin, K* __restrict__ kout, uint32_t* __restrict__ vout,
    uint64_t n, int shift, unsigned mask, uint64_t ntiles, const uint32_t* __restrict__ offsets) {
    constexpr int TILE = RS_THREADS * ITEMS, RS_WARPS = RS_THREADS / 32;
    extern __shared__ __align__(16) unsigned char rs_smem[];
    K* skey = (K*)rs_smem;                                   // the tile in digit order
    uint32_t* sval = (uint32_t*)(rs_smem + sizeof(K) * TILE);
    __shared__ uint32_t wc[RS_WARPS][RS_BINS];               // digit counts per warp, then where each warp's run starts
    __shared__ uint32_t dst[RS_BINS];                        // a digit's output start minus its start in the tile
    __shared__ uint32_t wsum[RS_BINS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const uint64_t tile0 = (uint64_t)blockIdx.x * TILE;
    const int left = (int)(n - tile0 < (uint64_t)TILE ? n - tile0 : (uint64_t)TILE);
    const int seg = warp * (32 * ITEMS);
    for (int d = lane; d < RS_BINS; d += 32) wc[warp][d] = 0;
    K key[ITEMS];
    uint32_t rank[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int i = seg + j * 32 + lane;
        key[j] = i < left ? kin[tile0 + i] : K(0);
    }
    const uint32_t out0 = threadIdx.x <= mask ? offsets[(uint64_t)threadIdx.x * ntiles + blockIdx.x] : 0u;
    __syncwarp();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const bool valid = seg + j * 32 + lane < left;
        const unsigned d = (unsigned)(key[j] >> shift) & mask;
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            if (!(mask >> b & 1u)) break;
            const unsigned ones = __ballot_sync(0xffffffffu, d >> b & 1u);
            peers &= d >> b & 1u ? ones : ~ones;
        }
        const uint32_t before = valid ? wc[warp][d] : 0u;
        rank[j] = before + __popc(peers & lt);
        __syncwarp();
        if (valid && (peers & lt) == 0) wc[warp][d] = before + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    {
        // thread d < RS_BINS: digit d's total, its start in the tile, and each warp's start within it
        const bool digit = threadIdx.x < RS_BINS;
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < RS_WARPS; ++w) tot += digit ? wc[w][threadIdx.x] : 0u;
        uint32_t inc = tot;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, inc, s);
            if (lane >= s) inc += u;
        }
        if (digit && lane == 31) wsum[warp] = inc;
        __syncthreads();
        if (digit) {
            uint32_t at = inc - tot;
            for (int w = 0; w < warp; ++w) at += wsum[w];
            dst[threadIdx.x] = out0 - at;
#pragma unroll
            for (int w = 0; w < RS_WARPS; ++w) {
                const uint32_t c = wc[w][threadIdx.x];
                wc[w][threadIdx.x] = at;
                at += c;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int i = seg + j * 32 + lane;
        if (i >= left) continue;
        const unsigned d = (unsigned)(key[j] >> shift) & mask;
        const uint32_t p = wc[warp][d] + rank[j];
        skey[p] = key[j];
        // read only now: values held through the ranking took the registers of half the warps
        sval[p] = vin ? vin[tile0 + i] : (uint32_t)(tile0 + i);
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const int p = j * RS_THREADS + threadIdx.x;
        if (p >= left) continue;
        const K kk = skey[p];
        const uint32_t o = dst[(unsigned)(kk >> shift) & mask] + (uint32_t)p;
        kout[o] = kk;
        vout[o] = sval[p];
    }
}

template <typename K, typename T>
tm_status radix_pass(const K* ki, const uint32_t* vi, K* ko, uint32_t* vo, uint64_t n, int shift, unsigned mask,
                     uint32_t* counts, void* scan_tmp, cudaStream_t st) {
    const uint64_t ntiles = ceil_div(n, T::THREADS * T::ITEMS);
    constexpr int bytes = T::THREADS * T::ITEMS * (int)(sizeof(K) + 4);
    if (bytes > 24 * 1024)
        TM_CUDA(cudaFuncSetAttribute(radix_scatter_kernel<K, T::THREADS, T::ITEMS>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    radix_hist_kernel<K, T::THREADS, T::ITEMS><<<(unsigned)ntiles, T::THREADS, 0, st>>>(ki, n, shift, mask, ntiles, counts);
    note_launches(1);
    TM_CUDA(cudaGetLastError());
    tm_status s = exclusive_scan(counts, counts, ntiles * (mask + 1u), (uint32_t*)scan_tmp, st);
    if (s != TM_OK) return s;
    radix_scatter_kernel<K, T::THREADS, T::ITEMS><<<(unsigned)ntiles, T::THREADS, bytes, st>>>(ki, vi, ko, vo, n, shift, mask,
                                                                                             ntiles, counts);
    note_launches(1);
    TM_CUDA(cudaGetLastError());
    return TM_OK;
}
}  // namespace

size_t radix_temp_bytes(uint64_t n) {
    const uint64_t cnt = ceil_div(n > 0 ? n : 1, rs_tile(n)) * RS_BINS;
    return ((cnt * 4 + 255) / 256) * 256 + scan_temp_bytes(cnt);
}

template <typename K>
tm_status radix_sort_pairs(const K* keys_in, const uint32_t* vals_in, K* const keys[2], uint32_t* const vals[2], uint64_t n,
                           int bits, void* temp, size_t temp_bytes, cudaStream_t st, int* which) {
    *which = 0;
    if (n == 0) return TM_OK;
    if (temp_bytes < radix_temp_bytes(n)) return TM_E_INVALID;
    uint32_t* counts = (uint32_t*)temp;
    const uint64_t cnt = ceil_div(n, rs_tile(n)) * RS_BINS;
    void* scan_tmp = (char*)temp + ((cnt * 4 + 255) / 256) * 256;
    bits = std::max(bits, 1);          // one distinct key: a stable copy
    const int passes = (bits + 7) / 8, per = (bits + passes - 1) / passes;
    for (int p = 0; p * per < bits; ++p) {
        const unsigned mask = (1u << std::min(per, bits - p * per)) - 1u;
        const K* ki = p == 0 ? keys_in : keys[*which];
        const uint32_t* vi = p == 0 ? vals_in : vals[*which];
        const int to = p == 0 ? 0 : *which ^ 1;
        tm_status s = n <= RS_SMALL_N ? radix_pass<K, RsSmall>(ki, vi, keys[to], vals[to], n, p * per, mask, counts, scan_tmp, st)
                                      : radix_pass<K, RsBig>(ki, vi, keys[to], vals[to], n, p * per, mask, counts, scan_tmp, st);
        if (s != TM_OK) return s;
        *which = to;
    }
    return TM_OK;
}

template tm_status radix_sort_pairs<uint64_t>(const uint64_t*, const uint32_t*, uint64_t* const[2], uint32_t* const[2],
                                              uint64_t, int, void*, size_t, cudaStream_t, int*);
template tm_status radix_sort_pairs<uint32_t>(const uint32_t*, const uint32_t*, uint32_t* const[2], uint32_t* const[2],
                                              uint64_t, int, void*, size_t, cudaStream_t, int*);

}  // namespace tmg
