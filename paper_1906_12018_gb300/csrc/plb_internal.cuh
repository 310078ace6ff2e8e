// Internal device/host helpers of the labeling library (sm_103a).
//
// Label entries are packed 32-bit words: bits 31..8 = hub rank (24 bits),
// bits 7..0 = distance.  Within a row, entries are sorted by hub rank, so a
// plain unsigned comparison of packed words orders them by hub (hubs are
// unique per row).  0xFFFFFFFF never occurs as an entry (distance 255 is
// reserved) and marks empty hash slots.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "plb.h"

namespace plb {

constexpr uint32_t kEmpty = 0xFFFFFFFFu;
constexpr unsigned kFull = 0xFFFFFFFFu;
constexpr int kHubShift = 8;

__host__ __device__ __forceinline__ uint32_t pack(uint32_t hub, uint32_t d) { return (hub << kHubShift) | d; }
__host__ __device__ __forceinline__ uint32_t hub_of(uint32_t e) { return e >> kHubShift; }
__host__ __device__ __forceinline__ uint32_t dist_of(uint32_t e) { return e & 0xFFu; }

// frontier row descriptor: start (40 bits) | count (24 bits)
__host__ __device__ __forceinline__ uint64_t fpack(uint64_t start, uint32_t cnt) { return (start << 24) | cnt; }
__host__ __device__ __forceinline__ uint64_t fstart(uint64_t x) { return x >> 24; }
__host__ __device__ __forceinline__ uint32_t fcount(uint64_t x) { return (uint32_t)(x & 0xFFFFFFu); }

// Fibonacci hashing of a hub rank into a table of 2^logcap slots.
__device__ __forceinline__ uint32_t hslot(uint32_t key, int logcap) {
    return (key * 0x9E3779B1u) >> (32 - logcap);
}

// Insert key into an open-addressing set; returns true if it was new.
// The caller guarantees the table never fills (load <= 1/2 plus the number
// of concurrently inserting threads).
// (Every probe loop below is bounded by the table size, so a table broken by
// a bug can never spin a kernel forever.)
__device__ __forceinline__ bool set_insert(uint32_t* tab, int logcap, uint32_t key) {
    const uint32_t mask = (1u << logcap) - 1u;
    uint32_t s = hslot(key, logcap);
#pragma unroll 1
    for (uint32_t i = 0; i <= mask; ++i) {
        const uint32_t old = atomicCAS(tab + s, kEmpty, key);
        if (old == kEmpty) return true;
        if (old == key) return false;
        s = (s + 1) & mask;
    }
    return false;
}

// Hub-keyed tables of packed label entries (at least 32 slots, at most half
// full, 16-byte aligned): buckets of four slots, filled from the first slot
// on and, when a bucket is full, on into the next ones.  A look-up reads a
// bucket in one 16-byte load and ends there unless the bucket is full without
// the hub (2% of the buckets at load 1/4, 14% at 1/2): probing slot by slot
// took a loop whose length was the longest chain among the warp's lanes.
__device__ __forceinline__ uint32_t bslot(uint32_t key, int logcap) { return hslot(key, logcap) & ~3u; }

// Insert a packed label entry keyed by its hub (keys unique by construction).
__device__ __forceinline__ void map_insert(uint32_t* tab, int logcap, uint32_t e) {
    const uint32_t mask = (1u << logcap) - 1u;
    uint32_t s = bslot(hub_of(e), logcap);
#pragma unroll 1
    for (uint32_t i = 0; i <= mask && atomicCAS(tab + s, kEmpty, e) != kEmpty; ++i) s = (s + 1) & mask;
}

// Whether a bucket holds hub xh >> 8 at a distance of at most lim <= 254 (xh:
// the hub as a packed entry of distance 0; an empty slot never matches).
__device__ __forceinline__ bool bucket_has(uint4 y, uint32_t xh, uint32_t lim) {
    return y.x - xh <= lim || y.y - xh <= lim || y.z - xh <= lim || y.w - xh <= lim;
}

// Whether the table holds hub xh >> 8 at a distance of at most lim, the bucket
// at s having been read as y: follows the chain of full buckets (at most the
// whole table).
__device__ __forceinline__ bool map_has_from(const uint32_t* tab, int logcap, uint32_t s, uint4 y, uint32_t xh,
                                             uint32_t lim) {
    const uint32_t mask = (1u << logcap) - 1u;
#pragma unroll 1
    for (uint32_t i = 0; i <= mask; i += 4) {
        if (bucket_has(y, xh, lim)) return true;
        if (y.w == kEmpty) return false;
        s = (s + 4) & mask;
        y = *reinterpret_cast<const uint4*>(tab + s);
    }
    return false;
}

// Whether hub w is in the table.
__device__ __forceinline__ bool map_has(const uint32_t* tab, int logcap, uint32_t w) {
    const uint32_t s = bslot(w, logcap);
    return map_has_from(tab, logcap, s, *reinterpret_cast<const uint4*>(tab + s), pack(w, 0), 254u);
}

__device__ __forceinline__ int warp_incl_scan(int x, int lane) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += t;
    }
    return x;
}

// Runs of equal keys over the lanes (each key's lanes consecutive, as the
// rows of consecutive arcs): returns, in every lane, the sum of x over the
// lane's run, which holds lanes *first..*last.  All 32 lanes call it.
__device__ __forceinline__ int run_sum(int64_t key, int x, int lane, int* first, int* last) {
    const int incl = warp_incl_scan(x, lane);
    const int64_t kprev = __shfl_up_sync(kFull, key, 1);
    const int64_t knext = __shfl_down_sync(kFull, key, 1);
    const unsigned starts = __ballot_sync(kFull, lane == 0 || kprev != key);
    const unsigned ends = __ballot_sync(kFull, lane == 31 || knext != key);
    const int f = 31 - __clz(starts & (0xFFFFFFFFu >> (31 - lane)));  // last run start at or below the lane
    const int l = __ffs(ends & (0xFFFFFFFFu << lane)) - 1;            // first run end at or above it
    const int before = __shfl_sync(kFull, incl - x, f);
    *first = f;
    *last = l;
    return __shfl_sync(kFull, incl, l) - before;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(kFull, x, o);
    return x;
}

// Largest lane k whose exclusive prefix excl_k <= item (excl non-decreasing
// over lanes).  All 32 lanes must call.
__device__ __forceinline__ int warp_owner(int excl, int item) {
    int k = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const int e = __shfl_sync(kFull, excl, k + step);
        if (e <= item) k += step;
    }
    return k;
}

// Number of entries of sorted a[0..len) that are < key (hub comparison on
// packed entries when the key is given as a packed word with distance 0).
__device__ __forceinline__ int64_t lower_bound_u32(const uint32_t* a, int64_t len, uint32_t key) {
    int64_t lo = 0, hi = len;
#pragma unroll 1
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (a[mid] < key) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// Row r of offsets off[] containing item p (largest r with off[r] <= p) in [lo,
// hi], by a whole warp, 32 probes at a time (a binary search is a chain of
// log2(rows) dependent loads; all lanes call and get the result).
__device__ __forceinline__ int64_t warp_row_of(const int64_t* off, int64_t lo, int64_t hi, int64_t p) {
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) / 32;
        const int64_t r = lo + (lane + 1) * step;
        const int c = __popc(__ballot_sync(kFull, r <= hi && off[r] <= p));  // (off is non-decreasing)
        lo += c * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

// Flat passes over the items of rows (arcs, label entries): tiles of kTileItems
// consecutive items per block of kTileThreads threads, so that rows of any
// length are spread evenly.
constexpr int kTileItems = 2048;
constexpr int kTileThreads = 256;

// Row of every item of the tile [p0, p1): srow[i] = row of item p0 + i, less
// *r0 (the tile's first row; *r1 its last).  The first and last row are found
// by two warps, each row's start is marked in srow and a running maximum gives
// every item its row: one thread searching both ends cost 40 dependent loads
// per tile (20 us), and a search per item 8 to 9 more (builds, before -> after,
// with the two-launch scans: 4K vertices 1.76 -> 1.25 ms, 61K 3.4 -> 2.7 ms).
// All threads call.
struct TileScratch {
    int64_t r[2];
    int wmax[kTileThreads / 32];
};
__device__ __forceinline__ void tile_rows(const int64_t* off, int64_t nrows, int64_t p0, int64_t p1, int* srow,
                                             TileScratch* sh, int64_t* r0, int64_t* r1) {
    constexpr int kPer = kTileItems / kTileThreads;
    static_assert(kPer == 8, "eight items per thread");
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    __syncthreads();  // (srow and sh may still be read for the tile before)
    if (wid < 2) {
        const int64_t r = warp_row_of(off, 0, nrows - 1, wid == 0 ? p0 : p1 - 1);
        if (lane == 0) sh->r[wid] = r;
    }
    int4* s4 = reinterpret_cast<int4*>(srow) + 2 * tid;
    s4[0] = make_int4(0, 0, 0, 0);
    s4[1] = make_int4(0, 0, 0, 0);
    __syncthreads();
    const int64_t a = sh->r[0], b = sh->r[1];
    for (int64_t r = a + 1 + tid; r <= b; r += kTileThreads) {
        const int64_t q = off[r] - p0;
        if (q >= 0 && q < kTileItems) atomicMax(&srow[(int)q], (int)(r - a));  // (always, in a valid CSR)
    }
    __syncthreads();
    int4 x = s4[0], y = s4[1];
    x.y = max(x.y, x.x);
    x.z = max(x.z, x.y);
    x.w = max(x.w, x.z);
    y.x = max(y.x, x.w);
    y.y = max(y.y, y.x);
    y.z = max(y.z, y.y);
    y.w = max(y.w, y.z);
    int m = y.w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(kFull, m, o);
        if (lane >= o) m = max(m, t);
    }
    if (lane == 31) sh->wmax[wid] = m;
    int before = __shfl_up_sync(kFull, m, 1);
    if (lane == 0) before = 0;
    __syncthreads();
    for (int k = 0; k < wid; ++k) before = max(before, sh->wmax[k]);
    s4[0] = make_int4(max(x.x, before), max(x.y, before), max(x.z, before), max(x.w, before));
    s4[1] = make_int4(max(y.x, before), max(y.y, before), max(y.z, before), max(y.w, before));
    __syncthreads();
    *r0 = a;
    *r1 = b;
}

// Which of an edge's two arcs the input checks look up (see k_check_cols).
__device__ __forceinline__ bool looked_up(const int64_t* row_ptr, int64_t u, int64_t c) {
    const int64_t du = row_ptr[u + 1] - row_ptr[u], dc = row_ptr[c + 1] - row_ptr[c];
    return dc < du || (dc == du && c < u);
}

// Bitonic sort of a[0..P) (P a power of two) by a group of nthreads threads.
// Each step runs over the P/2 compare-exchange pairs (i, i + j), i the pair
// index t with a zero bit inserted at bit log2(j): no idle half of the
// threads.
template <typename Sync>
__device__ void group_bitonic_sort(uint32_t* a, int P, int tid, int nthreads, Sync sync) {
    const int half = P >> 1;
#pragma unroll 1
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
#pragma unroll 1
            for (int t = tid; t < half; t += nthreads) {
                const int i = 2 * t - (t & (j - 1));
                const int l = i + j;
                const uint32_t x = a[i], y = a[l];
                const bool up = (i & k) == 0;
                if ((x > y) == up) {
                    a[i] = y;
                    a[l] = x;
                }
            }
            sync();
        }
    }
}

__host__ __device__ __forceinline__ int ceil_log2_i64(int64_t x) {
    int b = 0;
    while ((int64_t(1) << b) < x) ++b;
    return b;
}

}  // namespace plb

// ---------------------------------------------------------------- host side
struct plb_labels {
    int64_t n = 0;
    int64_t total = 0;
    int64_t* off = nullptr;        // n+1, by original id
    uint32_t* packed = nullptr;    // total, (hub rank << 8) | dist, rows sorted by hub
    uint32_t* hub = nullptr;       // total
    uint8_t* dist = nullptr;       // total
    int32_t* order = nullptr;      // n, rank -> id
    int32_t max_dist = 0;
    int32_t rounds = 0;
    int64_t bytes = 0;
    plb_build_stats stats{};
    void* shared = nullptr;        // storage shared by the sets of one batched build
};

namespace plb {

// Stream-ordered allocation from the library's per-device pool (freed with
// cudaFreeAsync, or cudaFree after synchronising).
cudaError_t dev_alloc(void** p, size_t bytes, cudaStream_t s);

// Device-wide exclusive scan of int64 values; out may alias in.
// count(i) is evaluated for i in [0, n) and out[n] receives the total.
cudaError_t exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, int64_t* block_sums,
                               cudaStream_t s, const int* skip = nullptr, int64_t align = 1);
int64_t scan_scratch_elems(int64_t n);
int scan_launch_count(int64_t n);

}  // namespace plb
