// Degree order (Sec. 6.1: vertices ordered by degree, the heuristic of the
// original PLL): rank -> id with degree descending and ties by smaller id.
// Up to kBitonicMax vertices, and without scratch of its own (the allocation-free
// entry point), a bitonic network over unique keys (0x7FFFFFFF - degree) << 32 |
// id; beyond, a stable radix sort by degree that starts in id order.
#include <algorithm>

#include "plb_internal.cuh"

namespace plb {
namespace {

constexpr int kSortTile = 2048;
constexpr int kSortThreads = 1024;
// The radix sort's 15 launches take 60 to 70 us however few the vertices; the
// bitonic network pads to a power of two: 2,049 to 4,096 vertices 41-43 us (radix
// 60-66), up to 8,192 59 us (62-70), up to 16,384 80 us (62-70).
constexpr int64_t kBitonicMax = 8192;

__global__ void k_deg_keys(const int64_t* row_ptr, int64_t n, int64_t n2, uint64_t* keys) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
        uint64_t k = ~0ull;
        if (i < n) {
            const int64_t deg = row_ptr[i + 1] - row_ptr[i];
            k = ((uint64_t)(0x7FFFFFFFll - deg) << 32) | (uint64_t)i;
        }
        keys[i] = k;
    }
}

__device__ __forceinline__ void cswap(uint64_t* a, int i, int l, bool up) {
    const uint64_t x = a[i], y = a[l];
    if ((x > y) == up) {
        a[i] = y;
        a[l] = x;
    }
}

// Full bitonic sort of each tile (stages k = 2 .. tile), directions taken
// from the global index so that the tiles feed the global merge stages.
__global__ void __launch_bounds__(kSortThreads) k_sort_tiles(uint64_t* keys, int tile) {
    __shared__ uint64_t sk[kSortTile];
    const int64_t base = (int64_t)blockIdx.x * tile;
    for (int i = threadIdx.x; i < tile; i += blockDim.x) sk[i] = keys[base + i];
    __syncthreads();
    for (int k = 2; k <= tile; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int i = threadIdx.x; i < tile; i += blockDim.x) {
                const int l = i ^ j;
                if (l > i) cswap(sk, i, l, ((base + i) & k) == 0);
            }
            __syncthreads();
        }
    }
    for (int i = threadIdx.x; i < tile; i += blockDim.x) keys[base + i] = sk[i];
}

// One global compare-exchange step (stride j >= tile) of merge stage k.
__global__ void k_sort_global_step(uint64_t* keys, int64_t n2, int64_t j, int64_t k) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n2; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = i ^ j;
        if (l > i) {
            const uint64_t x = keys[i], y = keys[l];
            const bool up = (i & k) == 0;
            if ((x > y) == up) {
                keys[i] = y;
                keys[l] = x;
            }
        }
    }
}

// Remaining strides j < tile of merge stage k, inside each tile.
__global__ void __launch_bounds__(kSortThreads) k_sort_tile_merge(uint64_t* keys, int tile, int64_t k) {
    __shared__ uint64_t sk[kSortTile];
    const int64_t base = (int64_t)blockIdx.x * tile;
    for (int i = threadIdx.x; i < tile; i += blockDim.x) sk[i] = keys[base + i];
    __syncthreads();
    for (int j = tile >> 1; j > 0; j >>= 1) {
        for (int i = threadIdx.x; i < tile; i += blockDim.x) {
            const int l = i ^ j;
            if (l > i) cswap(sk, i, l, ((base + i) & k) == 0);
        }
        __syncthreads();
    }
    for (int i = threadIdx.x; i < tile; i += blockDim.x) keys[base + i] = sk[i];
}

__global__ void k_keys_to_order(const uint64_t* keys, int64_t n, int32_t* order) {
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
        order[r] = (int32_t)(keys[r] & 0xFFFFFFFFull);
}

// ------------------------------------------------------------ radix sort
// LSD passes over the four bytes of 0x7FFFFFFF - degree, each stable: a count
// pass makes a (digit, tile) histogram, its exclusive scan in digit-major order
// gives every tile its first place per digit, and a scatter pass writes each
// entry there plus its rank among the tile's earlier equal digits.  Passes whose
// digit is the same everywhere (the high ones: degrees are small) do nothing;
// `moved` counts the others, so every pass finds its input.  Bound by memory and
// the scattered writes: 4.0M vertices take 1,894 us in the bitonic network (77
// passes over the keys) and 164 us here.
constexpr int kRadixTile = 4096;
constexpr int kRadixThreads = 256;
constexpr int kRadixWarps = kRadixThreads / 32;
constexpr int kRadixItems = kRadixTile / kRadixThreads;  // per lane, 32 consecutive entries per step of a warp

__device__ __forceinline__ uint32_t degree_key(const int64_t* row_ptr, int64_t i) {
    return (uint32_t)(0x7FFFFFFFll - (row_ptr[i + 1] - row_ptr[i]));
}

// Entry i: key << 32 | id (pass 0 makes it from the row offsets).
__device__ __forceinline__ uint64_t radix_entry(const int64_t* row_ptr, const uint64_t* src, int64_t i) {
    return src ? src[i] : ((uint64_t)degree_key(row_ptr, i) << 32) | (uint64_t)i;
}

// varying: the bits in which some keys differ.
__global__ void __launch_bounds__(kRadixThreads) k_radix_varying(const int64_t* row_ptr, int64_t n, uint32_t* varying) {
    const uint32_t first = degree_key(row_ptr, 0);
    uint32_t x = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x |= degree_key(row_ptr, i) ^ first;
    x = __reduce_or_sync(kFull, x);
    if ((threadIdx.x & 31) == 0 && x) atomicOr(varying, x);
}

// Whether pass p moves entries, and where its input is (the passes before it that
// moved alternate between the two buffers; none: the row offsets).
__device__ __forceinline__ bool radix_pass(uint32_t varying, int p, uint64_t* buf0, uint64_t* buf1, const uint64_t** src,
                                           uint64_t** dst) {
    int moved = 0;
    for (int q = 0; q < p; ++q) moved += ((varying >> (8 * q)) & 0xFFu) ? 1 : 0;
    *src = moved == 0 ? nullptr : (moved & 1) ? buf0 : buf1;
    *dst = (moved & 1) ? buf1 : buf0;
    return ((varying >> (8 * p)) & 0xFFu) != 0u;
}

__global__ void __launch_bounds__(kRadixThreads) k_radix_count(const int64_t* row_ptr, int64_t n, uint64_t* buf0,
                                                               uint64_t* buf1, const uint32_t* varying, int p,
                                                               int64_t tiles, int64_t* hist) {
    __shared__ int h[256];
    const uint64_t* src;
    uint64_t* dst;
    const bool moves = radix_pass(*varying, p, buf0, buf1, &src, &dst);
    if (!moves) return;
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kRadixTile;
    for (int k = 0; k < kRadixItems; ++k) {
        const int64_t i = base + k * kRadixThreads + threadIdx.x;
        if (i < n) atomicAdd(&h[(uint32_t)(radix_entry(row_ptr, src, i) >> (32 + 8 * p)) & 0xFFu], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

__global__ void __launch_bounds__(kRadixThreads) k_radix_scatter(const int64_t* row_ptr, int64_t n, uint64_t* buf0,
                                                                 uint64_t* buf1, const uint32_t* varying, int p,
                                                                 int64_t tiles, const int64_t* place) {
    __shared__ int64_t at[kRadixWarps][256];  // next place of each warp per digit
    const uint64_t* src;
    uint64_t* dst;
    if (!radix_pass(*varying, p, buf0, buf1, &src, &dst)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const unsigned lt = (1u << lane) - 1u;
    for (int q = 0; q < kRadixWarps; ++q) at[q][threadIdx.x] = 0;
    __syncthreads();
    // warp w holds the tile's w-th run of entries, in order
    const int64_t base = (int64_t)blockIdx.x * kRadixTile + (int64_t)w * (kRadixItems * 32);
    uint64_t e[kRadixItems];
    unsigned dg[kRadixItems], peers[kRadixItems];
#pragma unroll
    for (int k = 0; k < kRadixItems; ++k) {
        const int64_t i = base + 32 * k + lane;
        e[k] = i < n ? radix_entry(row_ptr, src, i) : ~0ull;
        dg[k] = i < n ? (unsigned)(e[k] >> (32 + 8 * p)) & 0xFFu : 256u;
    }
#pragma unroll
    for (int k = 0; k < kRadixItems; ++k) {
        peers[k] = __match_any_sync(kFull, dg[k]);
        if (dg[k] < 256u && (peers[k] & lt) == 0u) at[w][dg[k]] += __popc(peers[k]);
        __syncwarp();
    }
    __syncthreads();
    {  // digit threadIdx.x: the warps' counts to places
        int64_t run = place[(int64_t)threadIdx.x * tiles + blockIdx.x];
        for (int q = 0; q < kRadixWarps; ++q) {
            const int64_t c = at[q][threadIdx.x];
            at[q][threadIdx.x] = run;
            run += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kRadixItems; ++k) {
        int64_t to = 0;
        if (dg[k] < 256u) to = at[w][dg[k]] + __popc(peers[k] & lt);
        __syncwarp();
        if (dg[k] < 256u) {
            dst[to] = e[k];
            if ((peers[k] & lt) == 0u) at[w][dg[k]] += __popc(peers[k]);
        }
        __syncwarp();
    }
}

__global__ void k_radix_order(int64_t n, uint64_t* buf0, uint64_t* buf1, const uint32_t* varying, int32_t* order) {
    const uint64_t* src;
    uint64_t* dst;
    radix_pass(*varying, 4, buf0, buf1, &src, &dst);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        order[i] = src ? (int32_t)(src[i] & 0xFFFFFFFFull) : (int32_t)i;
}

// Scratch of the radix sort in 8-byte words: two entry buffers, the histogram
// with its total, the scan's scratch, the varying bits.
int64_t radix_scratch_words(int64_t n) {
    const int64_t bins = 256 * ((n + kRadixTile - 1) / kRadixTile);
    return 2 * n + bins + 1 + scan_scratch_elems(bins) + 1;
}

cudaError_t degree_order_radix(const int64_t* row_ptr, int64_t n, int32_t* order, uint64_t* scratch, cudaStream_t s) {
    const int64_t tiles = (n + kRadixTile - 1) / kRadixTile, bins = 256 * tiles;
    uint64_t *buf0 = scratch, *buf1 = scratch + n;
    int64_t* hist = reinterpret_cast<int64_t*>(scratch + 2 * n);
    int64_t* scan = hist + bins + 1;
    uint32_t* varying = reinterpret_cast<uint32_t*>(scan + scan_scratch_elems(bins));
    cudaError_t e = cudaMemsetAsync(varying, 0, sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    const unsigned flat = (unsigned)std::min<int64_t>((n + 1023) / 1024, 2048);
    k_radix_varying<<<flat, kRadixThreads, 0, s>>>(row_ptr, n, varying);
    for (int p = 0; p < 4; ++p) {
        k_radix_count<<<(unsigned)tiles, kRadixThreads, 0, s>>>(row_ptr, n, buf0, buf1, varying, p, tiles, hist);
        // (a pass that moves nothing leaves stale counts: they are scanned and not read)
        e = exclusive_scan_i64(hist, hist, bins, scan, s);
        if (e != cudaSuccess) return e;
        k_radix_scatter<<<(unsigned)tiles, kRadixThreads, 0, s>>>(row_ptr, n, buf0, buf1, varying, p, tiles, hist);
    }
    k_radix_order<<<flat, kRadixThreads, 0, s>>>(n, buf0, buf1, varying, order);
    return cudaGetLastError();
}

}  // namespace

// Sorts keys[0..n2) ascending (n2 a power of two).
cudaError_t bitonic_sort_u64(uint64_t* keys, int64_t n2, cudaStream_t s) {
    const int tile = (int)(n2 < kSortTile ? n2 : kSortTile);
    const int64_t tiles = n2 / tile;
    k_sort_tiles<<<(unsigned)tiles, kSortThreads, 0, s>>>(keys, tile);
    for (int64_t k = 2 * (int64_t)tile; k <= n2; k <<= 1) {
        for (int64_t j = k >> 1; j >= tile; j >>= 1) {
            int64_t blocks = (n2 + 255) / 256;
            if (blocks > 65535) blocks = 65535;
            k_sort_global_step<<<(unsigned)blocks, 256, 0, s>>>(keys, n2, j, k);
        }
        k_sort_tile_merge<<<(unsigned)tiles, kSortThreads, 0, s>>>(keys, tile, k);
    }
    return cudaGetLastError();
}

cudaError_t degree_order_with_scratch(const int64_t* row_ptr, int64_t n, int32_t* order, uint64_t* keys,
                                      int64_t n2, cudaStream_t s) {
    int64_t blocks = (n2 + 255) / 256;
    if (blocks > 65535) blocks = 65535;
    k_deg_keys<<<(unsigned)blocks, 256, 0, s>>>(row_ptr, n, n2, keys);
    cudaError_t e = bitonic_sort_u64(keys, n2, s);
    if (e != cudaSuccess) return e;
    k_keys_to_order<<<(unsigned)blocks, 256, 0, s>>>(keys, n, order);
    return cudaGetLastError();
}

}  // namespace plb

extern "C" int plb_degree_order(const plb_csr* g, int32_t* order_out, plb_stream stream) {
    if (!g || g->n < 0 || (g->n > 0 && (!g->row_ptr || !order_out))) return PLB_ERR_INVALID;
    if (g->n >= PLB_MAX_VERTICES) return PLB_ERR_TOO_LARGE;
    if (g->n == 0) return PLB_OK;
    cudaStream_t s = (cudaStream_t)stream;
    int64_t n2 = 1;
    while (n2 < g->n) n2 <<= 1;
    const bool radix = g->n > plb::kBitonicMax;
    uint64_t* keys = nullptr;
    if (plb::dev_alloc((void**)&keys, sizeof(uint64_t) * (radix ? plb::radix_scratch_words(g->n) : n2), s) !=
        cudaSuccess) {
        (void)cudaGetLastError();
        return PLB_ERR_OOM;
    }
    const cudaError_t e = radix ? plb::degree_order_radix(g->row_ptr, g->n, order_out, keys, s)
                                : plb::degree_order_with_scratch(g->row_ptr, g->n, order_out, keys, n2, s);
    cudaFreeAsync(keys, s);
    return e == cudaSuccess ? PLB_OK : PLB_ERR_CUDA;
}
