// Batched 2-hop distance queries (Sec. 2.1):
//   Dis(s, t) = min over hubs h in L(s) and L(t) of d(s,h) + d(h,t).
// One warp per pair.  The 32 highest-ranked hubs of both rows, compared in
// registers, give an upper bound `best` that is usually the answer or next to
// it.  A smaller sum has an entry of at most (best - 1) / 2 on one of its
// sides: both rows are streamed once, entries that near are collected, and only
// full warps of these are looked up in the other row by binary search (on
// R-MAT 2^22, 750 entries per row, 27 of them at distance 1, about 60 of 750
// searches remain).  Pairs whose shorter row has up to 96 entries look all of
// them up at once instead, up to three per lane (fewer instructions than
// streaming both rows).  Bound by instruction issue and the searches' dependent
// loads; when every entry was searched, 32 at a time, 65,536 pairs took 471 us
// on R-MAT 2^22 (now 220), 86 us on directed R-MAT 2^18 (49), and a million
// pairs over 33 sets 490 us (340).
#include <algorithm>

#include "plb_internal.cuh"

namespace plb {
namespace {

constexpr int kQThreads = 128;  // (pairs differ in cost: a block waits for its slowest warp)
constexpr int kMaxSets = 128;
constexpr int kShortRow = 3;  // shorter row up to 32 x this: every entry is looked up
constexpr int kNearWords = 160;  // near entries of a warp: fewer than 32 kept, 128 read

struct SetDesc {
    const int64_t* off;
    const uint32_t* packed;
    int64_t n;
};

struct SetTable {
    SetDesc s[kMaxSets];
};

// Smallest sum (at most 510, or kEmpty) of the entry x of one row (kEmpty: none)
// with its hub's entry in the other row ent[0, len).
__device__ __forceinline__ uint32_t look_up(uint32_t x, const uint32_t* ent, int len) {
    if (x == kEmpty) return kEmpty;
    const uint32_t key = pack(hub_of(x), 0);
    int lo = 0, hi = len;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (ent[mid] < key) lo = mid + 1; else hi = mid;
    }
    if (lo >= len) return kEmpty;
    const uint32_t y = ent[lo];
    return hub_of(y) == hub_of(x) ? dist_of(x) + dist_of(y) : kEmpty;
}

// Smallest sum of the entries of row a[0, al) with their hubs' entries in row
// b[0, bl): up to K entries per lane (al <= 32 K), searched side by side.
template <int K>
__device__ __forceinline__ uint32_t look_up_all(const uint32_t* a, int al, const uint32_t* b, int bl) {
    const int lane = threadIdx.x & 31;
    uint32_t x[K];
    int pos[K];
#pragma unroll
    for (int u = 0; u < K; ++u) {
        x[u] = 32 * u + lane < al ? a[32 * u + lane] : kEmpty;
        pos[u] = 0;
    }
    for (int step = 1 << (31 - __clz(bl)); step > 0; step >>= 1) {
#pragma unroll
        for (int u = 0; u < K; ++u) {
            const int q = pos[u] + step;
            if (q <= bl && b[q - 1] < (x[u] & ~0xFFu)) pos[u] = q;
        }
    }
    uint32_t best = kEmpty;
#pragma unroll
    for (int u = 0; u < K; ++u) {
        const uint32_t y = pos[u] < bl ? b[pos[u]] : 0u;
        // (rows never hold hub kEmpty >> 8)
        if (pos[u] < bl && hub_of(y) == hub_of(x[u])) best = min(best, dist_of(x[u]) + dist_of(y));
    }
    return __reduce_min_sync(kFull, best);
}

// Rows: s in the set (off_s, ent_s), t in (off_t, ent_t); the same set for
// undirected labels, L_out and L_in for directed ones (d(s -> t)).
__device__ __forceinline__ int32_t answer_pair2(const int64_t* off_s, const uint32_t* ent_s, const int64_t* off_t,
                                                const uint32_t* ent_t, int64_t n, int32_t s, int32_t t, uint32_t* buf) {
    if (s < 0 || t < 0 || (int64_t)s >= n || (int64_t)t >= n) return PLB_BAD_PAIR;
    const int lane = threadIdx.x & 31;
    const int64_t ab = off_s[s], ae = off_s[s + 1], bb = off_t[t], be = off_t[t + 1];
    const uint32_t* a = ent_s + ab;
    const uint32_t* b = ent_t + bb;
    int al = (int)(ae - ab), bl = (int)(be - bb);  // (a row has at most n < 2^24 entries)
    if (al > bl) {
        const uint32_t* e = a;
        a = b;
        b = e;
        const int x = al;
        al = bl;
        bl = x;
    }
    // short rows (at least one entry each: the vertex itself)
    if (al <= 32 * kShortRow) {
        const uint32_t m = al <= 32 ? look_up_all<1>(a, al, b, bl) : al <= 64 ? look_up_all<2>(a, al, b, bl)
                                                                             : look_up_all<kShortRow>(a, al, b, bl);
        return m == kEmpty ? PLB_UNREACHABLE : (int32_t)m;
    }
    // the first 32 hubs of both rows (each longer): lane i's hub of a among b's lanes
    const uint32_t x = a[lane], y = b[lane];
    int k = 0;  // largest lane with y <= x's hub at any distance
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
        const uint32_t z = __shfl_sync(kFull, y, k + step);
        if (z <= (x | 0xFFu)) k += step;
    }
    const uint32_t z = __shfl_sync(kFull, y, k);
    uint32_t best = __reduce_min_sync(kFull, hub_of(z) == hub_of(x) ? dist_of(x) + dist_of(z) : kEmpty);
    if (best > 1) {  // (a sum of 0 or 1 is the distance)
        // near entries of a, then of b, looked up in the other row, 32 at a
        // time from the end of buf (its first na are a's)
        const unsigned lt = (1u << lane) - 1u;
        int nf = 0, na = 0;
        auto flush = [&](int cnt) {
            nf -= cnt;
            const int i = nf + lane;
            const uint32_t e = lane < cnt ? buf[i] : kEmpty;
            const bool of_a = i < na;
            best = min(best, __reduce_min_sync(kFull, look_up(e, of_a ? b : a, of_a ? bl : al)));
            na = min(na, nf);
        };
#pragma unroll 1
        for (int side = 0; side < 2 && best > 2; ++side) {
            const uint32_t* row = side ? b : a;
            const int len = side ? bl : al;
            // the first 32 entries up to the other row's 32nd have been compared
            const uint32_t seen = __shfl_sync(kFull, side ? x : y, 31) | 0xFFu;
#pragma unroll 1
            for (int j0 = 0; j0 < len && best > 2; j0 += 128) {
                uint32_t e[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) e[u] = j0 + 32 * u + lane < len ? row[j0 + 32 * u + lane] : kEmpty;
                const uint32_t reach = min((best - 1u) >> 1, 254u);  // (no common hub yet: every entry)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const bool take = dist_of(e[u]) <= reach && (u > 0 || j0 > 0 || e[u] > seen);
                    const unsigned m = __ballot_sync(kFull, take);
                    if (take) buf[nf + __popc(m & lt)] = e[u];
                    nf += __popc(m);
                }
                if (side == 0) na = nf;
                __syncwarp();
                while (nf >= 32 && best > 2) flush(32);
                __syncwarp();
            }
            if (side == 0 && best == kEmpty) {
                // no entry so far has its hub in the other row: with the rest of
                // the shorter row looked up too, none has
                if (nf > 0) flush(nf);
                if (best == kEmpty) break;
            }
        }
        if (nf > 0 && best > 2) flush(min(nf, 32));
        // below 2 only the rows' own vertices (distance 0, the last entries) can go
        if (best == 2) {
            const uint32_t e = lane == 0 ? a[al - 1] : lane == 1 ? b[bl - 1] : kEmpty;
            best = min(best, __reduce_min_sync(kFull, look_up(e, lane == 0 ? b : a, lane == 0 ? bl : al)));
        }
        __syncwarp();
    }
    return best == kEmpty ? PLB_UNREACHABLE : (int32_t)best;
}

__device__ __forceinline__ int32_t answer_pair(const int64_t* off, const uint32_t* ent, int64_t n, int32_t s,
                                               int32_t t, uint32_t* buf) {
    return answer_pair2(off, ent, off, ent, n, s, t, buf);
}

__global__ void __launch_bounds__(kQThreads) k_query2(const int64_t* off_s, const uint32_t* ent_s,
                                                      const int64_t* off_t, const uint32_t* ent_t, int64_t n,
                                                      const int32_t* pairs, int64_t q, int32_t* out) {
    __shared__ uint32_t bufs[kQThreads / 32][kNearWords];
    uint32_t* buf = bufs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < q; i += nw) {
        const int32_t r = answer_pair2(off_s, ent_s, off_t, ent_t, n, pairs[2 * i], pairs[2 * i + 1], buf);
        if (lane == 0) out[i] = r;
    }
}

__global__ void __launch_bounds__(kQThreads) k_query(const int64_t* off, const uint32_t* ent, int64_t n,
                                                     const int32_t* pairs, int64_t q, int32_t* out) {
    __shared__ uint32_t bufs[kQThreads / 32][kNearWords];
    uint32_t* buf = bufs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < q; i += nw) {
        const int32_t s = pairs[2 * i], t = pairs[2 * i + 1];
        const int32_t r = answer_pair(off, ent, n, s, t, buf);
        if (lane == 0) out[i] = r;
    }
}

__global__ void __launch_bounds__(kQThreads) k_query_multi(SetTable tab, int set_lo, int set_hi, int64_t m,
                                                           const int32_t* set_idx, const int32_t* pairs, int64_t q,
                                                           int32_t* out) {
    __shared__ uint32_t bufs[kQThreads / 32][kNearWords];
    uint32_t* buf = bufs[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < q; i += nw) {
        const int32_t k = set_idx[i];
        if (k < 0 || (int64_t)k >= m) {
            if (set_lo == 0 && lane == 0) out[i] = PLB_BAD_PAIR;
            continue;
        }
        if (k < set_lo || k >= set_hi) continue;
        const SetDesc& d = tab.s[k - set_lo];
        const int32_t r = answer_pair(d.off, d.packed, d.n, pairs[2 * i], pairs[2 * i + 1], buf);
        if (lane == 0) out[i] = r;
    }
}

int query_grid(int64_t q) {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 132;
    }
    int64_t blocks = (q * 32 + kQThreads - 1) / kQThreads;
    const int64_t cap = (int64_t)sms * 64;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

}  // namespace
}  // namespace plb

extern "C" int plb_query_batch(const plb_labels* L, const int32_t* pairs, int64_t q, int32_t* dist_out,
                               plb_stream stream) {
    if (!L || q < 0 || (q > 0 && (!pairs || !dist_out))) return PLB_ERR_INVALID;
    if (q == 0) return PLB_OK;
    (void)cudaGetLastError();
    plb::k_query<<<plb::query_grid(q), plb::kQThreads, 0, (cudaStream_t)stream>>>(L->off, L->packed, L->n, pairs, q,
                                                                                  dist_out);
    return cudaGetLastError() == cudaSuccess ? PLB_OK : PLB_ERR_CUDA;
}

extern "C" int plb_query_directed(const plb_labels* L_out, const plb_labels* L_in, const int32_t* pairs, int64_t q,
                                  int32_t* dist_out, plb_stream stream) {
    if (!L_out || !L_in || L_out->n != L_in->n || q < 0 || (q > 0 && (!pairs || !dist_out))) return PLB_ERR_INVALID;
    if (q == 0) return PLB_OK;
    (void)cudaGetLastError();
    plb::k_query2<<<plb::query_grid(q), plb::kQThreads, 0, (cudaStream_t)stream>>>(
        L_out->off, L_out->packed, L_in->off, L_in->packed, L_out->n, pairs, q, dist_out);
    return cudaGetLastError() == cudaSuccess ? PLB_OK : PLB_ERR_CUDA;
}

extern "C" int plb_query_multi(const plb_labels* const* sets, int64_t m, const int32_t* set_idx, const int32_t* pairs,
                               int64_t q, int32_t* dist_out, plb_stream stream) {
    if (m < 0 || q < 0 || (m > 0 && !sets) || (q > 0 && (!pairs || !dist_out || !set_idx))) return PLB_ERR_INVALID;
    for (int64_t k = 0; k < m; ++k)
        if (!sets[k]) return PLB_ERR_INVALID;
    if (q == 0) return PLB_OK;
    (void)cudaGetLastError();
    const int grid = plb::query_grid(q);
    for (int64_t lo = 0; lo < std::max<int64_t>(m, 1); lo += plb::kMaxSets) {
        plb::SetTable tab{};
        const int64_t hi = std::min<int64_t>(m, lo + plb::kMaxSets);
        for (int64_t k = lo; k < hi; ++k) tab.s[k - lo] = {sets[k]->off, sets[k]->packed, sets[k]->n};
        plb::k_query_multi<<<grid, plb::kQThreads, 0, (cudaStream_t)stream>>>(tab, (int)lo, (int)hi, m, set_idx, pairs,
                                                                              q, dist_out);
        if (cudaGetLastError() != cudaSuccess) return PLB_ERR_CUDA;
    }
    return PLB_OK;
}
