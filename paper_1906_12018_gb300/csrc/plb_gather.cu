// Gather + prune kernels of rounds d >= 2 (Alg. 3, Sec. 3.1): for every
// receiver v, the unique messages of round d (hubs h < v of the neighbours'
// frontier rows dL_{d-1}, not already hubs of v) and the distance check of
// each candidate against the labels of round d - 1 (the snapshot: accept
// (h, d) iff no common hub w has d(w, v) + d(w, h) <= d).
//   k_gp_warp   one vertex per warp, tables in shared memory;
//   k_gp_block  one vertex per 256-thread block, any size.
// Both append the accepted hubs to the new frontier in rank order (the block
// tier lists the few vertices whose row it could not sort for the row sort).
// Loops with a run-time trip count are not unrolled: the warps of an SM are at
// different places of these kernels, and code that outgrows the instruction
// caches costs more than the loop control (see witness4).
//
// Measured (builds, hash sets and one check of all candidates -> hub maps, the
// two-step prefilter, the lane/group/warp checks and the bucketed tables -> with
// frontier sectors, split hubs, top-hub columns, the cache's share of shared
// memory and the warp tier's wider bound besides): R-MAT 2^22, 64M edges 1,213 ->
// 834 -> 534 ms; Chung-Lu 2^20 39.1 -> 34.8 -> 21.7 ms; directed R-MAT 2^20
// 185.9 -> 140.9 -> 91 ms.
#include "plb_kernels.cuh"
#include "plb_round.cuh"

namespace plb {
namespace {
__device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
}  // namespace

// Side B of the check (see check_chunk), per tier (measured: side B saves most
// on power-law graphs with heavy hubs in both tiers).
constexpr int kWarpSideBMin = 16, kWarpSideBShift = 1;
constexpr int kBlockSideBMin = 16, kBlockSideBShift = 1;

// 32 bytes of global memory (one sector) in one load; p is 32-byte aligned.
__device__ __forceinline__ void load_sector(const uint32_t* p, uint32_t (&x)[8]) {
    asm("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7])
        : "l"(p));
}

// Top-hub witness prefilter: candidate h has a witness among the kTopHubs
// highest-ranked hubs when E_i(v) & C_j(h) != 0 for some i >= 1,
// j = min(d - i, kTopLevels) >= 1, where E_i(v) (v's hubs at distance exactly
// i) is staged in shared memory (ev, kTopLevels x kTopWords words) and C_j(h)
// is h's cumulative mask.  One level pair (i, j) = one 32-byte mask of h.
static_assert(kTopWords == 8, "a mask is one 32-byte sector");
__device__ __forceinline__ uint32_t top_pair(const uint32_t* top, int64_t n, const uint32_t* ev, int i, int j,
                                             uint32_t h) {
    uint32_t c[8];
    load_sector(top + ((j - 1) * n + h) * kTopWords, c);
    const uint4* e4 = reinterpret_cast<const uint4*>(ev + (i - 1) * kTopWords);
    const uint4 e = e4[0], g = e4[1];
    return (c[0] & e.x) | (c[1] & e.y) | (c[2] & e.z) | (c[3] & e.w) | (c[4] & g.x) | (c[5] & g.y) | (c[6] & g.z) |
           (c[7] & g.w);
}

// The prefilter runs in two steps.  The first tests one level pair (i0, d -
// i0), i0 the smallest distance at which v has a top hub, for two candidates
// per lane at once (independent loads, nothing else in flight behind them):
// it settles most candidates (R-MAT 2^22: 73% in round 2, where it is the
// whole prefilter, and nearly all of round 3's 6.5G).  Only its survivors,
// compacted into full warps, go on to check_chunk, which tests the other
// pairs.  Weighted rounds (many distances, few hubs at each) test every pair
// in the first step.
__device__ __forceinline__ int first_level(const uint32_t* ev, int imax, int lane) {
    int i0 = 1;
#pragma unroll 1
    for (int i = 1; i <= imax; ++i) {
        if (__any_sync(kFull, ev[(i - 1) * kTopWords + (lane & 7)] != 0u)) {
            i0 = i;
            break;
        }
    }
    return i0;
}
__device__ __forceinline__ void prefilter_first(const GpParams& p, const uint32_t* ev, int d, int imax, int i0,
                                                uint32_t h0, bool v0, uint32_t h1, bool v1, unsigned* m0,
                                                unsigned* m1) {
    const int ia = p.sender_bits == 0 ? i0 : 1, ib = p.sender_bits == 0 ? i0 : imax;
    uint32_t x0 = 0, x1 = 0;
#pragma unroll 1
    for (int i = ia; i <= ib; ++i) {
        const int j = min(d - i, kTopLevels);
        if (v0) x0 |= top_pair(p.top_h, p.n, ev, i, j, h0);
        if (v1) x1 |= top_pair(p.top_h, p.n, ev, i, j, h1);
    }
    *m0 = __ballot_sync(kFull, v0 && x0 == 0u);  // the lanes whose candidate goes on
    *m1 = __ballot_sync(kFull, v1 && x1 == 0u);
}

// Stage E_i(v) = C_i(v) & ~C_{i-1}(v), i = 1..kTopLevels, into ev (cooperative:
// thread t of nthr handles words t, t + nthr, ...).
__device__ __forceinline__ void stage_exact_levels(const uint32_t* top, int64_t n, int32_t v, uint32_t* ev, int t,
                                                   int nthr) {
    const uint32_t* tv = top + (int64_t)v * kTopWords;
#pragma unroll 1
    for (int q = t; q < kTopRow; q += nthr) {
        const int lev = q / kTopWords, w = q % kTopWords;
        const uint32_t c = tv[lev * n * kTopWords + w];
        const uint32_t prev = lev > 0 ? tv[(lev - 1) * n * kTopWords + w] : 0u;
        ev[q] = c & ~prev;
    }
}

// Distance check of up to 32 candidates held one per lane (valid lanes).
// A witness for candidate h is a hub w of both v and h with
// d(w,v) + d(w,h) <= d (the test of Alg. 3 with the labels of round d-1).
// Each candidate scans one side:
//   A: the entries of L(h) (its last entry, (h,0), is never a witness and is
//      skipped), each looked up in the hub-keyed table M of L(v) (shared
//      memory, or v's row of the global probe index when mv_global);
//   B: the entries of L(v) with hub < h (only those can be hubs of h), each
//      probed in h's row of the global probe index (rows of >= 16 entries).
// B is considered only for |L(h)| >= b_min (the count of L(v)'s hubs below h
// is a binary search in L(v)'s row) and taken when it is the shorter scan, by
// a factor 2^b_shift against a shared-memory M (whose probes are cheaper
// than the global table's).  Either way a scan is a row of entries and a hash
// table to look them up in, and it ends at its first witness.  Every lane
// first looks up kFirstItems entries of its own candidate (all loads in flight
// at once: most scans end there); longer scans go on eight at a time, four
// lanes and 16 entries per step each, and very long ones on the whole warp.
// Every candidate has passed the first step of the top-hub prefilter (level
// i0; i0 = 0: none yet) and goes through the rest of it here; the whole is
// exact for the kTopHubs highest-ranked hubs while d <= kTopLevels + 1
// (a witness w has 1 <= d(w,v), d(w,h) <= d - 1): for a candidate it does not
// prune, no top hub is a witness, so both scans start past the top hubs
// (L(h)'s count of them comes with h's check record, L(v)'s is tv_top).
// Returns the lanes whose candidate survives.
constexpr int kFirstItems = 4;   // entries of a scan that its own lane looks up
constexpr int kGroupItems = 96;  // longest scan of a group of four lanes

// Looks up the entries ent[j], ent[j + st], ent[j + 2 st], ent[j + 3 st] (those
// below n) in the table tab of 2^tlog slots; true when one of them gives a
// witness, a distance sum of at most d (in rank batches some labels are longer
// than the round).  The four buckets are requested together.  One copy of the
// code: the gather kernels' warps are at different places of it, and the warp
// tier waited for instructions more than for anything else when its code grew
// from 55 to 81 KB.
__device__ __noinline__ bool witness4(const uint32_t* ent, int j, int st, int n, const uint32_t* tab, int tlog,
                                      uint32_t d) {
    uint32_t x[4], sl[4], lim[4];
    uint4 y[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = j + u * st < n ? ent[j + u * st] : kEmpty;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        sl[u] = bslot(hub_of(x[u]), tlog);
        lim[u] = dist_of(x[u]) < d ? d - dist_of(x[u]) : 0u;  // (0: no entry is that near)
        y[u] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        if (x[u] != kEmpty) y[u] = *reinterpret_cast<const uint4*>(tab + sl[u]);
    }
    bool hit = false, full = false;
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        hit = hit || bucket_has(y[u], x[u] & ~0xFFu, lim[u]);
        full = full || y[u].w != kEmpty;
    }
    if (full && !hit) {  // some full bucket without a witness: its chain goes on
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (y[u].w != kEmpty) hit = hit || map_has_from(tab, tlog, sl[u], y[u], x[u] & ~0xFFu, lim[u]);
    }
    return hit;
}
__device__ __forceinline__ unsigned check_chunk(const GpParams& p, uint32_t d, const uint32_t* M, int log_m,
                                                bool mv_global, int b_min, int b_shift, const uint32_t* lv,
                                                int64_t lvlen, int tv_top, uint32_t h, bool valid,
                                                unsigned long long& probed, const uint32_t* tv, int i0,
                                                unsigned long long& prefiltered) {
    const int lane = threadIdx.x & 31;
    const uint32_t* ent = lv;  // scanned entries: A: L(h), B: L(v)
    const uint32_t* tab = M;   // looked up in: A: L(v)'s table, B: h's probe table
    int tlog = log_m, items = 0;
    // h's check record (row bounds and probe-table descriptor: one 16-byte
    // load, one memory sector) is requested before the rest of the top-hub
    // prefilter reads h's masks, so the loads overlap
    uint4 rec = make_uint4(0u, 0u, 0u, 0u);
    if (valid) rec = p.hrec_h[h];
    const int imax = min((int)d - 1, kTopLevels);
    if (i0 == 0 || (p.sender_bits == 0 && imax > 1)) {
        uint32_t hit = 0;
        if (valid)
#pragma unroll 1
            for (int i = 1; i <= imax; ++i)
                if (i != i0) hit |= top_pair(p.top_h, p.n, tv, i, min((int)d - i, kTopLevels), h);
        const unsigned pf = __ballot_sync(kFull, hit != 0);
        if (lane == 0) prefiltered += __popc(pf);
        if (hit) valid = false;
    }
    // past the top hubs when the prefilter settles them (see above)
    const bool skip_top = d <= (uint32_t)kTopLevels + 1u;
    if (valid) {
        const uint64_t row = ((uint64_t)rec.y << 32) | rec.x;
        const int64_t hb = (int64_t)(row >> 24);
        const int la = (int)(row & 0xFFFFFFu) - 1;
        const uint64_t hd = (((uint64_t)rec.w << 32) | rec.z) & kHrecDescMask;
        const int top_h = (int)(rec.w >> kHrecTopShift);  // entries of L(h) with a top hub
        const int sa = skip_top ? min(top_h, la) : 0;  // side A starts past L(h)'s top hubs
        ent = p.lent_h + hb + sa;
        items = la - sa;
        if (la >= b_min && hd) {
            const int lb = (int)lower_bound_u32(lv, lvlen, pack(h, 0));
            const int sb = skip_top ? min(tv_top, lb) : 0;  // side B starts past L(v)'s top hubs
            if (mv_global ? lb - sb < la - sa : ((lb - sb) << b_shift) < la - sa) {
                items = lb - sb;
                ent = lv + sb;
                tab = p.htab_h + (hd >> 8);
                tlog = (int)(hd & 0xFFu);
            }
        }
    }
    bool alive = valid;
    if (items > 0) {
        alive = !witness4(ent, 0, 1, min(items, kFirstItems), tab, tlog, d);
        probed += (unsigned)min(items, kFirstItems);
    }
    // scans of up to kGroupItems entries: group g of four lanes takes the g-th
    unsigned todo = __ballot_sync(kFull, alive && items > kFirstItems && items <= kGroupItems);
#pragma unroll 1
    while (todo) {
        const unsigned batch = todo;
        int k = -1;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
            if ((lane >> 2) == g) k = __ffs(todo) - 1;
            todo &= todo - 1u;
        }
        const int src = k < 0 ? lane : k;
        const uint32_t* ek = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)ent, src));
        const uint32_t* tk = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)tab, src));
        int nk = __shfl_sync(kFull, items, src);
        const int lk = __shfl_sync(kFull, tlog, src);
        if (k < 0) nk = 0;
        unsigned won = 0;  // lanes of the groups that found a witness
#pragma unroll 1
        for (int j = kFirstItems + (lane & 3); __any_sync(kFull, j < nk); j += 16) {
            const bool hit = j < nk && witness4(ek, j, 4, nk, tk, lk, d);
            const unsigned hm = __ballot_sync(kFull, hit);
            probed += (unsigned)min(4, (max(nk - j, 0) + 3) / 4);
            if ((hm >> (lane & ~3)) & 0xFu) nk = 0;
            won |= hm;
        }
        const int g = __popc(batch & ((1u << lane) - 1u));  // this lane's candidate is the batch's g-th
        if (((batch >> lane) & 1u) && g < 8 && ((won >> (4 * g)) & 0xFu)) alive = false;
    }
    // longer scans: one candidate at a time, 128 entries per step
    todo = __ballot_sync(kFull, alive && items > kGroupItems);
#pragma unroll 1
    while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1u;
        const uint32_t* ek = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)ent, k));
        const uint32_t* tk = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)tab, k));
        const int nk = __shfl_sync(kFull, items, k), lk = __shfl_sync(kFull, tlog, k);
#pragma unroll 1
        for (int j = kFirstItems + lane; j - lane < nk; j += 128) {
            probed += (unsigned)min(4, (max(nk - j, 0) + 31) / 32);
            if (__any_sync(kFull, j < nk && witness4(ek, j, 32, nk, tk, lk, d))) {
                if (lane == k) alive = false;
                break;
            }
        }
    }
    return __ballot_sync(kFull, alive);
}

// The cost model's reads of one candidate's check (profiled builds): L(v)'s
// entries below h, and L(h).
__device__ __noinline__ void count_reads(const int64_t* loff_h, const uint32_t* lv, int64_t lvlen, uint32_t h,
                                         unsigned long long* chk) {
    chk[0] += (unsigned long long)lower_bound_u32(lv, lvlen, pack(h, 0));
    chk[1] += (unsigned long long)(loff_h[h + 1] - loff_h[h]);
}

// The same for the candidates hb + b, b the bits of c, with one search for all of
// them (one each: 1,330 instead of 650 ms for a profiled build of R-MAT 2^22).
__device__ __noinline__ void count_reads64(const int64_t* loff, const uint32_t* lv, int64_t lvlen, uint32_t hb,
                                           unsigned long long c, unsigned long long* cnt) {
    if (c == 0) return;
    int64_t at = lower_bound_u32(lv, lvlen, pack(hb, 0));
    cnt[0] += (unsigned long long)at * (unsigned)__popcll(c);
#pragma unroll 1
    for (; at < lvlen && hub_of(lv[at]) - hb < 64u; ++at)
        cnt[0] += (unsigned)__popcll(c >> (hub_of(lv[at]) - hb) >> 1);  // candidates past this hub
#pragma unroll 1
    for (; c; c &= c - 1) {
        const int64_t* l = loff + hb + (__ffsll((long long)c) - 1);
        cnt[1] += (unsigned long long)(l[1] - l[0]);
    }
}

// Warp tier: gather of v's messages (hubs below v of the neighbours' frontier
// rows; the rows are sorted, so each row's share is found by binary search).
// Hubs below vb + W are marked in the bitmap X, the others go into the set S
// (cleared when the first of them arrives).  Warp-level load-balanced expansion
// over 32 neighbours at a time, each step's load issued before the hubs of the
// step before it are used.  *top: one past the highest hub marked, from vb.
// Returns false when the set would exceed `limit` entries.
__device__ __forceinline__ bool gather_range(const GpParams& p, int64_t nb, int64_t ne, uint32_t v, uint32_t vb,
                                             uint32_t W, uint32_t* X, uint32_t* S, int log_s, int limit, int* cnt_sm,
                                             uint32_t* top, unsigned long long& msgs) {
    const int lane = threadIdx.x & 31;
    uint32_t hmax = 0;
    bool clean = false;
#pragma unroll 1
    for (int64_t base = nb; base < ne; base += 32) {
        const int64_t j = base + lane;
        int c = 0;
        int64_t st = 0;
        if (j < ne) {
            const int32_t a = p.rcol[j];
            const uint64_t f = p.fse[a];
            const uint32_t n0 = fcount(f);
            if (n0) {
                // the hubs of a frontier row of sender a are <= a (a itself
                // only in round 0): for a < v the whole row lies below v
                st = (int64_t)fstart(f);
                c = sender_of(p, a) < v ? (int)n0 : (int)lower_bound_u32(p.fhub + st, n0, v);
            }
        }
        const int incl = warp_incl_scan(c, lane);
        const int total = __shfl_sync(kFull, incl, 31);
        const int excl = incl - c;
        const uint32_t* row = p.fhub + (st - excl);  // message i of the tile, in this lane's row, is row[i]
        msgs += (lane == 0) ? (unsigned long long)total : 0ull;
        uint32_t h = kEmpty;
#pragma unroll 1
        for (int ib = 0; ib < total + 32; ib += 32) {
            const int it = ib + lane;
            const int k = warp_owner(excl, it);
            const uint32_t* rk = reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)row, k));
            const uint32_t hn = it < total ? rk[it] : kEmpty;
            const uint32_t hr = h - vb;
            if (hr < W) {
                // (a set bit is not set again: in dense graphs the lanes of a
                // step share few words, and atomics on one word take turns)
                if (!((X[hr >> 5] >> (hr & 31)) & 1u)) atomicOr(&X[hr >> 5], 1u << (hr & 31));
                hmax = max(hmax, hr + 1u);
            }
            const bool big = h != kEmpty && hr >= W;
            if (__any_sync(kFull, big)) {
                if (!clean) {
#pragma unroll 1
                    for (int s = lane; s < (1 << log_s); s += 32) S[s] = kEmpty;
                    clean = true;
                    __syncwarp();
                }
                int nins = 0;
                if (big) nins = set_insert(S, log_s, h) ? 1 : 0;
                nins = __popc(__ballot_sync(kFull, nins));
                if (lane == 0) *cnt_sm += nins;
                __syncwarp();
                if (*(volatile int*)cnt_sm > limit) return false;
            }
            h = hn;
        }
    }
    *top = __reduce_max_sync(kFull, hmax);
    return true;
}

// Block-wide exclusive scan of one int per thread (blockDim <= 1024);
// wsum is shared scratch of 32 ints.  Returns the thread's exclusive prefix
// and the block total in *total.
__device__ __forceinline__ int block_excl_scan(int x, int* wsum, int* total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    const int incl = warp_incl_scan(x, lane);
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    if (wid == 0) {
        const int w = lane < nw ? wsum[lane] : 0;
        const int wi = warp_incl_scan(w, lane);
        wsum[lane] = wi - w;
        if (lane == 31) wsum[32] = wi;
    }
    __syncthreads();
    const int r = wsum[wid] + incl - x;
    *total = wsum[32];
    return r;
}

// Shrink the hub range of a pass whose set overflowed: histogram the keys of
// S below hi over 256 buckets of [lo, hi) and cut hi at the first bucket where
// the running count would pass half the capacity.  The kept count is read off
// the histogram; when it fits (always, unless the first bucket alone is too
// full, then the range is narrowed to that bucket and the histogram redone,
// keys at or above hi being ignored), S is rebuilt from the kept keys (C is
// scratch).  All threads call; returns with *hi_sm and *cnt_sm set.
__device__ void shrink_pass(uint32_t* S, int log_s, uint32_t* C, int limit, uint32_t lo, uint32_t* hi_sm,
                            int* cnt_sm, int* hist, int* tmp) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int S_CAP = 1 << log_s;
#pragma unroll 1
    while (true) {
        const uint32_t hi = *(volatile uint32_t*)hi_sm;
        const uint32_t bw = (hi - lo + 255u) / 256u;
#pragma unroll 1
        for (int b = tid; b < 256; b += nthr) hist[b] = 0;
        __syncthreads();
#pragma unroll 1
        for (int sl = tid; sl < S_CAP; sl += nthr) {
            const uint32_t key = S[sl];
            if (key != kEmpty && key < hi) atomicAdd(&hist[(key - lo) / bw], 1);
        }
        __syncthreads();
        if (tid == 0) {
            int cum = 0, b = 0;
#pragma unroll 1
            while (b < 255 && cum + hist[b] <= limit / 2) cum += hist[b++];
            if (b == 0) {  // the first bucket alone passes half the capacity: keep it whole
                b = 1;
                cum = hist[0];
            }
            uint32_t nh = lo + (uint32_t)b * bw;
            if (nh > hi) nh = hi;
            *hi_sm = nh;
            tmp[0] = cum;  // keys below nh
            tmp[1] = 0;
        }
        __syncthreads();
        const uint32_t nh = *(volatile uint32_t*)hi_sm;
        const int kept = *(volatile int*)&tmp[0];
        if (kept > limit) continue;  // narrow further (S untouched; keys >= nh are ignored)
#pragma unroll 1
        for (int sl = tid; sl < S_CAP; sl += nthr) {
            const uint32_t key = S[sl];
            if (key != kEmpty && key < nh) C[atomicAdd(&tmp[1], 1)] = key;
        }
        __syncthreads();
#pragma unroll 1
        for (int sl = tid; sl < S_CAP; sl += nthr) S[sl] = kEmpty;
        __syncthreads();
#pragma unroll 1
        for (int q = tid; q < kept; q += nthr) set_insert(S, log_s, C[q]);
        if (tid == 0) *cnt_sm = kept;
        __syncthreads();
        return;
    }
}

// A hub past the map: into the set S, unless it is in L(v) (M) or the set is
// full (*ovf_sm).  Returns 1 when it is new.
__device__ __noinline__ int set_add(uint32_t* S, int log_s, const uint32_t* M, int log_m, int limit,
                                    volatile int* cnt_sm, volatile int* ovf_sm, uint32_t h) {
    if (M && map_has(M, log_m, h)) return 0;
    if (*cnt_sm >= limit) {
        *ovf_sm = 1;
        return 0;
    }
    return set_insert(S, log_s, h) ? 1 : 0;
}

// Block-wide load-balanced gather of v's messages with hub in [lo, *hi_sm):
// hubs below vb + W (vb: the first rank of v's graph) are marked in the map B
// (a bit each; L(v)'s hubs are cleared afterwards; looking first whether the bit
// is set already, as the warp tier does, made R-MAT 2^22 2% slower: the lanes of
// a step read different sectors and seldom meet in a word), the others go into
// the set S.  Neighbours are taken in tiles of blockDim; each
// thread finds the sectors (eight hubs) of its neighbour's row dL_{d-1}(a) that
// overlap the range (the row is sorted), a block-wide exclusive scan of their
// counts assigns every warp an equal, contiguous share, and every lane reads
// one sector per step: the search for a lane's row, 20 instructions, then
// serves eight messages instead of one (R-MAT 2^22 took 134 + 72 ms of warp
// time in rounds 2 and 3 to gather its 52G messages one per lane).  When the
// set would exceed `limit`, its range (hubs >= vb + W) is shrunk (shrink_pass: S
// keeps the keys below the new bound) and every warp resumes its share of the
// tile from the step where it stopped, now dropping hubs at or above the new
// bound (a later pass takes them): no message of the tile is read twice, except
// those of the step that met the overflow.
__device__ __noinline__ void gather_block(const GpParams& p, int64_t nb, int64_t ne, uint32_t lo, uint32_t* hi_sm, uint32_t* B,
                             uint32_t vb, uint32_t W, uint32_t* S, int log_s, const uint32_t* M, int log_m, int limit,
                             int* cnt_sm, volatile int* ovf_sm, int* wsum, int* sex, int64_t* sst, uint32_t* C,
                             int* hist, int* tmp, unsigned long long& msgs) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int nw = nthr >> 5, lane = tid & 31;
    const uint32_t set_lo = max(lo, vb + W);  // S holds hubs from here on
    if (lo > vb) W = 0;                       // the map is the first pass's
#pragma unroll 1
    for (int64_t t0 = nb; t0 < ne; t0 += nthr) {
        const uint32_t hi = *(volatile uint32_t*)hi_sm;
        const int64_t j = t0 + tid;
        int c = 0;  // sectors
        int64_t st = 0;
        if (j < ne) {
            const int32_t a = p.rcol[j];
            const uint64_t f = p.fse[a];
            const int n0 = (int)fcount(f);
            if (n0) {
                // the hubs of a frontier row of sender a are <= a (a itself
                // only in round 0): for a < hi the whole row lies below hi
                const uint32_t* row = p.fhub + fstart(f);
                const int a0 = lo > vb ? (int)lower_bound_u32(row, n0, lo) / kRowAlign : 0;
                int a1 = (n0 + kRowAlign - 1) / kRowAlign;
                if (sender_of(p, a) >= hi) {  // sectors whose first hub is below hi
                    int l = a0;
#pragma unroll 1
                    while (l < a1) {
                        const int mid = (l + a1) >> 1;
                        if (row[kRowAlign * mid] < hi) l = mid + 1; else a1 = mid;
                    }
                }
                st = (int64_t)fstart(f) + (int64_t)kRowAlign * a0;
                c = a1 - a0;
            }
        }
        // sector offsets of the tile's non-empty rows, compacted (rows cut
        // to nothing by the hub range are common and would otherwise be
        // stepped over item by item)
        int total, nne;
        const int excl = block_excl_scan(c, wsum, &total);
        __syncthreads();
        const int fidx = block_excl_scan(c > 0 ? 1 : 0, wsum, &nne);
        if (c > 0) {
            sex[fidx] = excl;
            sst[fidx] = st;
        }
        if (tid == 0) sex[nne] = total;
        __syncthreads();
        // each warp takes a contiguous range of the tile's sectors and walks
        // it in windows of 32 rows: lane j holds the start of row k0 + j, and
        // 32 consecutive sectors at a time find their row by a warp-shuffle
        // search
        const int per_w = (((total + nw - 1) / nw) + 31) & ~31;
        const int wbeg = (tid >> 5) * per_w, wend = min(total, wbeg + per_w);
        int pos = wbeg;  // this warp's sectors before pos are done
        unsigned n_msgs = 0;
#pragma unroll 1
        while (true) {
            // hubs at or above hcut are left to a later pass (hcut = hi
            // until the set's range shrinks within this tile)
            const uint32_t hcut = *(volatile uint32_t*)hi_sm;
            if (pos < wend) {
                int k0 = 0, hk = nne - 1;  // row of pos: largest k with sex[k] <= pos
#pragma unroll 1
                while (k0 < hk) {
                    const int mid = (k0 + hk + 1) >> 1;
                    if (sex[mid] <= pos) k0 = mid; else hk = mid - 1;
                }
                bool stop = false;
#pragma unroll 1
                for (int it0 = pos; it0 < wend && !stop; k0 += 32) {
                    const int kr = k0 + lane;
                    const int ex = kr < nne ? sex[kr] : total;
                    // sector i of the tile, in this lane's row, is at row + 8 i
                    const uint32_t* row = p.fhub + ((kr < nne ? sst[kr] : 0) - (int64_t)kRowAlign * ex);
                    const int wend_w = min(wend, k0 + 32 < nne ? sex[k0 + 32] : total);
#pragma unroll 1
                    for (int ib = it0; ib < wend_w; ib += 32) {
                        const int it = ib + lane;
                        const int kk = warp_owner(ex, it);
                        const uint32_t* rk =
                            reinterpret_cast<const uint32_t*>(__shfl_sync(kFull, (unsigned long long)row, kk));
                        uint32_t x[kRowAlign];
                        if (it < wend_w) {
                            load_sector(rk + (int64_t)kRowAlign * it, x);
                        } else {
#pragma unroll
                            for (int q = 0; q < kRowAlign; ++q) x[q] = kEmpty;
                        }
                        unsigned past = 0, got = 0;  // hubs past the map, messages of the range
#pragma unroll
                        for (int q = 0; q < kRowAlign; ++q) {
                            const uint32_t hr = x[q] - vb;
                            if (hr < W) {
                                atomicOr(&B[hr >> 5], 1u << (hr & 31));
                            } else if (x[q] - set_lo < hcut - set_lo) {
                                past |= 1u << q;
                            }
                            got += x[q] - lo < hi - lo ? 1u : 0u;
                        }
                        if (__any_sync(kFull, past != 0u)) {
                            int nins = 0;
#pragma unroll
                            for (int q = 0; q < kRowAlign; ++q)
                                if ((past >> q) & 1u)
                                    nins += set_add(S, log_s, M, log_m, limit, cnt_sm, ovf_sm, x[q]);
                            nins = warp_sum(nins);
                            if (lane == 0 && nins) atomicAdd(cnt_sm, nins);
                            if (__any_sync(kFull, *ovf_sm != 0)) {
                                stop = true;  // resume from this step after the shrink
                                pos = ib;
                                break;
                            }
                        }
                        n_msgs += got;
                    }
                    if (!stop) it0 = wend_w;
                }
                if (!stop) pos = wend;
            }
            __syncthreads();
            // concurrent inserts can pass the limit without raising the flag
            if (*ovf_sm || *(volatile int*)cnt_sm > limit) {
                shrink_pass(S, log_s, C, limit, set_lo, hi_sm, cnt_sm, hist, tmp);
                if (tid == 0) *ovf_sm = 0;
                __syncthreads();
                continue;  // every warp resumes at its pos with the smaller range
            }
            break;
        }
        msgs += n_msgs;
        __syncthreads();  // sex / sst are rewritten by the next tile
    }
}

// One warp per vertex (tables in shared memory):
//  1. gather the messages: hubs among the first 32 x M_CAP of v's graph are
//     marked in a bitmap, the others (few: ranks follow degree) go into the set
//     S; drop L(v)'s hubs;
//  2. list the candidates in S, the bitmap's in rank order;
//  3. first prefilter step; when it leaves any, stage L(v) into the hub-keyed
//     map M, in the bitmap's place (or, with few candidates against a long row,
//     look L(v) up in v's row of the global probe index), and check them;
//  4. append the accepted hubs to the new frontier: in order, the set's sorted.
// A vertex with more than cand_limit candidates in the set, or more in all than
// the list holds, goes to the block tier.
// What bounds it is instruction issue (each of 24 independent warps per SM
// issues every 12 cycles) and the instructions' way to the SM: the bitmap
// replaced a hash set with a look-up in M per message, its compaction and a
// bitonic sort of the accepted hubs.
__global__ void __launch_bounds__(256, 3) k_gp_warp(GpParams p) {
    extern __shared__ uint32_t sm[];
    const int lane = lane_id(), wib = threadIdx.x >> 5;
    const int nwarps = blockDim.x >> 5;
    const int M_CAP = 1 << p.log_m;
    int* wsc = reinterpret_cast<int*>(sm) + wib * 4;  // [0] entries of the set
    // per warp: the set, then the candidates and, in its last words, v's
    // exact-distance top-hub masks
    uint32_t* S = sm + 4 * nwarps + wib * (p.s_words + M_CAP);
    uint32_t* X = S + p.s_words;                       // hub bitmap (zero between vertices), then L(v)'s map
    const int cap = p.s_words - kTopRow;               // most candidates
    uint32_t* tv = S + cap;
    const unsigned lt = (1u << lane) - 1u;
    unsigned long long c_arcs = 0, c_msgs = 0, c_uniq = 0, c_staged = 0, c_probed = 0, c_acc = 0, c_vert = 0;
    unsigned long long c_pref = 0, c_chk[2] = {0, 0};
    if (p.ctr->done) return;
    const uint32_t d = p.ctr->d;
    const int imax = min((int)d - 1, kTopLevels);
    const int nlist = *p.list_n;
    if (nlist <= 0) return;
#pragma unroll 1
    for (int s = lane; s < M_CAP; s += 32) X[s] = 0u;
    // vertices are handed out one at a time (they differ in cost by orders of
    // magnitude), the next one while this one is worked on
    int next = 0;
    if (lane == 0) next = atomicAdd(p.work, 1);
#pragma unroll 1
    while (true) {
        __syncwarp();
        const int i = __shfl_sync(kFull, next, 0);
        if (i >= nlist) break;
        if (lane == 0) next = atomicAdd(p.work, 1);
        const int32_t v = p.list[i];
        const uint32_t vb = base_of(p.vbase, v);
        const int64_t lb = p.loff[v], ll = p.loff[v + 1] - lb;
        const int64_t nb = p.roff[v], ne = p.roff[v + 1];
        const uint32_t* lv = p.lent + lb;
        const uint32_t bnd = p.rbound[v];
        // the set sized for v's candidate bound (when within the tier's limit)
        const int log_s = bnd <= (uint32_t)p.cand_limit ? max(5, ceil_log2_i64(2 * (int64_t)bnd)) : p.log_s;
        const uint32_t W = min(32u * (uint32_t)M_CAP, (uint32_t)v - vb);
        if (lane == 0) wsc[0] = 0;
        __syncwarp();
        uint32_t top = 0;
        const bool ok = gather_range(p, nb, ne, (uint32_t)v, vb, W, X, S, log_s, p.cand_limit, &wsc[0], &top, c_msgs);
        __syncwarp();
        // candidates: the bitmap's without L(v)'s hubs ...
        const int words = (int)((top + 31u) >> 5);
        int nbm = 0, nset = 0;
        if (ok) {
            // (four loads in flight, here and where the map is staged: one at a
            // time, each waited for, weighted Chung-Lu 2^20 took 56.0 ms instead
            // of 54.1, the batch of 200 graphs 49.1 instead of 47.7)
#pragma unroll 1
            for (int j = lane; j < (int)ll; j += 128) {
                uint32_t w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) w[q] = j + 32 * q < (int)ll ? hub_of(lv[j + 32 * q]) - vb : kEmpty;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (w[q] < top) atomicAnd(&X[w[q] >> 5], ~(1u << (w[q] & 31)));
            }
            __syncwarp();
            // ... and the set's, compacted in place (write position never
            // passes the read position)
            const bool any = *(volatile int*)&wsc[0] > 0;
            if (any || bnd > (uint32_t)cap) {
#pragma unroll 1
                for (int q = lane; q < words; q += 32) nbm += __popc(X[q]);
                nbm = warp_sum(nbm);
            }
            if (any) {
#pragma unroll 1
                for (int sb = 0; sb < (1 << log_s); sb += 32) {
                    const uint32_t h = S[sb + lane];
                    __syncwarp();
                    bool has = h != kEmpty;
                    if (has) {
                        const int64_t at = lower_bound_u32(lv, ll, pack(h, 0));
                        has = at >= ll || hub_of(lv[at]) != h;
                    }
                    const unsigned m = __ballot_sync(kFull, has);
                    if (has) S[nset + __popc(m & lt)] = h;
                    nset += __popc(m);
                }
                __syncwarp();
            }
        }
        if (!ok || nbm + nset > cap) {
#pragma unroll 1
            for (int q = lane; q < (int)((W + 31u) >> 5); q += 32) X[q] = 0u;
            if (lane == 0) {
                const int o = atomicAdd(p.esc_n, 1);
                p.esc[o] = v;
            }
            continue;
        }
        // list them: the set's moved up behind the bitmap's
        if (nset > 0 && nbm > 0) {
#pragma unroll 1
            for (int c = (nset - 1) & ~31; c >= 0; c -= 32) {
                const uint32_t h = c + lane < nset ? S[c + lane] : 0u;
                __syncwarp();
                if (c + lane < nset) S[nbm + c + lane] = h;
                __syncwarp();
            }
        }
        int nc = 0;
#pragma unroll 1
        for (int q0 = 0; q0 < words; q0 += 128) {  // four words (128 hubs) per lane
            uint4* x4 = reinterpret_cast<uint4*>(X + q0) + lane;
            uint4 y = make_uint4(0u, 0u, 0u, 0u);
            if (q0 + 4 * lane < words) y = *x4;
            if (!__any_sync(kFull, (y.x | y.y | y.z | y.w) != 0u)) continue;
            const int c = __popc(y.x) + __popc(y.y) + __popc(y.z) + __popc(y.w);
            const int incl = warp_incl_scan(c, lane);
            uint32_t* o = S + nc + incl - c;
            uint32_t hb = vb + 32u * (uint32_t)(q0 + 4 * lane) - 1u;
            if (c) *x4 = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll 1
            for (; y.x; y.x &= y.x - 1u) *o++ = hb + (uint32_t)__ffs(y.x);
            hb += 32u;
#pragma unroll 1
            for (; y.y; y.y &= y.y - 1u) *o++ = hb + (uint32_t)__ffs(y.y);
            hb += 32u;
#pragma unroll 1
            for (; y.z; y.z &= y.z - 1u) *o++ = hb + (uint32_t)__ffs(y.z);
            hb += 32u;
#pragma unroll 1
            for (; y.w; y.w &= y.w - 1u) *o++ = hb + (uint32_t)__ffs(y.w);
            nc += __shfl_sync(kFull, incl, 31);
        }
        nc += nset;
        __syncwarp();
        if (lane == 0) {
            c_arcs += ne - nb;
            c_vert += 1;
            c_uniq += nc;
        }
        if (nc == 0) continue;
        stage_exact_levels(p.top, p.n, v, tv, lane, 32);
        __syncwarp();
        // first prefilter step, 64 candidates at a time, then the distance
        // checks of its survivors, 32 at a time; both compact S in place and in
        // order.  A single chunk goes to the checks at once (i0 = 0: the masks
        // and the check records of its candidates are then requested together)
        int i0 = 0, ns = nc;
        if (p.count_check)
#pragma unroll 1
            for (int j = lane; j < nc; j += 32) count_reads(p.loff_h, lv, ll, S[j], c_chk);
        if (nc > 32) {
            i0 = first_level(tv, imax, lane);
            ns = 0;
#pragma unroll 1
            for (int cb = 0; cb < nc; cb += 64) {
                const bool v0 = cb + lane < nc, v1 = cb + 32 + lane < nc;
                const uint32_t h0 = v0 ? S[cb + lane] : 0u, h1 = v1 ? S[cb + 32 + lane] : 0u;
                unsigned m0, m1;
                prefilter_first(p, tv, (int)d, imax, i0, h0, v0, h1, v1, &m0, &m1);
                if ((m0 >> lane) & 1u) S[ns + __popc(m0 & lt)] = h0;
                ns += __popc(m0);
                if ((m1 >> lane) & 1u) S[ns + __popc(m1 & lt)] = h1;
                ns += __popc(m1);
                __syncwarp();
            }
            if (lane == 0) c_pref += nc - ns;
            if (ns == 0) continue;
        }
        // L(v) look-ups: the map staged in shared memory, or, for a receiver
        // with few candidates against a long (indexed) row, v's row of the
        // global probe index, which saves staging the whole row
        const uint64_t hdv = (p.stage_ratio > 0 && ll >= kIndexMinLen &&
                              (int64_t)bnd * p.stage_ratio < ll) ? p.hdesc[v] : 0ull;
        const bool mglob = hdv != 0;
        const int log_m = mglob ? (int)(hdv & 0xFFu) : max(5, ceil_log2_i64(2 * ll));
        const uint32_t* Mv = mglob ? p.htab + (hdv >> 8) : X;
        // L(v)'s sorted row, copied behind the candidates (the set's slots
        // past ns are free now) when it fits: the checks' binary searches in
        // L(v) and their side-B scans of it then read shared memory
        const uint32_t* lvp = lv;
        const bool copy = (int64_t)ns + ll <= cap;
        uint32_t* lvs = S + (cap - ll);
        if (copy) lvp = lvs;
        if (!mglob) {
#pragma unroll 1
            for (int s = lane; s < (1 << log_m); s += 32) X[s] = kEmpty;
            __syncwarp();
        }
        if (!mglob || copy) {
#pragma unroll 1
            for (int j = lane; j < (int)ll; j += 128) {
                uint32_t e[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) e[q] = j + 32 * q < (int)ll ? lv[j + 32 * q] : kEmpty;
#pragma unroll 1
                for (int q = 0; q < 4; ++q, e[0] = e[1], e[1] = e[2], e[2] = e[3]) {
                    if (j + 32 * q >= (int)ll) break;
                    if (!mglob) map_insert(X, log_m, e[0]);
                    if (copy) lvs[j + 32 * q] = e[0];
                }
            }
        }
        if (lane == 0) c_staged += mglob ? 0 : ll;
        __syncwarp();
        // entries of L(v) with a top hub (the checks' side B starts past them)
        const int lv_top = (int)lower_bound_u32(lvp, ll, pack(vb + (uint32_t)kTopHubs, 0));
        int nacc = 0, ntail = 0;  // accepted; of them past the bitmap's hubs
#pragma unroll 1
        for (int cb = 0; cb < ns; cb += 32) {
            const bool valid = cb + lane < ns;
            const uint32_t h = valid ? S[cb + lane] : 0u;
            __syncwarp();
            const unsigned okm = check_chunk(p, d, Mv, log_m, mglob, kWarpSideBMin, kWarpSideBShift, lvp, ll, lv_top,
                                             h, valid, c_probed, tv, i0, c_pref);
            const bool acc = (okm >> lane) & 1u;
            if (acc) S[nacc + __popc(okm & lt)] = h;
            nacc += __popc(okm);
            if (nset > 0) ntail += __popc(__ballot_sync(kFull, acc && h - vb >= W));
            __syncwarp();
        }
        if (!mglob)
#pragma unroll 1
            for (int s = lane; s < (1 << log_m); s += 32) X[s] = 0u;
        if (nacc > 0) {
            unsigned long long start = 0;
            const int padded = (int)row_pad(nacc);
            if (lane == 0)
                start = p.ostart ? (unsigned long long)p.ostart[v]
                                 : atomicAdd(&p.ctr->cursor, (unsigned long long)padded);
            start = __shfl_sync(kFull, start, 0);
            if (start + padded <= p.fcap) {
                uint32_t* row = p.fhub_new + start;
                if (nacc + lane < padded) row[nacc + lane] = kEmpty;
                // the new row leaves sorted by hub rank: the bitmap's hubs as
                // they are, then the set's, moved to the front of S and sorted
                const int n0 = nacc - ntail;
#pragma unroll 1
                for (int j = lane; j < n0; j += 32) row[j] = S[j];
                if (ntail > 0) {
                    int P = 32;
#pragma unroll 1
                    while (P < ntail) P <<= 1;  // <= cap: at most cand_limit
#pragma unroll 1
                    for (int j0 = 0; j0 < P; j0 += 32) {
                        const uint32_t h = j0 + lane < ntail ? S[n0 + j0 + lane] : kEmpty;
                        __syncwarp();
                        S[j0 + lane] = h;
                        __syncwarp();
                    }
                    group_bitonic_sort(S, P, lane, 32, WarpSync());
#pragma unroll 1
                    for (int j = lane; j < ntail; j += 32) row[n0 + j] = S[j];
                }
                if (lane == 0) p.fse_new[v] = fpack(start, (uint32_t)nacc);
            } else if (lane == 0) {
                p.ctr->fovf = 1;
            }
            if (lane == 0) c_acc += nacc;
        }
    }
    c_probed = warp_sum(c_probed);
    c_msgs = warp_sum(c_msgs);
    if (p.count_check) {
        c_chk[0] = warp_sum(c_chk[0]);
        c_chk[1] = warp_sum(c_chk[1]);
        if (lane == 0) {
            atomicAdd(&p.ctr->chk_lv, c_chk[0]);
            atomicAdd(&p.ctr->chk_lh, c_chk[1]);
        }
    }
    if (lane == 0) {
        atomicAdd(&p.ctr->arcs, c_arcs);
        atomicAdd(&p.ctr->msgs, c_msgs);
        atomicAdd(&p.ctr->uniq, c_uniq);
        atomicAdd(&p.ctr->staged, c_staged);
        atomicAdd(&p.ctr->probed, c_probed);
        atomicAdd(&p.ctr->accepted, c_acc);
        atomicAdd(&p.ctr->tier[0], c_vert);
        atomicAdd(&p.ctr->prefiltered, c_pref);
    }
}

// Block-per-vertex scalars in shared memory (ints)
enum { SH_UNIQ = 0, SH_OVF = 1, SH_ACC = 2 /* accepted, from the set */, SH_NC = 3, SH_HI = 4, SH_TMP = 5 /* 2 ints */,
       SH_START = 8 /* 2 ints */, SH_NEXT = 10, SH_REST = 11, SH_MACC = 12 /* accepted, from the map */,
       SH_ITEM = 13, SH_LAST = 14, SH_NE = 15 /* rows of the first prefilter step */,
       SH_WCNT = 16 /* 8 warps */, SH_WORDS = 48 };

// Accepted candidates of a chunk (okm): those of the map are marked there
// again (extraction cleared them), the set's go to this block's global scratch.
__device__ __forceinline__ void keep_accepted(unsigned okm, uint32_t h, uint32_t vb, uint32_t W, uint32_t* B,
                                              uint32_t* gacc, int* sh) {
    const int lane = threadIdx.x & 31;
    const uint32_t hr = h - vb;
    const bool ok = (okm >> lane) & 1u, inmap = hr < W;
    if (ok && inmap) {
        atomicOr(&B[hr >> 5], 1u << (hr & 31));
    }
    const unsigned mm = __ballot_sync(kFull, ok && inmap), ms = okm & ~mm;
    int base = 0;
    if (lane == 0) {
        if (mm) atomicAdd(&sh[SH_MACC], __popc(mm));
        if (ms) base = atomicAdd(&sh[SH_ACC], __popc(ms));
    }
    base = __shfl_sync(kFull, base, 0);
    if (ok && !inmap) gacc[base + __popc(ms & ((1u << lane) - 1u))] = h;
}

// Emits the marked hubs of the map (W hubs from vb) to row in rank order and
// clears them (row null: only clears).  Warp w takes the w-th slice.
__device__ void emit_map(uint32_t* B, uint32_t vb, uint32_t W, uint32_t* row, int* sh) {
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = blockDim.x >> 5;
    uint4* w4 = reinterpret_cast<uint4*>(B);
    // units of 32 lanes x 16 bytes (128 hubs per lane)
    const int uw = (int)((W + 4095) / 4096);
    const int w0 = uw * wid / nw, w1 = uw * (wid + 1) / nw;
    int cw = 0;
#pragma unroll 1
    for (int u = w0; u < w1; ++u) {
        const uint4 x = w4[32 * u + lane];
        cw += __popc(x.x) + __popc(x.y) + __popc(x.z) + __popc(x.w);
    }
    cw = warp_sum(cw);
    if (lane == 0) sh[SH_WCNT + wid] = cw;
    __syncthreads();
    if (cw == 0) return;
    const int c = lane < nw ? sh[SH_WCNT + lane] : 0;
    int pos = __shfl_sync(kFull, warp_incl_scan(c, lane) - c, wid);
#pragma unroll 1
    for (int u = w0; u < w1; ++u) {
        const int x = 32 * u + lane;
        const uint4 y = w4[x];
        if (!__any_sync(kFull, (y.x | y.y | y.z | y.w) != 0u)) continue;
        const int k = __popc(y.x) + __popc(y.y) + __popc(y.z) + __popc(y.w);
        const int incl = warp_incl_scan(k, lane);
        int o = pos + incl - k;
        if (k) w4[x] = make_uint4(0u, 0u, 0u, 0u);
        if (row && k) {
            const uint32_t q[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const uint32_t hb = vb - 1u + 128u * (uint32_t)x + 32u * (uint32_t)j;
#pragma unroll 1
                for (uint32_t w = q[j]; w; w &= w - 1u) row[o++] = hb + (uint32_t)__ffs(w);
            }
        }
        pos += __shfl_sync(kFull, incl, 31);
    }
}

// The marked hubs of the map (W of them) OR-ed into a split receiver's global
// bitmap; the map is left empty.
__device__ void flush_map(uint32_t* B, uint32_t W, uint32_t* gbits) {
#pragma unroll 1
    for (int q = threadIdx.x; q < (int)((W + 31u) >> 5); q += blockDim.x) {
        const uint32_t w = B[q];
        if (w) B[q] = 0u;
        // (most of it is there already once a few parts have been merged)
        if (w & ~__ldcg(gbits + q)) atomicOr(gbits + q, w);
    }
}

// The map of a split receiver from its global bitmap, which is left empty.
__device__ void load_map(uint32_t* B, uint32_t W, uint32_t* gbits) {
#pragma unroll 1
    for (int q = threadIdx.x; q < (int)((W + 31u) >> 5); q += blockDim.x) {
        const uint32_t w = __ldcg(gbits + q);
        if (w == 0u) continue;
        gbits[q] = 0u;
        B[q] = w;
    }
}

// One block per vertex, any size.  The candidates are processed in passes
// over hub ranges [lo, hi): each pass gathers the messages of its range into
// the hub map (the first pass) and the shared-memory set (shrinking hi when
// the set would overflow) and checks them.
//
// What bounds it is latency: three blocks of 8 warps per SM wait on random
// 32-byte sectors (masks, check records, probe tables) of arrays far larger
// than L2, and one chunk of 32 candidates checked from end to end took 5,000
// to 12,000 cycles although most of its candidates need one mask only.  So the
// check is split: each warp takes units of the map and of the set from a
// shared counter, prunes them by the top-hub columns (64 candidates per lane:
// testing one 32-byte mask per candidate, and listing candidates for it, took
// 108 and 143 ms of warp time in rounds 2 and 3 of R-MAT 2^22), and runs
// check_chunk on full warps of survivors; the warps' last survivors are pooled
// and spread over all warps.
// L(v) is staged into the shared-memory map when it fits; otherwise it is
// looked up in v's row of the global probe index.  Accepted hubs are marked in
// the map and leave it in rank order, so the new row needs no later sort.
__device__ void gp_block_vertex(const GpParams& p, uint32_t d, int32_t v, uint32_t* S, uint32_t* M, uint32_t* C,
                                uint32_t* B, uint32_t* gacc, int* sh, int* wsum, int* sex, int64_t* sst, int* hist,
                                uint32_t* tv, unsigned long long* cnt, uint32_t* gbits) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int lane = tid & 31, wid = tid >> 5, nw = nthr >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int64_t lb = p.loff[v], ll = p.loff[v + 1] - lb;
    const int64_t nb = p.roff[v], ne = p.roff[v + 1];
    const uint32_t* lv = p.lent + lb;
    const int log_s = p.log_s, S_CAP = 1 << log_s, limit = p.cand_limit;
    int log_m = ceil_log2_i64(2 * ll + 2 * nthr);
    if (log_m < 5) log_m = 5;
    const bool useM = log_m <= p.log_m;
    // L(v) lookups: the shared-memory map, or v's row of the global probe
    // index (a row too long for the map has more than 64 >= kIndexMinLen
    // entries, so it is indexed)
    static_assert(kIndexMinLen <= 64, "rows beyond the block map must be indexed");
    const uint32_t* Mp = M;
    int log_mp = log_m;
    if (!useM) {
        const uint64_t hd = p.hdesc[v];
        Mp = p.htab + (hd >> 8);
        log_mp = (int)(hd & 0xFFu);
    }
    if (useM) {
#pragma unroll 1
        for (int s = tid; s < (1 << log_m); s += nthr) M[s] = kEmpty;
        __syncthreads();
#pragma unroll 1
        for (int64_t j = tid; j < ll; j += nthr) map_insert(M, log_m, lv[j]);
    }
    if (tid == 0) {
        cnt[0] += ne - nb;
        cnt[3] += ll;
        cnt[6] += 1;
        sh[SH_ACC] = 0;
        sh[SH_MACC] = 0;
    }
    stage_exact_levels(p.top, p.n, v, tv, tid, nthr);
    const uint32_t vb = base_of(p.vbase, v);  // v's hubs are ranks [vb, v)
    uint32_t lo = vb;
    int64_t width = (int64_t)v - vb;
    uint32_t* hi_sm = reinterpret_cast<uint32_t*>(&sh[SH_HI]);
    // hubs below vb + W (the most frequent messages) are deduplicated in the
    // map, in the first pass
    const uint32_t W = min((uint32_t)kMapHubs, (uint32_t)v - vb);
    uint32_t* surv = S + wid * kWarpStage;  // (S is free once compacted)
    uint32_t cwords;
    const uint32_t* cols = columns_of(p.cols_h, vb, &cwords);
    const int imax = min((int)d - 1, kTopLevels);
#pragma unroll 1
    while (lo < (uint32_t)v) {
        if (lo > vb || (uint32_t)v - vb > W) {  // (no message reaches the set when the map holds every hub of v)
            uint4* s4 = reinterpret_cast<uint4*>(S);
#pragma unroll 1
            for (int s = tid; s < S_CAP / 4; s += nthr) s4[s] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
        }
        if (tid == 0) {
            sh[SH_UNIQ] = 0;
            sh[SH_OVF] = 0;
            sh[SH_NC] = 0;
            sh[SH_NEXT] = 0;
            sh[SH_REST] = 0;
            *hi_sm = (uint32_t)min((int64_t)v, (int64_t)lo + width);
        }
        __syncthreads();
        if (gbits)
            load_map(B, W, gbits);
        else
            gather_block(p, nb, ne, lo, hi_sm, B, vb, W, S, log_s, useM ? M : nullptr, log_m, limit, &sh[SH_UNIQ],
                         (volatile int*)&sh[SH_OVF], wsum, sex, sst, C, hist, &sh[SH_TMP], cnt[1]);
        __syncthreads();
        const uint32_t hi = *(volatile uint32_t*)hi_sm;
        const bool maps = lo == vb;
        if (maps) {  // first pass: drop L(v)'s hubs from the map
#pragma unroll 1
            for (int64_t j = tid; j < ll; j += nthr) {
                const uint32_t w = hub_of(lv[j]) - vb;
                if (w < W) atomicAnd(&B[w >> 5], ~(1u << (w & 31)));
            }
        }
        // compact the set into C (any order)
        if (*(volatile int*)&sh[SH_UNIQ] > 0) {
#pragma unroll 1
            for (int sb = 32 * wid; sb < S_CAP; sb += 32 * nw) {
                const uint32_t h = S[sb + lane];
                const bool has = h != kEmpty;
                const unsigned m = __ballot_sync(kFull, has);
                int base = 0;
                if (lane == 0 && m) base = atomicAdd(&sh[SH_NC], __popc(m));
                base = __shfl_sync(kFull, base, 0);
                const int idx = base + __popc(m & lt);
                if (has) {
                    if (idx < limit) C[idx] = h;
                    else p.ctr->guard = 1;  // invariant broken: report instead of writing out of bounds
                }
            }
        }
        __syncthreads();  // every warp has read the set
        // L(v)'s sorted row in the set's free tail (its head stages the warps'
        // candidates): the checks' binary searches in L(v) and their side-B
        // scans of it then read shared memory
        const uint32_t* lvp = lv;
        if (ll + (int64_t)nw * kWarpStage <= (int64_t)S_CAP) {
            uint32_t* lvs = S + (S_CAP - ll);
#pragma unroll 1
            for (int64_t j = tid; j < ll; j += nthr) lvs[j] = lv[j];
            lvp = lvs;
        }
        // the rows of the first prefilter step (column offsets, in hist; filled
        // up to a multiple of four): v's top hubs at distance i0, or at every
        // distance in weighted rounds; none for a graph without columns, whose
        // candidates take the whole prefilter in check_chunk
        const int i0 = first_level(tv, imax, lane);
        if (wid == nw - 1) {
            int ne = 0;
#pragma unroll 1
            for (int i = p.sender_bits ? 1 : i0; cwords && i <= (p.sender_bits ? imax : i0); ++i) {
                uint32_t m = lane < kTopWords ? tv[(i - 1) * kTopWords + lane] : 0u;
                const int c = __popc(m);
                const int incl = warp_incl_scan(c, lane);
                int o = ne + incl - c;
                const int row0 = (min((int)d - i, kTopLevels) - 1) * kTopHubs + 32 * lane - 1;
#pragma unroll 1
                for (; m; m &= m - 1u) hist[o++] = (row0 + __ffs(m)) * (int)cwords;
                ne += __shfl_sync(kFull, incl, 31);
            }
            __syncwarp();
            if (ne > 0 && lane < ((4 - ne) & 3)) hist[ne + lane] = hist[0];
            if (lane == 0) sh[SH_NE] = ne;
        }
        __syncthreads();
        const int n_rows = *(volatile int*)&sh[SH_NE];
        // entries of L(v) with a top hub (the checks' side B starts past them)
        const int lv_top = (int)lower_bound_u32(lvp, ll, pack(vb + (uint32_t)kTopHubs, 0));
        const int nc_set = min(*(volatile int*)&sh[SH_NC], limit);  // candidates from the set
        // units: 2,048 hubs of the map (64 per lane, cleared as they are read),
        // pruned by the receiver's rows of the top-hub columns, or 32 of the
        // set's candidates, pruned by their own masks.  The warps take them from
        // a shared counter and check full warps of survivors
        const int um = maps ? (int)((W + 2047) / 2048) : 0;
        const int units = um + (nc_set + 31) / 32;
        bool more = true, last = false;
        int ns = 0;                           // survivors
        uint32_t c0 = 0, c1 = 0, hb = 0;      // this lane's of the current unit: hub hb + b for every bit b of c1 c0
#pragma unroll 1
        while (!last) {
#pragma unroll 1
            while (ns < 32 && more) {
                const bool has = (c0 | c1) != 0u;
                const unsigned m = __ballot_sync(kFull, has);
                if (m) {
                    if (has) {
                        const uint32_t b = c0 ? (uint32_t)__ffs(c0) - 1u : (uint32_t)__ffs(c1) + 31u;
                        if (c0) c0 &= c0 - 1u;
                        else c1 &= c1 - 1u;
                        surv[ns + __popc(m & lt)] = hb + b;
                    }
                    ns += __popc(m);
                    continue;
                }
                int u = 0;
                if (lane == 0) u = atomicAdd(&sh[SH_NEXT], 1);
                u = __shfl_sync(kFull, u, 0);
                if (u >= units) {
                    more = false;
                } else if (u < um) {
                    const int x = 64 * u + 2 * lane;  // first of the lane's two words, as bits
                    uint2* q = reinterpret_cast<uint2*>(B + x);
                    const uint2 y = *q;
                    c0 = y.x;
                    c1 = y.y;
                    if (c0 | c1) *q = make_uint2(0u, 0u);
                    hb = vb + 32u * (uint32_t)x;
                    if (!__any_sync(kFull, (c0 | c1) != 0u)) continue;
                    const int found = __popc(c0) + __popc(c1);
                    if (p.count_check)
                        count_reads64(p.loff_h, lvp, ll, hb, (unsigned long long)c1 << 32 | c0, cnt + 8);
                    // (x < the row's words: hubs of v's graph within the map,
                    // rounded up to 128; rows are 16-byte aligned; a graph
                    // without columns has no rows to read)
                    const uint32_t* cx = cols + min((uint32_t)x, cwords - 2u);
#pragma unroll 1
                    for (int k = 0; k < n_rows; k += 4) {
                        const int4 o = *reinterpret_cast<const int4*>(hist + k);
                        const uint2 t0 = *reinterpret_cast<const uint2*>(cx + o.x);
                        const uint2 t1 = *reinterpret_cast<const uint2*>(cx + o.y);
                        const uint2 t2 = *reinterpret_cast<const uint2*>(cx + o.z);
                        const uint2 t3 = *reinterpret_cast<const uint2*>(cx + o.w);
                        c0 &= ~(t0.x | t1.x | t2.x | t3.x);
                        c1 &= ~(t0.y | t1.y | t2.y | t3.y);
                        if (!__any_sync(kFull, (c0 | c1) != 0u)) break;
                    }
                    cnt[2] += found;
                    cnt[7] += found - __popc(c0) - __popc(c1);
                } else {
                    const int x = 32 * (u - um) + lane;
                    bool valid = x < nc_set;
                    hb = valid ? C[x] : 0u;
                    // without the map, set candidates may be hubs of v already
                    if (!useM && valid && map_has(Mp, log_mp, hb)) valid = false;
                    if (p.count_check && valid) count_reads(p.loff_h, lvp, ll, hb, cnt + 8);
                    unsigned m0, m1;
                    prefilter_first(p, tv, (int)d, imax, i0, hb, valid, 0u, false, &m0, &m1);
                    c0 = (m0 >> lane) & 1u;
                    c1 = 0;
                    cnt[2] += valid ? 1 : 0;
                    cnt[7] += valid && !c0 ? 1 : 0;
                }
            }
            __syncwarp();
            if (ns < 32) {
                // no unit is left: the warps' last survivors (fewer than 32
                // each) are pooled behind C's candidates and spread over the
                // warps, so that one warp's scans are not what the others wait for
                int base = 0;
                if (lane == 0 && ns) base = atomicAdd(&sh[SH_REST], ns);
                base = __shfl_sync(kFull, base, 0);
                if (lane < ns) C[limit + base + lane] = surv[lane];
                __syncthreads();
                const int nrest = *(volatile int*)&sh[SH_REST];
                const int per = max(4, (nrest + nw - 1) / nw);  // at most 31
                ns = max(0, min(per, nrest - wid * per));
                if (lane < ns) surv[lane] = C[limit + wid * per + lane];
                __syncwarp();
                last = true;
            }
#pragma unroll 1
            while (ns >= 32 || (last && ns > 0)) {
                const int k = min(ns, 32);
                ns -= k;
                const bool valid = lane < k;
                const uint32_t h = valid ? surv[ns + lane] : 0u;
                const unsigned okm = check_chunk(p, d, Mp, log_mp, !useM, kBlockSideBMin, kBlockSideBShift, lvp, ll,
                                                 lv_top, h, valid, cnt[4], tv, cwords ? i0 : 0, cnt[7]);
                keep_accepted(okm, h, vb, W, B, gacc, sh);
            }
            __syncwarp();
        }
        __syncthreads();
        width = 2 * (int64_t)(hi - lo);
        lo = hi;
    }
    // the new row: the map's hubs in rank order, then the set's (all of them
    // past the map), sorted in shared memory (more than the set's slots hold:
    // listed for the row sort)
    const int macc = *(volatile int*)&sh[SH_MACC], sacc = *(volatile int*)&sh[SH_ACC];
    const int64_t total_acc = (int64_t)macc + sacc;
    if (total_acc > 0) {
        if (tid == 0) {
            const unsigned long long start =
                p.ostart ? (unsigned long long)p.ostart[v]
                         : atomicAdd(&p.ctr->cursor, (unsigned long long)row_pad(total_acc));
            *(unsigned long long*)(sh + SH_START) = start;
        }
        __syncthreads();
        const unsigned long long start = *(volatile unsigned long long*)(sh + SH_START);
        const bool fits = start + row_pad(total_acc) <= p.fcap;
        uint32_t* row = p.fhub_new + start;
        if (fits && total_acc + tid < row_pad(total_acc)) row[total_acc + tid] = kEmpty;
        if (macc > 0) emit_map(B, vb, W, fits ? row : nullptr, sh);
        if (fits) {
            const bool sorted = sacc <= S_CAP;
            if (sacc > 1 && sorted) {
                int P = 2;
#pragma unroll 1
                while (P < sacc) P <<= 1;
#pragma unroll 1
                for (int j = tid; j < P; j += nthr) S[j] = j < sacc ? gacc[j] : kEmpty;
                __syncthreads();
                group_bitonic_sort(S, P, tid, nthr, BlockSync());
#pragma unroll 1
                for (int j = tid; j < sacc; j += nthr) row[macc + j] = S[j];
            } else {
#pragma unroll 1
                for (int j = tid; j < sacc; j += nthr) row[macc + j] = gacc[j];
            }
            if (tid == 0) {
                p.fse_new[v] = fpack(start, (uint32_t)total_acc);
                if (!sorted && p.unsorted) p.unsorted[atomicAdd(&p.ctr->nU, 1)] = v;  // sorted after the round
            }
        } else if (tid == 0) {
            p.ctr->fovf = 1;
        }
        if (tid == 0) cnt[5] += total_acc;
    }
    __syncthreads();
}

__global__ void __launch_bounds__(256, 3) k_gp_block(GpParams p) {
    extern __shared__ uint32_t sm[];
    int* sh = reinterpret_cast<int*>(sm);
    int* wsum = sh + SH_WORDS;                                      // 33 ints (+ 3 pad)
    int* hist = wsum + 36;                                          // 256 ints
    uint32_t* tv = reinterpret_cast<uint32_t*>(hist + 256);         // v's exact-distance top-hub masks
    int* sex = reinterpret_cast<int*>(tv + kTopRow);                // blockDim + 1 ints
    int64_t* sst = reinterpret_cast<int64_t*>(sex + ((blockDim.x + 4) & ~3u));  // blockDim int64
    uint32_t* S = reinterpret_cast<uint32_t*>(sst + blockDim.x);
    uint32_t* M = S + (1 << p.log_s);
    uint32_t* C = M + (1 << p.log_m);
    uint32_t* B = C + p.cand_limit + (int)blockDim.x;  // kMapWords words
    uint32_t* gacc = p.gscratch + (int64_t)blockIdx.x * p.gscratch_words;
    unsigned long long cnt[10] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
    if (p.ctr->done) return;
    const uint32_t d = p.ctr->d;
    const int n1 = *p.list_n, np = p.split.max > 0 ? min(p.ctr->nP, p.split.max_parts) : 0;
    if ((int)blockIdx.x >= np + n1) return;  // (as many blocks as entries are enough)
    // the hub map is empty between vertices
#pragma unroll 1
    for (int q = threadIdx.x; q < kMapWords; q += blockDim.x) B[q] = 0u;
    // parts of split receivers first, then the list's vertices (in rank order:
    // the largest first), handed out one at a time
    int next = 0;
    if (threadIdx.x == 0) sh[SH_ITEM] = atomicAdd(p.work, 1);
    __syncthreads();
#pragma unroll 1
    while (true) {
        const int i = *(volatile int*)&sh[SH_ITEM];
        if (i >= np + n1) break;
        if (threadIdx.x == 0) next = atomicAdd(p.work, 1);
        int32_t v = 0;
        uint32_t* gbits = nullptr;
        bool whole = true;
        if (i < np) {
            const int2 part = p.split.parts[i];
            v = p.split.v[part.x];
            gbits = p.split.bits + (int64_t)part.x * p.split.words;
            const uint32_t vb = base_of(p.vbase, v), W = (uint32_t)v - vb;  // (all of v's hubs fit the map)
            const int64_t nb = p.roff[v] + (int64_t)part.y * kSplitPart;
            const int64_t ne = min(p.roff[v + 1], nb + kSplitPart);
            uint32_t* hi_sm = reinterpret_cast<uint32_t*>(&sh[SH_HI]);
            if (threadIdx.x == 0) {
                sh[SH_UNIQ] = 0;
                sh[SH_OVF] = 0;
                *hi_sm = (uint32_t)v;
            }
            __syncthreads();
            gather_block(p, nb, ne, vb, hi_sm, B, vb, W, S, p.log_s, nullptr, 0, p.cand_limit, &sh[SH_UNIQ],
                         (volatile int*)&sh[SH_OVF], wsum, sex, sst, C, hist, &sh[SH_TMP], cnt[1]);
            __syncthreads();
            flush_map(B, W, gbits);
            __threadfence();
            __syncthreads();
            if (threadIdx.x == 0) {
                const bool last = atomicAdd(&p.split.done[part.x], 1) == p.split.nparts[part.x] - 1;
                if (last) p.split.done[part.x] = 0;
                sh[SH_LAST] = last;
            }
            __syncthreads();
            __threadfence();
            whole = *(volatile int*)&sh[SH_LAST] != 0;
        } else {
            v = p.list[i - np];
        }
        if (whole) gp_block_vertex(p, d, v, S, M, C, B, gacc, sh, wsum, sex, sst, hist, tv, cnt, gbits);
        if (threadIdx.x == 0) sh[SH_ITEM] = next;
        __syncthreads();
    }
    cnt[1] = warp_sum(cnt[1]);
    cnt[2] = warp_sum(cnt[2]);
    cnt[4] = warp_sum(cnt[4]);
    cnt[7] = warp_sum(cnt[7]);
    if (p.count_check) {
        cnt[8] = warp_sum(cnt[8]);
        cnt[9] = warp_sum(cnt[9]);
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&p.ctr->chk_lv, cnt[8]);
            atomicAdd(&p.ctr->chk_lh, cnt[9]);
        }
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&p.ctr->msgs, cnt[1]);
        atomicAdd(&p.ctr->probed, cnt[4]);
        atomicAdd(&p.ctr->prefiltered, cnt[7]);
        atomicAdd(&p.ctr->uniq, cnt[2]);
    }
    if (threadIdx.x == 0) {
        atomicAdd(&p.ctr->arcs, cnt[0]);
        atomicAdd(&p.ctr->staged, cnt[3]);
        atomicAdd(&p.ctr->accepted, cnt[5]);
        atomicAdd(&p.ctr->tier[1], cnt[6]);
    }
}

// Check records of all rows, from the label offsets and the probe index as
// they stand for the coming gather (a finished round returns at once).
__global__ void k_pack_hrec(const int64_t* loff, const uint32_t* lent, const uint64_t* hdesc, const int32_t* vbase,
                            uint4* hrec, int64_t n, RoundCounters* ctr) {
    if (ctr->done) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) {  // after k_collect: its list sizes; the next active list starts empty
        ctr->nO1_base = ctr->nO1;
        ctr->nG_base = ctr->nG = min(ctr->nG, kMaxSplit);
        if (ctr->nA > 0) ctr->nA_saved = ctr->nA;  // (0: the gather runs again)
        ctr->nA = 0;
    }
#pragma unroll 1
    for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n; v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t a = loff[v], len = loff[v + 1] - a;
        const uint64_t row = hrec_row((uint64_t)a, (uint64_t)len);
        // entries of L(v) with a top hub (rows are hub-sorted)
        const uint64_t top =
            (uint64_t)lower_bound_u32(lent + a, len, pack(base_of(vbase, v) + (uint32_t)kTopHubs, 0));
        const uint64_t hd = hdesc[v] | (top << (32 + kHrecTopShift));
        hrec[v] = make_uint4((uint32_t)row, (uint32_t)(row >> 32), (uint32_t)hd, (uint32_t)(hd >> 32));
    }
}

}  // namespace plb
