// Host-side helpers of the build drivers (undirected: plb_build.cu;
// directed: plb_directed.cu; weighted: plb_weighted.cu): device allocations
// of one build, CUDA-event timers, launch geometry, the last CUDA error of
// this thread.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdio>
#include <initializer_list>
#include <vector>

#include "plb_round.cuh"

namespace plb {

constexpr int kFlatThreads = kTileThreads;
constexpr int kGpWarpThreads = 256;

// Device allocations of one build (stream-ordered, from the library pool),
// all returned when the build ends.
struct DevPool {
    cudaStream_t s;
    std::vector<void*> ptrs;
    bool failed = false;
    explicit DevPool(cudaStream_t st) : s(st) {}
    template <typename T>
    T* alloc(int64_t count) {
        void* p = nullptr;
        const size_t bytes = (size_t)std::max<int64_t>(count, 1) * sizeof(T);
        if (plb::dev_alloc(&p, bytes, s) != cudaSuccess) {
            (void)cudaGetLastError();
            failed = true;
            return nullptr;
        }
        ptrs.push_back(p);
        return static_cast<T*>(p);
    }
    void release(void* p) {
        auto it = std::find(ptrs.begin(), ptrs.end(), p);
        if (it != ptrs.end()) {
            cudaFreeAsync(p, s);
            ptrs.erase(it);
        }
    }
    // Frees every allocation except those in keep (stream-ordered).
    void release_all_except(std::initializer_list<const void*> keep) {
        std::vector<void*> kept;
        for (void* p : ptrs) {
            if (std::find(keep.begin(), keep.end(), p) != keep.end()) kept.push_back(p);
            else cudaFreeAsync(p, s);
        }
        ptrs.swap(kept);
    }
    ~DevPool() {
        for (void* p : ptrs) cudaFreeAsync(p, s);
    }
};

// CUDA-event spans per kernel class (profile option).
struct Timer {
    bool on;
    cudaStream_t s;
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev[8];
    std::vector<cudaEvent_t> all;  // every event once (spans may share an end point)
    explicit Timer(bool enabled, cudaStream_t st) : on(enabled), s(st) {}
    cudaEvent_t mark() {
        cudaEvent_t e;
        cudaEventCreate(&e);
        cudaEventRecord(e, s);
        all.push_back(e);
        return e;
    }
    void span(int cls, cudaEvent_t a, cudaEvent_t b) { ev[cls].push_back({a, b}); }
    double total(int cls) {
        double t = 0;
        for (auto& p : ev[cls]) {
            float ms = 0;
            cudaEventElapsedTime(&ms, p.first, p.second);
            t += ms;
        }
        return t;
    }
    ~Timer() {
        for (cudaEvent_t e : all) cudaEventDestroy(e);
        (void)cudaGetLastError();
    }
};
enum { T_PREP = 0, T_FRONT = 1, T_GPW = 2, T_GPB = 3, T_GPG = 4, T_MERGE = 5, T_FINAL = 6, T_ALL = 7 };

inline int grid_for(int64_t items, int threads, int max_blocks) {
    int64_t b = (items + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > max_blocks) b = max_blocks;
    return (int)b;
}

inline int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 132;
    }
    return sms;
}

inline int pow2_at_least(int64_t x) {
    int p = 1;
    while (p < x) p <<= 1;
    return p;
}

// Dynamic shared memory of k_gp_block in bytes, in the order the kernel
// carves it up: scalars (48 words) + warp sums (34, padded to 36) + histogram
// (256) + top-hub masks + prefix per thread + 64-bit row start per thread + set
// (also kWarpStage per warp of staged candidates) + map + candidate list
// (limit + 32 per warp) + hub map.  The masks, the set and the hub map are
// read as 16-byte words.
inline size_t gp_block_smem_bytes(int bthr, int log_s, int log_m, int cand_limit) {
    return sizeof(uint32_t) * (48 + 36 + 256 + kTopRow + (size_t)((bthr + 4) & ~3) + 2 * (size_t)bthr +
                               ((size_t)1 << log_s) + ((size_t)1 << log_m) + (size_t)cand_limit + (size_t)bthr +
                               kMapWords);
}

// Warp tier: words per warp for the set (2^log_s slots), the candidates and the
// top-hub masks, which lie in the set's last words: for the default options
// three blocks then take 196 KB of an SM's 256, as the block tier's do (with the
// masks beside the set 198: see kMapHubs).  Small sets keep all their slots for
// candidates.
inline int warp_set_words(int log_s) { return log_s >= 10 ? 1 << log_s : (1 << log_s) + kTopRow; }
inline size_t gp_warp_smem_bytes(int warps, int log_s, int log_m) {
    return sizeof(uint32_t) * (size_t)warps * (4 + (size_t)warp_set_words(log_s) + ((size_t)1 << log_m));
}

// Whether the tables of the options fit: the bounds are those of the larger
// layouts that the options were specified with (a hub map of 32 KB, masks beside
// the set).
inline bool tiers_fit(int warps, int w_log_s, int w_log_m, size_t b_smem) {
    const size_t w = sizeof(uint32_t) * (size_t)warps * (4 + kTopRow + ((size_t)1 << w_log_s) + ((size_t)1 << w_log_m));
    return w <= 227 * 1024 && b_smem - sizeof(uint32_t) * kMapWords + 32768 <= 227 * 1024;
}

// Tier of a receiver.  The bound counts messages; the candidates, which have to
// fit the warp tier's list (968 for the default 512), are fewer, by 2 to 5 times
// on power-law graphs in degree order, and a receiver with more goes on to the
// block tier.  With the bound at 2 x warp_cand for all, the block tier took
// receivers that a warp finishes sooner than a block starts; with long rows L(v) a
// warp does less well (staging them, and no pruning by columns) and keeps that
// bound.  All rows 2 | 3 | 4 | 8 x warp_cand | 4 x up to 128 entries and 2.5 x beyond,
// ms: Chung-Lu 2^20 23.4 | 22.2 | 21.9 | 22.0 | 21.8; batch of 200 graphs 47.7 |
// 46.2 | 45.5 | 45.6 | 45.6; directed R-MAT 2^20 95.8 | 93.4 | 94.4 | 98.7 | 93.4;
// R-MAT 2^22 535.6 | 536 | 538 | 545 | 537; 1.5 x: 25.1, 49.3, 100.6, 547.  Rows up
// to which the larger bound holds, none | 64 | 128 | 256 | any: Chung-Lu 22.8 |
// 22.1 | 22.1 | 22.1 | 22.2; batch 45.5 | 44.5 | 44.5 | 44.5 | 44.6; directed 91.6 |
// 90.7 | 90.9 | 91.8 | 92.1; R-MAT 2^22 532 | 534 | 535 | 535 | 535.  Longer rows 1.5 |
// 2 | 2.5 x: Chung-Lu 22.0 | 22.2 | 22.3, directed 89.7 | 89.2 | 89.3, batch, weighted
// and R-MAT 2^22 equal; in random order, where rows are long and few messages
// repeat, Chung-Lu with 5,000 vertices 9.6 | 10.1 | 10.5, R-MAT 2^13 10.4 | 10.9 |
// 11.3.  What a wider bound costs: receivers whose candidates do not fit after all
// are gathered twice, the second time beside nothing else (see launch_tiers).
// In dense graphs few candidates come in very many messages, 8 us per thousand for
// a warp: receivers with more than warp_msgs are gathered by a block.  Complete
// graphs of 600 | 900 | 1,500 vertices took 2.4 | 6.2 | 13.7 ms without this limit
// (warps with half a million messages each, crowded into the SMs that the block tier
// left first), 1.0 | 1.2 | 2.3 with it (262,144: 2.4 | 1.2 | 2.3; counting the rows as
// they are cut at v: 1.4 | 2.2 | 3.1); directed R-MAT 2^20 90.8 ms without, 88.9 with
// it, the other builds equal.  16,384 is up to 2% faster still, but then graphs from
// 182 vertices instead of 363 have columns (warp_only_vertices).
inline TierLimits tier_limits(int warp_cand, int warp_label) {
    TierLimits lim;
    lim.warp_bound = 2 * (int64_t)warp_cand;
    lim.short_bound = 4 * (int64_t)warp_cand;
    lim.short_label = 128;
    lim.warp_label = warp_label;
    lim.warp_deg = (int64_t)32 * 64;
    lim.warp_msgs = 65536;
    return lim;
}

// The most vertices of a graph whose receivers all stay in the warp tier: arcs,
// label row, candidate bound and candidates are each at most the vertex count,
// and the tier's limits on them are no smaller than these (tier_limits; the set
// holds warp_cand entries, the candidate list as many); a neighbour of rank a
// sends at most a hubs, so the messages are at most n (n - 1) / 2.  Only a CSR
// with repeated arcs, which the input check refuses, can take such a receiver to
// the block tier.
inline int64_t warp_only_vertices(const plb_options& o) {
    const int warp_cand = pow2_at_least(std::max(32, o.warp_cand_cap)), warp_label = std::max(16, o.warp_label_cap);
    const TierLimits lim = tier_limits(warp_cand, warp_label);
    int64_t n = std::min<int64_t>({warp_cand, warp_label, lim.warp_deg});
    while (n * (n - 1) / 2 > lim.warp_msgs) --n;
    return n;
}

// Lists and bitmaps of the split receivers of a build over n vertices (the
// largest graph of a union: max_part_n) and nnz arcs.  A receiver is split from
// kSplitArcs arcs on, so at most nnz / kSplitArcs receivers are, and their
// parts number at most nnz / kSplitPart + one each.
inline SplitLists split_lists(DevPool& pool, int64_t n, int64_t max_part_n, int64_t nnz, cudaStream_t s) {
    SplitLists l{};
    const int64_t most = std::min<int64_t>(kMaxSplit, nnz / kSplitArcs);
    if (most <= 0 || n <= 0) return l;
    l.max = (int)most;
    l.max_parts = (int)(nnz / kSplitPart + most);
    l.words = (int)((std::min<int64_t>(max_part_n, kMapHubs) + 31) / 32);
    l.v = pool.alloc<int32_t>(most);
    l.nparts = pool.alloc<int>(most);
    l.done = pool.alloc<int>(most);
    l.bits = pool.alloc<uint32_t>(most * l.words);
    l.parts = pool.alloc<int2>(l.max_parts);
    if (pool.failed || cudaMemsetAsync(l.done, 0, sizeof(int) * most, s) != cudaSuccess ||
        cudaMemsetAsync(l.bits, 0, sizeof(uint32_t) * most * l.words, s) != cudaSuccess)
        pool.failed = true;
    return l;
}

// The block tier's stream beside the build's own, with its fork and join events.
// Declared after the build's DevPool: a build that fails between fork and join
// waits here for the side stream's kernels, since the pool takes their buffers
// back in the order of the build's own stream, which has not joined them.
struct SideStream {
    cudaStream_t st = nullptr;
    cudaEvent_t fork = nullptr, join = nullptr;
    bool open = false;  // launched into, and not joined
    cudaError_t create() {
        cudaError_t e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
        return e;
    }
    ~SideStream() {
        if (open) cudaStreamSynchronize(st);
        if (fork) cudaEventDestroy(fork);
        if (join) cudaEventDestroy(join);
        if (st) cudaStreamDestroy(st);
    }
};

// One gather + prune of a round.  The two tiers run side by side (in a captured
// round the side stream becomes a branch of the graph):
// the block tier on the side stream over k_collect's block list O1 (and the
// split receivers), the warp tier on the build's stream, escalating into O2,
// which one more block-tier launch takes after both (the tails of the two
// kernels overlap).  w, b: the tiers' parameters without lists; tm and mark:
// where to record the end of the warp tier (profiled builds), or null.
inline cudaError_t launch_tiers(GpParams w, GpParams b, const SplitLists& split, int32_t* O1, int32_t* O2,
                                RoundCounters* ctr, int grid_w, size_t w_smem, int grid_b, int bthr, size_t b_smem,
                                cudaStream_t s, SideStream& side, Timer* tm, cudaEvent_t* mark = nullptr) {
    w.list_n = &ctr->nR;
    w.work = &ctr->wkR;
    w.esc = O2;
    w.esc_n = &ctr->nO2;
    b.esc = nullptr;  // the block tier never escalates
    b.esc_n = nullptr;
    b.list = O1;
    b.list_n = &ctr->nO1;
    b.work = &ctr->wkO1;
    b.split = split;
    cudaError_t e = cudaEventRecord(side.fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side.st, side.fork, 0);
    if (e != cudaSuccess) return e;
    side.open = true;
    k_gp_block<<<grid_b, bthr, b_smem, side.st>>>(b);
    k_gp_warp<<<grid_w, kGpWarpThreads, w_smem, s>>>(w);
    if (tm) *mark = tm->mark();
    e = cudaEventRecord(side.join, side.st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, side.join, 0);
    if (e != cudaSuccess) return e;
    side.open = false;
    b.list = O2;
    b.list_n = &ctr->nO2;
    b.work = &ctr->wkO2;
    b.split = SplitLists{};
    k_gp_block<<<grid_b, bthr, b_smem, s>>>(b);
    return cudaGetLastError();
}

// Block tier, per block: accepted hubs past the map (those within it stay
// marked there).
inline int64_t accepted_words(int64_t max_part_n) {
    return std::max<int64_t>(max_part_n - kMapHubs, 1);
}

// The top-hub columns of a graph, empty (quads: the words per row, in units of 4,
// of all graphs of a union, see column_quads; by_base: their places).
inline TopColumns top_columns(DevPool& pool, int64_t quads, const int2* by_base, cudaStream_t s) {
    TopColumns c{};
    c.by_base = by_base;
    c.one = make_int2(0, (int)quads);
    c.bits = pool.alloc<uint32_t>(quads * 4 * kTopRows);
    if (!pool.failed && cudaMemsetAsync(c.bits, 0, sizeof(uint32_t) * quads * 4 * kTopRows, s) != cudaSuccess)
        pool.failed = true;
    return c;
}

// Records the failing CUDA call for plb_last_error (this thread).
void set_last_error(cudaError_t e, int line);

}  // namespace plb
