// Kernels of the vertex-centric labeling rounds (Alg. 3, Sec. 3.1), in rank
// space: vertex i is the vertex of rank i, so "h outranks v" is h < v.
//
// Round 1 is k_round1 (no candidate can be pruned).  Per round d >= 2
// (labels L and frontier dL_{d-1} as they stood after round d-1):
//   k_mark         every active a (dL_{d-1}(a) non-empty) flags the neighbours
//                  v that some hub of dL_{d-1}(a) outranks (scatter, Alg. 3).
//   k_collect      flagged vertices become this round's receivers, routed by
//                  their candidate bound, |L(v)| and degree to a tier.
//   k_gp_warp      gather + dedup + distance check, one vertex per warp, with
//                  L(v) staged hub-keyed in shared memory (the gather of
//                  Alg. 3: unique messages, then d < min over common hubs).
//   k_gp_block     the same with one vertex per block (any size: hub-range
//                  passes, a bitmap for the top hubs).
//   k_sort_rows_*  rows of the new frontier that were written unsorted (round
//                  1; the block tier's) sorted by hub rank (the warp tier
//                  writes its rows sorted);
//   k_merge_rows   L(v) <- L(v) U dL_d(v), keeping rows sorted by hub rank;
//                  then the probe index of L is rebuilt (k_index_*).
#pragma once

#include "plb_internal.cuh"

namespace plb {

struct RoundCounters {
    unsigned long long cursor;    // append cursor of the new frontier buffer
    unsigned long long accepted;  // new labels this round
    unsigned long long arcs, msgs, uniq, staged, probed;
    unsigned long long tier[3];
    unsigned long long bound_sum; // sum over receivers of the candidate bound min(v, messages), as padded rows
    unsigned long long prefiltered; // candidates pruned by the top-hub witness prefilter
    unsigned long long chk_lv, chk_lh;  // checked candidates (h at v): sums of |L(v) entries with hub < h|
                                        // and of |L(h)| (counted when GpParams::count_check is set)
    int nR, nO1, nO2;             // receivers: warp tier, block tier, escalated by the warp tier
    int nBig, nGiant;             // new frontier rows too long for a warp / for shared memory to sort
    int nU;                       // vertices whose new frontier row was written unsorted (block tier)
    int wkR, wkO1, wkO2;          // next entry of each tier's list (taken by whoever is free)
    int nG, nP;                   // split receivers and their parts (see SplitLists)
    int nO1_base, nG_base;        // list sizes made by k_collect (for reruns and statistics)
    int fovf;                     // new-frontier buffer overflow
    int nA;                       // next active list (kept across the per-round reset, which ends here)
    unsigned int max_dist;        // finalize: largest stored distance
    int guard;                    // a kernel met a broken capacity invariant (internal error)
    // loop control (kept across rounds)
    unsigned int d;               // current round (distance of the labels being accepted)
    int done;                     // no further round runs; round kernels return at once
    int fallback;                 // graph mode stopped at a capacity limit: resume on the host
    int err;                      // status set by the device (PLB_ERR_DIST_OVERFLOW)
    int nA_saved;                 // active count of the current round (restored on fallback)
    int cur;                      // buffer parity holding L and the previous frontier
    long long T;                  // labels so far (graph mode)
    long long lcap, hcap;         // label and probe-index buffer capacities (graph mode)
    long long fcap[2];            // new-frontier buffer capacity per parity (graph mode)
    long long hnext;              // probe index: first free table slot
    int hovf;                     // probe index: a table did not fit (the index must be rebuilt)
};

// RoundCounters::fallback: why a graph stopped (1: after the gather, a buffer
// was too small; kStopBeforeGather: the candidate bound exceeds the frontier
// buffer; kStopIndex: after a complete round, the probe index needs a rebuild).
constexpr int kStopBeforeGather = 2;
constexpr int kStopIndex = 3;

// Per-round statistics written on the device (graph mode).
struct RoundStat {
    long long receivers, accepted, uniq, probed, msgs, pref, arcs, staged, tier0, tier1, chk_lv, chk_lh;
};

// Receivers with many arcs (hubs) are split: blocks gather parts of kSplitPart
// arcs into shared-memory bitmaps and OR these into the receiver's global bitmap;
// the block that ends last goes on with the merged bitmap.  No block waits for
// another.  (One block takes 4 to 5 us per 256 arcs of dependent loads: a hub
// with 209,550 arcs kept a round from ending for up to 4 ms.)  Only for
// receivers whose hubs all fit the map.
constexpr int kSplitArcs = 2048;   // arcs from which a receiver is split
constexpr int kSplitPart = 1024;   // arcs per part
constexpr int kMaxSplit = 512;     // split receivers per round (further ones are not split)
struct SplitLists {
    int32_t* v;        // [max] receivers
    int* nparts;       // [max] parts of each
    int* done;         // [max] parts gathered (zero between launches)
    uint32_t* bits;    // [max x words] bitmaps (zero between launches)
    int2* parts;       // (receiver's index, part)
    int max, max_parts, words;
};

// The top-hub masks by hub instead of by vertex: per graph, level t and top hub
// w a row of bits over the graph's first vertices (those the block tier's map
// hold), bit x: w in L(x) at distance <= t.  A receiver prunes the candidates
// in its map 64 per lane and row: OR of the rows of its own top hubs.
struct TopColumns {
    uint32_t* bits;       // rows (t, w) of 4 one.y words each, from 4 x kTopRows x one.x words on
    const int2* by_base;  // disjoint union: {x, y} of each graph, at the index of its first rank; else null
    int2 one;             // one graph: {0, y}
};

struct GpParams {
    const int64_t* roff;
    const int32_t* rcol;
    const int64_t* loff;
    const uint32_t* lent;
    const uint64_t* fse;       // frontier of round d-1: start|count per vertex
    const uint32_t* fhub;      // frontier hubs of round d-1 (rows sorted)
    uint64_t* fse_new;         // frontier of round d
    uint32_t* fhub_new;
    unsigned long long fcap;   // capacity of fhub_new
    const int32_t* list;       // vertices handled by this tier
    const int* list_n;
    int* work;                 // counter that hands out the list's entries (after the parts)
    SplitLists split;          // block tier: parts to gather before the list's vertices (split.max = 0: none)
    int32_t* esc;              // escalation list (next tier)
    int* esc_n;
    RoundCounters* ctr;        // also holds the round number d (ctr->d)
    int log_s, log_m;          // table sizes (log2 slots): candidate set, L(v) map (block tier: largest)
    int cand_limit;            // max unique candidates per pass (power of two)
    int s_words;               // warp tier: words per warp of the set, the candidates and the top-hub masks
    uint32_t* gscratch;        // block tier: per-block buffer of accepted hubs
    int64_t gscratch_words;    // words per block
    const uint64_t* hdesc;     // probe index of L: per row (table start << 8 | log2 slots), 0 = no table
    const uint32_t* htab;
    int64_t n;                 // vertices
    const uint32_t* top;       // top-hub masks by distance level, then vertex (see kTopHubs)
    // The candidates' side of the check: rows, probe index and top-hub masks
    // of the labels h contributes (the same arrays as above for undirected
    // graphs; for L_in(v) of a directed graph the L_out of h, and vice versa).
    const int64_t* loff_h;
    const uint32_t* lent_h;
    const uint64_t* hdesc_h;
    const uint32_t* htab_h;
    const uint32_t* top_h;
    const uint4* hrec_h;       // per vertex of the candidates' side: {row start << 24 | row length (64
                               // bits), probe-table descriptor (64 bits)}, one 16-byte load per check
    const uint32_t* rbound;    // per receiver: candidate bound min(v, messages)
    const int64_t* ostart;     // per receiver: start of its new frontier row (the scan of the bounds),
                               // or null (rows reserved with an atomic cursor)
    int stage_ratio;           // warp tier: L(v) read from v's probe table when rbound[v] * stage_ratio
                               // < |L(v)| (0: always staged in shared memory)
    int32_t* unsorted;         // block tier: list of the vertices whose new row it wrote (unsorted;
                               // count ctr->nU), or null (every new row is sorted after the round)
    int sender_bits;           // rcol holds frontier descriptor indices whose low sender_bits bits are
                               // the sending vertex (weighted rounds), or 0: the vertex itself
    TopColumns cols_h;         // the candidates' side's top-hub masks by hub
    const int32_t* vbase;      // per vertex: first rank of its graph in a disjoint union, or null (one graph:
                               // 0).  The top hubs and the maps are those of the vertex's own graph
    int count_check;           // 1: count the label entries each check would read by the paper's cost
                               // model (RoundCounters::chk_lv / chk_lh; a search per candidate, or per 64
                               // hubs of the block tier's bitmap)
};

// First rank of v's graph (see GpParams::vbase).
__device__ __forceinline__ uint32_t base_of(const int32_t* vbase, int64_t v) {
    return vbase ? (uint32_t)vbase[v] : 0u;
}

// The sending vertex of an arc's descriptor index (see GpParams::sender_bits).
__device__ __forceinline__ uint32_t sender_of(const GpParams& p, int32_t a) {
    return p.sender_bits ? (uint32_t)a & ((1u << p.sender_bits) - 1u) : (uint32_t)a;
}

// Witness prefilter: for the kTopHubs highest-ranked hubs of its graph (in a
// disjoint union each graph has its own, ranks vbase .. vbase + kTopHubs - 1:
// the union's first 256 ranks all belong to its first graph; with those as the
// only masks a batch of 200 graphs of 1K-64K vertices settled 2% of its
// candidates without a scan and took 135.2 ms, with each graph's own it takes
// 69.3 ms), every vertex x keeps kTopLevels bitmasks C_t(x) = {w : w in L(x), d(w, x) <= t}, t = 1..
// kTopLevels (8 words each).  A candidate h at round d has a witness among
// those hubs when E_i(v) & C_{d-i}(h) != 0 for some i, E_i = C_i & ~C_{i-1}:
// the label test restricted to those hubs and distances (exact: a hit is a
// real witness).
#ifndef PLB_TOP_HUBS
#define PLB_TOP_HUBS 256
#endif
constexpr int kTopHubs = PLB_TOP_HUBS;  // a multiple of 128 (uint4 loads)
static_assert(kTopHubs % 128 == 0, "top-hub masks are read as uint4");
constexpr int kTopWords = kTopHubs / 32;             // words per mask
constexpr int kTopLevels = 7;                        // distance levels 1..7
constexpr int kTopRow = kTopLevels * kTopWords;      // words per vertex
constexpr int kTopRows = kTopLevels * kTopHubs;      // rows of TopColumns
// Layout: the masks of level 1 of all vertices, then level 2's, ...: a round
// reads one or two levels of candidates that are mostly of high rank, so that
// what it reads lies together (the 32-byte masks of 2^17 hubs in 4 MB; with
// all levels of a vertex side by side they were spread over 29 MB).

// Frontier rows start at multiples of kRowAlign hubs (32 bytes) and are filled
// up to one with kEmpty: the block tier reads them a sector at a time.
constexpr int kRowAlign = 8;
__host__ __device__ __forceinline__ int64_t row_pad(int64_t c) { return (c + kRowAlign - 1) & ~(int64_t)(kRowAlign - 1); }

// Block tier: the highest-ranked hubs (of the vertex's graph) are deduplicated
// in a shared-memory bitmap instead of the hash set.  On R-MAT 2^22 28% of round
// 3's messages and 32% of its candidates rank past 32,768, 1.6% and 2% past
// 131,072.  Every receiver of the block tier uses it (only those with 2,048
// candidates or more, the others hashing: R-MAT 2^22 741 instead of 722 ms).
// What shared memory leaves is the L1 cache, which the checks' masks, records
// and probe tables pass through: three blocks of either tier take 196 KB (a
// carve-out the SM offers; the next is 228) of its 256, so 60 KB are cache
// instead of 28.  Both have to: the tiers run side by side, and an SM keeps one
// carve-out for both (the block tier alone at 196 left R-MAT 2^22 at 616 ms when
// it ran beside the warp tier, 553 without).  16 KB of bytes (plain stores) for
// the first 16,384 hubs and 16 KB of bits for the next 131,072, at 228 KB, took
// 618 ms on R-MAT 2^22, 100 on directed R-MAT 2^20, 24.2 on Chung-Lu 2^20; this
// bitmap 535, 96 and 23.6 (131,072 or 196,608 hubs: within 1%; both tiers within
// 164 KB, by shorter candidate lists in the warp tier: 547, 104, 23.4).
constexpr int kMapHubs = 147456;
constexpr int kMapWords = kMapHubs / 32;
static_assert(kMapHubs % 4096 == 0, "whole scan units");
// Block tier, per warp: survivors of the first prefilter step (fewer than 32,
// plus 32 of one extraction).
constexpr int kWarpStage = 64;

// Rows of L with at least this many entries get a hub-keyed probe table.
constexpr int kIndexMinLen = 16;
// k_index_build: warps per block, and the largest table a warp may build in
// its shared-memory buffer (larger ones are filled in place).  The buffer is
// chosen per launch: 512 slots (16 KB per block, eight blocks per SM) while
// the rows are short, 2048 when they are long.
constexpr int kIndexWarps = 8;
constexpr int kIndexSmemSlotsMax = 2048;

// Check records (GpParams::hrec_h): row start << 24 | length, then the
// probe-table descriptor (table start << 8 | log2 slots, below 2^48) with the
// row's count of entries whose hub is one of its graph's kTopHubs in its top 16 bits.
__host__ __device__ __forceinline__ uint64_t hrec_row(uint64_t start, uint64_t len) { return (start << 24) | len; }
constexpr int kHrecTopShift = 16;  // within the record's last word
constexpr uint64_t kHrecDescMask = (uint64_t(1) << 48) - 1;
// A graph's rows and words per row (in units of 4) of the top-hub columns.
__device__ __forceinline__ uint32_t* columns_of(const TopColumns& c, uint32_t vb, uint32_t* words) {
    const int2 t = c.by_base ? c.by_base[vb] : c.one;
    *words = 4u * (uint32_t)t.y;
    return c.bits + (int64_t)t.x * (4 * kTopRows);
}
// Words per row, in units of 4, for a graph of n vertices: none for one of up to
// warp_only vertices (see warp_only_vertices), whose candidates are pruned by
// their own masks.  (A quad of columns takes 28,672 bytes: a union of a million
// graphs of 16 vertices had 28.7 GB of them, never read.)
inline int column_quads(int64_t n, int64_t warp_only) {
    if (n <= warp_only) return 0;
    const int64_t m = n < kMapHubs ? n : kMapHubs;
    return (int)((m + 127) / 128);
}
__global__ void k_pack_hrec(const int64_t* loff, const uint32_t* lent, const uint64_t* hdesc, const int32_t* vbase,
                            uint4* hrec, int64_t n, RoundCounters* ctr);

// Routing limits of k_collect (see the tier geometry in build_core).
struct TierLimits {
    int64_t warp_bound;   // candidate bound up to which the warp tier is tried
    int64_t short_bound;  // the same with |L(v)| <= short_label
    int64_t short_label;
    int64_t warp_label;   // largest |L(v)| of the warp tier
    int64_t warp_deg;     // largest degree of the warp tier
    int64_t warp_msgs;    // most messages of the warp tier (rows of the neighbours, not cut at v)
};

struct WarpSync {
    __device__ void operator()() const { __syncwarp(); }
};
struct BlockSync {
    __device__ void operator()() const { __syncthreads(); }
};

}  // namespace plb
