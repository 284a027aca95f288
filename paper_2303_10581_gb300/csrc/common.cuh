// common.cuh -- shared device definitions of the octagon-filter hull path:
// workspace layout, order-preserving float keys, the exact orientation
// predicate and the bounded-wait helpers.
//
// Method: Carrasco et al., "An Evaluation of GPU Filters for Accelerating
// the 2D Convex Hull", Sec. 3 / Algorithm 1.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "../../include/convhull.h"

namespace ch {

// ---------------------------------------------------------------------------
// launch geometry
// ---------------------------------------------------------------------------
constexpr int kExtThreads = 512;      // extremes sweep
constexpr int kExtPairs = 2048;       // point pairs (16 B) per extremes tile: 32 KB
constexpr int kFiltThreads = 256;     // fused test + compaction
constexpr int kFiltItems = 16;        // points per thread per tile
constexpr int kFiltTile = kFiltThreads * kFiltItems;   // 4096 points = 32 KB
constexpr int kFiltMaxBlocks = 4096;                  // grid cap of the two-pass filter
// Tiles [first_tile(T, G, b), first_tile(T, G, b + 1)) are block b's in the
// two-pass filter and in the passes that follow its count pass (G <= T
// blocks): shares that differ by one tile at most.  (Equal shares, the last
// blocks without any, left 119 of 608 blocks idle on 2442 tiles.)
__host__ __device__ inline int64_t first_tile(int64_t tiles, int64_t blocks, int64_t b) { return b * tiles / blocks; }
constexpr int kSortTile = 4096;       // keys per sort tile
constexpr int kSortPasses = 4;        // 32-bit x keys, 8-bit digits
constexpr int kLeafC = 16;            // points per leaf chain (one thread)
constexpr int kChainThreads = 256;    // leaves per super-chunk (one block)
constexpr int kChainC = kLeafC * kChainThreads;   // 4096 points per super-chunk
constexpr int kChainStride = kChainC + 8;          // chain slots per super-chunk (up to kChainC + 1 used)
constexpr int kElimPasses = 12;       // cap on the per-warp elimination passes
constexpr int kElimRounds = 24;       // cap on the rounds over a side's whole sequence
constexpr int kEmitThreads = 256;     // chunks per emit tile (one per thread)
constexpr int64_t kMaxHullN = (int64_t)1 << 30;
constexpr int64_t kMaxN = ((int64_t)1 << 32) - 1;

// device error codes mirror ch_status
constexpr uint32_t kErrNonFinite = CH_ERR_NONFINITE;
constexpr uint32_t kErrTimeout = CH_ERR_TIMEOUT;
// bounded waits: polls before a look-back wait is declared dead (each poll
// is followed by a short nanosleep once the first few fail)
constexpr uint32_t kSpinLimit = 1u << 22;

// look-back status words: [flag:2 | value:62]
constexpr uint64_t kFlagA = 1ull << 62;   // tile aggregate published
constexpr uint64_t kFlagP = 2ull << 62;   // inclusive prefix published
constexpr uint64_t kValMask = (1ull << 62) - 1;
// 32-bit variant for the radix-sort digit status: [flag:2 | value:30]
constexpr uint32_t kFlagA32 = 1u << 30;
constexpr uint32_t kFlagP32 = 2u << 30;
constexpr uint32_t kVal32 = (1u << 30) - 1;

// ---------------------------------------------------------------------------
// filter polygon (Sec. 3.1 -> Sec. 3.2)
// ---------------------------------------------------------------------------
struct Octagon {
    // edge k runs from vertex k to vertex k+1 (mod 8), vertices in the
    // order R, TR, T, TL, L, BL, B, BR
    float ax[8], ay[8];     // edge start
    float bx[8], by[8];     // edge end
    uint32_t valid;         // bit k: edge k has non-zero length
    uint32_t has_edges;     // at least one valid edge
    uint32_t abort;         // non-finite input: later stages do nothing
    uint32_t spec;          // 1: the speculative sweep's candidates hold every survivor
    float xl, xh, yl, yh;   // closed quick-discard rectangle (xl > xh: none)
    float cx, cy;           // bounding-box centre: origin of the affine forms, centre of the fan
    float bxl, bxh, byl, byh;   // closed bounding box of the eight vertices
    uint32_t box_check;     // 1: points may lie outside that box (caller-supplied vertices)
    float scale;            // power of two: the fan works on points times this (1 for boxes of ordinary sizes)
    float tx[8], ty[8], tz[8];   // edge k's affine form (octtest.cuh)
};

// extremes reduction state: left zeroed by the last block of every sweep.
// (No call zeroes it, so it lies at the same place in the workspace for every
// n: calls on other sizes must find it as it was left.)
struct ExtCtrl {
    unsigned long long ext_slot[8];   // packed (key, index) per extreme
    uint32_t ext_done;                // extremes blocks finished
    uint32_t nonfinite;               // a non-finite coordinate was seen
    uint32_t sample_kmax[8];          // ord_key of the speculative sample's largest slot keys
    uint32_t sample_done;             // its blocks finished
};

// second throw-away step of the hull step (kgon.cu): a fan of triangles
// around the bounding-box centre, one vertex per angular bin
// (27648 vertices of 8 bytes are 216 KB: with the filter pass's queues beside
// them, as many as one block's shared memory holds)
constexpr int kFanBins = 27648;

constexpr uint32_t kKgonMinS = 1u << 16;   // fewer octagon survivors: not worth a fan
struct KgonCtrl {                          // zeroed with the control block
    unsigned long long slot[kFanBins];     // packed (far_key << 32 | ~index): farthest sampled input point per bin
    uint32_t sample, inside;               // points sampled for the bins, octagon survivors among them
    uint32_t s_oct;                        // octagon survivors
    uint32_t rho_inv;                      // ~bits of a lower bound (binary32) on the squared distance from
                                           // c to the fan's boundary, the largest so far
    uint32_t edges;                        // consecutive vertex pairs with v != w
    uint32_t gaps;                         // 1: some of them not proven counter-clockwise around c
    uint32_t pad[2];
};

// second fan level (kgon.cu): over the first level's survivors, kFan2Sub
// sub-bins per bin, each vertex the farthest survivor of its sub-bin
constexpr int kFan2Sub = 8;
constexpr int kFan2Bins = kFanBins * kFan2Sub;   // 221184
constexpr uint32_t kFan2MinS = 1u << 19;         // fewer survivors of the first level: the sort takes them
constexpr int64_t kFan2MinN = 1 << 19;           // smaller sets get no tables

struct Fan2Ctrl {                          // zeroed with the control block
    uint32_t on;                           // 1: the second level runs this call
    uint32_t count_in;                     // survivors of the first level, its input
    uint32_t bad;                          // 1: no usable vertices (nothing is dropped)
    uint32_t kept;                         // survivors of the second level
    uint32_t done;                         // test blocks finished
    uint32_t edges;                        // consecutive vertex pairs with v != w
    uint32_t pad[2];
};

// (The vertices before empty bins are filled, x = NaN for none, lie in pay[1],
// free until the second level or the sort: a set with a fan has kKgonMinS
// points.)
static_assert(kFanBins <= (int)kKgonMinS, "a set's second payload buffer holds a vertex per bin");
struct Kgon {
    float cx, cy;                          // fan centre (it and the vertices times Octagon::scale)
    uint32_t ok;                           // 0: no fan this call
    uint32_t centre;                       // 1: c lies clearly inside the octagon
    float2 v[kFanBins];                    // vertex of every bin (x = NaN: none, and the wedges beside it keep their points)
};

// K-direction filter polygon (kfilter.cu; the learned proposal's filter)
constexpr int kMaxDirs = 64;

struct KxCtrl {                            // left zeroed by the last block of every sweep
    unsigned long long slot[kMaxDirs];     // packed (ord(key) << 32 | ~index) per direction
    uint32_t done;                         // sweep blocks finished
    uint32_t nonfinite;                    // a non-finite coordinate was seen
};

struct KPoly {
    uint32_t K;
    uint32_t nvalid;                       // edges of non-zero length
    unsigned long long valid;              // bit k: edge k (vertex k -> k+1) has non-zero length
    float xl, xh, yl, yh;                  // closed quick-discard rectangle (xl > xh: none)
    float cx, cy;                          // vertex bounding-box centre (facing-edge hint)
    uint32_t convex;                       // every vertex on or left of every valid edge, centre strictly inside
    uint32_t pad;
    float ax[kMaxDirs], ay[kMaxDirs];      // edge k: vertex k ...
    float bx[kMaxDirs], by[kMaxDirs];      // ... to vertex k + 1
};

// control block: zeroed at the start of every call (together with the
// filter's look-back status, which follows it)
struct Ctrl {
    uint32_t filt_ticket;             // tile tickets of the fused filter
    uint32_t surv_count;              // survivors
    uint32_t sort_ticket[kSortPasses];
    uint32_t hist[kSortPasses][256];  // digit histograms of the survivor keys
    uint32_t pass_src[kSortPasses];   // 0/1: buffer a pass reads
    uint32_t pass_skip[kSortPasses];  // pass is an identity (one digit only)
    uint32_t final_buf;               // buffer holding the sorted keys
    uint32_t hist_done;
    uint32_t emit_ticket[2];
    uint32_t h_lower, h_upper;
    uint32_t sort_in;                 // buffer holding the survivors for the sort (the filter writes buffer 0)
    uint32_t small_done;              // the one-block hull of few survivors wrote the hull: later kernels stop
};

// Points the sort and chain kernels of a single-set hull work on: none
// when the call was aborted or the one-block hull already finished it.
__device__ __forceinline__ uint32_t hull_stage_count(const Ctrl *ctrl, const Octagon *oct)
{
    return (oct->abort || ctrl->small_done) ? 0u : ctrl->surv_count;
}

// Speculative single sweep (extremes.cu, filter.cu): a test region from an
// input sample; the extremes sweep keeps the points it cannot prove inside
// it (the candidates: index in the second key buffer, point in the second
// payload buffer).  Segment j holds the candidates of sweep block j, in
// one slice of `cap` slots per warp.
constexpr int kSpecMaxSeg = 2048;         // sweep blocks (segments) at most
constexpr int kSpecWarps = kExtThreads / 32;   // slices per segment
constexpr int kSpecCapDiv = 32;           // all slices together hold n / 32 candidates
constexpr int kSpecKeptSmem = 2048;       // survivors per segment ranked in shared memory
constexpr int64_t kSpecMinN = 1 << 22;    // smaller sets: the plain two passes
struct SpecCtrl {                         // written anew by every call that speculates
    uint32_t fail;                        // a slice overflowed: fall back (zeroed by the sample kernel)
    uint32_t nseg;                        // segments (sweep blocks) of this call
    uint32_t cap;                         // candidate slots per slice
    uint32_t scnt[kSpecMaxSeg * kSpecWarps];   // candidates written per slice
    uint32_t skept[kSpecMaxSeg];          // survivors of the octagon per segment (their slots in utmp)
};

// ch_hull_learned: features, activations and outputs of the MLP, and the
// polygon it picks (K and the directions)
struct LearnScratch {
    float feat[1024];
    float out[68];
    float dirs[2 * kMaxDirs];
    int32_t K;
    int32_t pad[3];
};

// persistent words: survive calls, cleared by ch_last_error
struct Persist {
    uint32_t error;
    uint32_t error_site;
    uint32_t pad[62];
};

// Workspace layout for a problem of up to n points.
struct Layout {
    size_t persist, extctrl, oct, ext8;
    size_t kxctrl, kpoly;   // KxCtrl (self-resetting), KPoly
    size_t ctrl;            // Ctrl, immediately followed by
    size_t filt_status;     // u64[filt_tiles],
    size_t kgon_ctrl;       // KgonCtrl,
    size_t fan2;            // Fan2Ctrl,
    size_t fan2_slot;       // u64[fan2_bins]: per sub-bin the farthest survivor (far_key << 32 | ~position),
    size_t node_cnt;        // u32[n_nodes]: arrivals per merge-tree node, and
    size_t emit_status[2];  // u64[emit_tiles]: look-back of the chain compaction
    size_t zero_words;      // u64 words from ctrl to the end of emit_status[1]
    size_t keys[2];         // u32[n]: ord(x) of each survivor (sort key)
    size_t pay[2];          // u64[n]: ord(y) << 32 | point index (sort payload)
    size_t sort_status[2];  // u32[sort_tiles * 256]
    size_t chain_pos[2];    // u32[n_chunks * kChainStride]: sorted positions of chain vertices
    size_t chain_pt[2];     // float2[n_chunks * kChainStride]: their coordinates
    size_t chunk;           // int32[8 * n_chunks]: loL hiL loU hiU prvL nxtL prvU nxtU
    size_t node;            // int32[4 * n_nodes]: firstL lastL firstU lastU
    size_t emit_off[2];     // u32[n_chunks + 1]: output offset of each super-chunk's chain range, per side
    size_t keep_bits;       // u16[filt_tiles * kFiltThreads]: keep decisions of the count pass
    size_t filt_bsum;       // u32[kFiltMaxBlocks]: survivors per block of the count pass
    size_t kgon;            // Kgon
    size_t utmp;          // u32[n]
    size_t spec, p0;        // SpecCtrl, the speculative sweep's test region (SpecBox, extremes.cu)
    size_t learn;           // the learned proposal's scratch (LearnScratch)
    size_t fan2_v;          // float2[fan2_bins + 4]: the second fan level's vertices, the ends repeated
    size_t total;
    int64_t n, filt_tiles, sort_tiles, n_chunks, n_nodes, emit_tiles;
    int64_t fan2_bins;      // kFan2Bins for sets of at least kFan2MinN points, else 0 (no second level)
};

__host__ __device__ inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

__host__ __device__ inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

__host__ __device__ inline int64_t tree_nodes(int64_t nc)
{
    // nodes of all levels >= 1 of the binary merge tree over nc leaves
    int64_t total = 0, w = nc;
    while (w > 1) {
        w = (w + 1) / 2;
        total += w;
    }
    return total;
}

// Per-set bookkeeping of ch_hull_batched (all positions are global).
struct SetInfo {
    int64_t pt_begin;     // first point of the set in pts
    int64_t n;            // points in the set
    uint32_t tile_base;   // first 4096-point tile of the set
    uint32_t ntiles;
    uint32_t s;           // survivors of the filter
    uint32_t sc_base;     // first 4096-survivor super-chunk (= sort tile) of the set
    uint64_t surv_base;   // first survivor of the set in the sort arrays
    uint32_t nsc;         // super-chunks of the set
    uint32_t node_base;   // first merge-tree node of the set
    uint32_t hull;        // hull vertices of the set
    uint32_t pad[3];
};

// Batch-wide counters of ch_hull_batched (zeroed at the start of a call).
struct BatchCtrl {
    uint32_t tiles;       // point tiles over all sets
    uint32_t nsc;         // super-chunks over all sets
    uint32_t abort;       // bad offsets: nothing is computed
    uint32_t filt_ticket, emit_ticket;
    uint32_t nsc_sort;    // the sort's tiles among them (the sets that the chain kernel sorts come after)
    uint32_t sort_ticket[kSortPasses];
    uint32_t h_lower, h_upper;
    uint32_t nfan;        // sets that get a fan (kgon.cu)
    uint32_t nfan_items, nplain_items, nbin_items;   // work items
    uint32_t fan_ticket, plain_ticket;               // next work item of the filter passes
};
// The chain kernel sorts a set of so few survivors itself.  (1000 sets of 10^2
// to 10^4 points: 390 us with none, 364 so, 433 with 4096: the sort's passes
// run beside one another and wait for the larger sets anyway.)
constexpr uint32_t kBxLocalMax = 1024;
constexpr int kBxFanChunk = 32;       // tiles per work item of the fan sets' filter pass (built-in)
constexpr int kBxFanChunkMin = 8;     // the smallest tunable one (sizes the work-item lists)
constexpr int kBxTileBins = 1024;     // a set has up to this many bins per tile of 4096 points (kFanBins at most)
constexpr int kBxBinRun = 512;        // bins per block of the vertex kernel
constexpr int64_t kBxFanMinN = 16384; // smaller sets get no fan
constexpr int kBxPlainChunk = 16;     // tiles per work item of the sets without a fan
static_assert(2 * ((kBxFanMinN + kFiltTile - 1) / kFiltTile * kBxTileBins) + 1 <= kBxFanMinN && 2 * kBxTileBins < kFiltTile,
              "a set's stretch of the sort's payloads holds its fan tables");

// The fan of a set of ch_hull_batched.
struct FanInfo {
    uint32_t want;        // enough octagon survivors (an estimate) for a fan
    uint32_t tight;       // the points' distances from the centre differ by rounding only (a circle)
    uint32_t nb;          // bins
    uint32_t ready;       // the fan's proofs hold and it drops enough points
    float rho2;           // lower bound on the squared (scaled) distance from the centre to the fan's boundary (0: none)
};

// Extra workspace of ch_hull_batched, after the single-set regions.
struct BatchLayout {
    size_t sets;          // SetInfo[B]
    size_t octs;          // Octagon[B]
    size_t zero_begin;    // ---- zeroed by one memset per call:
    size_t bctrl;         // BatchCtrl
    size_t ext_slot;      // u64[B * 8]: packed extremes per set
    size_t nonfinite;     // u32[B]
    size_t hist;          // u32[B * kSortPasses * 256]
    size_t zero_end;      // ----
    size_t tile_set;      // u32[tiles_max]: set of each point tile
    size_t sc_set;        // u32[tiles_max]: set of each super-chunk
    size_t sc_off[2];     // u32[tiles_max + 1]: lower / upper chain offset of each super-chunk
    size_t lower;         // keys[1] again: free for the stages after the sort, which ends in buffer 0
    // the fan of the hull step, per set with many octagon survivors (kgon.cu)
    size_t soct;          // u32[B]: survivors per set (in the zeroed range)
    size_t fan;           // FanInfo[B]
    size_t fan_set;       // u32[max_fan]: the sets with a fan
    size_t fan_tab;       // the sets' fan tables: pay[1], free until the sort.  In a set's own stretch (from the
                          // first even point position): u64[nb], the farthest sampled point per bin, later the
                          // vertices, then float2[nb], the vertices before empty bins are filled.  (A set with
                          // a fan has at least kBxFanMinN points, and 2 nb + 1 <= n then.)
    size_t fan_items;     // uint2[max_items]: (set, first tile in the set) of each work item of the fan sets
    size_t plain_items;   // uint2[max_plain_items]: the same of the other sets
    size_t bin_items;     // uint2[max_bin_items]: (set, first bin) of each run of kBxBinRun bins
    size_t total;
    int64_t num_sets, tiles_max, max_fan, max_items, max_plain_items, max_bin_items;
};

__host__ __device__ inline Layout make_layout(int64_t n, int64_t sets = 0)
{
    Layout L{};
    if (n < 1) n = 1;
    L.n = n;
    L.filt_tiles = ceil_div(n, kFiltTile);
    L.sort_tiles = ceil_div(n, kSortTile);
    L.n_chunks = ceil_div(n, kChainC);
    L.n_nodes = tree_nodes(L.n_chunks) + 1;
    if (sets > 0) {
        // every set adds at most one ragged tile / super-chunk, and each
        // set's merge tree has fewer than twice as many nodes as leaves
        L.filt_tiles = L.n_chunks = ceil_div(n, kChainC) + sets;
        L.sort_tiles = L.sort_tiles > L.n_chunks ? L.sort_tiles : L.n_chunks;
        L.n_nodes = 2 * L.n_chunks + sets;
    }
    L.emit_tiles = ceil_div(L.n_chunks, kEmitThreads);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o = align_up(o + bytes, 256);
        return at;
    };
    L.persist = take(sizeof(Persist));
    L.extctrl = take(sizeof(ExtCtrl));
    L.oct = take(sizeof(Octagon));
    L.ext8 = take(8 * sizeof(uint32_t));
    L.kxctrl = take(sizeof(KxCtrl));
    L.kpoly = take(sizeof(KPoly));
    L.ctrl = take(sizeof(Ctrl));
    L.filt_status = take((size_t)L.filt_tiles * 8);
    L.kgon_ctrl = take(sizeof(KgonCtrl));
    L.fan2_bins = (sets == 0 && n >= kFan2MinN) ? kFan2Bins : 0;
    L.fan2 = take(sizeof(Fan2Ctrl));
    L.fan2_slot = take((size_t)L.fan2_bins * 8);
    L.node_cnt = take((size_t)L.n_nodes * 4);
    L.emit_status[0] = take((size_t)L.emit_tiles * 8);
    L.emit_status[1] = take((size_t)L.emit_tiles * 8);
    L.zero_words = (L.emit_status[1] + (size_t)L.emit_tiles * 8 - L.ctrl + 7) / 8;
    L.keys[0] = take((size_t)n * 4);
    L.keys[1] = take((size_t)n * 4);
    L.pay[0] = take((size_t)n * 8);
    L.pay[1] = take((size_t)n * 8);
    L.sort_status[0] = take((size_t)L.sort_tiles * 256 * 4);
    L.sort_status[1] = take((size_t)L.sort_tiles * 256 * 4);
    for (int side = 0; side < 2; ++side) {
        L.chain_pos[side] = take((size_t)L.n_chunks * kChainStride * 4);
        L.chain_pt[side] = take((size_t)L.n_chunks * kChainStride * 8);
    }
    L.chunk = take((size_t)L.n_chunks * 8 * 4);
    L.node = take((size_t)L.n_nodes * 4 * 4);
    L.emit_off[0] = take((size_t)(L.n_chunks + 1) * 4);
    L.emit_off[1] = take((size_t)(L.n_chunks + 1) * 4);
    L.keep_bits = take((size_t)L.filt_tiles * kFiltThreads * 2);
    L.filt_bsum = take((size_t)kFiltMaxBlocks * 4);
    L.kgon = take(sizeof(Kgon));
    L.utmp = take((size_t)n * 4);
    L.spec = take(sizeof(SpecCtrl));
    L.p0 = take(256);
    L.learn = take(sizeof(LearnScratch));
    L.fan2_v = take((size_t)(L.fan2_bins + 4) * 8);
    L.total = o;
    return L;
}

__host__ __device__ inline BatchLayout make_batch_layout(const Layout &L, int64_t sets)
{
    BatchLayout B{};
    B.num_sets = sets;
    B.tiles_max = L.n_chunks;
    size_t o = L.total;
    auto take = [&](size_t bytes) {
        size_t at = o;
        o = align_up(o + bytes, 256);
        return at;
    };
    B.sets = take((size_t)sets * sizeof(SetInfo));
    B.octs = take((size_t)sets * sizeof(Octagon));
    B.zero_begin = o;
    B.bctrl = take(sizeof(BatchCtrl));
    B.ext_slot = take((size_t)sets * 8 * 8);
    B.nonfinite = take((size_t)sets * 4);
    B.hist = take((size_t)sets * kSortPasses * 256 * 4);
    B.soct = take((size_t)sets * 4);
    B.zero_end = o;
    B.tile_set = take((size_t)B.tiles_max * 4);
    B.sc_set = take((size_t)B.tiles_max * 4);
    B.sc_off[0] = take((size_t)(B.tiles_max + 1) * 4);
    B.sc_off[1] = take((size_t)(B.tiles_max + 1) * 4);
    B.lower = L.keys[1];
    // sets with a fan, their tiles (n / kFiltTile and a ragged one each), the
    // others' and the runs of bins
    B.max_fan = sets < L.n / kBxFanMinN ? sets : L.n / kBxFanMinN;
    const int64_t fan_tiles = L.n / kFiltTile + B.max_fan, runs = kBxTileBins / kBxBinRun;
    B.max_items = fan_tiles / kBxFanChunkMin + B.max_fan + 1;
    B.max_plain_items = B.tiles_max / kBxPlainChunk + sets + 1;
    B.max_bin_items = (fan_tiles * runs < B.max_fan * (kFanBins / kBxBinRun) ? fan_tiles * runs
                                                                            : B.max_fan * (kFanBins / kBxBinRun)) + 1;
    B.fan = take((size_t)sets * sizeof(FanInfo));
    B.fan_set = take((size_t)B.max_fan * 4);
    B.fan_tab = L.pay[1];
    B.fan_items = take((size_t)B.max_items * 8);
    B.plain_items = take((size_t)B.max_plain_items * 8);
    B.bin_items = take((size_t)B.max_bin_items * 8);
    B.total = o;
    return B;
}

template <class T>
__host__ __device__ inline T *at(void *ws, size_t off)
{
    return reinterpret_cast<T *>(static_cast<char *>(ws) + off);
}

// ---------------------------------------------------------------------------
// order-preserving keys
// ---------------------------------------------------------------------------
// Map binary32 bits to uint32 so that unsigned order equals numeric order;
// -0 is first mapped to +0 so the two compare equal, as float compares do.
__device__ __forceinline__ uint32_t ord_key(float f)
{
    uint32_t b = __float_as_uint(f);
    if (b == 0x80000000u) b = 0;
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

__device__ __forceinline__ float key_float(uint32_t k)
{
    uint32_t b = (k & 0x80000000u) ? (k & 0x7fffffffu) : ~k;
    return __uint_as_float(b);
}

__device__ __forceinline__ float2 key_point(unsigned long long k)
{
    return make_float2(key_float((uint32_t)(k >> 32)), key_float((uint32_t)k));
}

// a - b = s + e and a + b = s + e exactly (Knuth's two-sum, binary32
// round to nearest; the intrinsics are never contracted into an FMA)
__device__ __forceinline__ void two_diff(float a, float b, float &s, float &e)
{
    s = __fsub_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fsub_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fadd_rn(b, bb));
}
__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e)
{
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// ---------------------------------------------------------------------------
// exact orientation: sign of (b - a) x (c - a) for binary32 inputs
// ---------------------------------------------------------------------------
// Tier 4: the determinant expands into six products of two binary32 values
// (the a.x*a.y terms cancel); each is exact in binary64.  They are summed
// without error by Grow-Expansion with Two-Sum (Shewchuk, "Adaptive
// Precision Floating-Point Arithmetic and Fast Robust Geometric
// Predicates", 1997, Sec. 2); the sign of a non-overlapping expansion is
// the sign of its largest non-zero component.
__device__ __forceinline__ void two_sum(double a, double b, double &s, double &e)
{
    s = __dadd_rn(a, b);
    double bv = __dsub_rn(s, a);
    double av = __dsub_rn(s, bv);
    e = __dadd_rn(__dsub_rn(a, av), __dsub_rn(b, bv));
}

static __device__ __noinline__ int orient_exact(float ax, float ay, float bx, float by, float cx, float cy)
{
    double t[6];
    t[0] = __dmul_rn((double)bx, (double)cy);
    t[1] = -__dmul_rn((double)bx, (double)ay);
    t[2] = -__dmul_rn((double)ax, (double)cy);
    t[3] = -__dmul_rn((double)by, (double)cx);
    t[4] = __dmul_rn((double)by, (double)ax);
    t[5] = __dmul_rn((double)ay, (double)cx);
    double e[6];
    int m = 0;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        double q = t[i];
        int k = 0;
#pragma unroll
        for (int j = 0; j < 6; ++j) {
            if (j < m) {
                double s, r;
                two_sum(q, e[j], s, r);
                q = s;
                if (r != 0.0) e[k++] = r;
            }
        }
        if (q != 0.0) e[k++] = q;
        m = k;
    }
    if (m == 0) return 0;
    return e[m - 1] > 0.0 ? 1 : -1;
}

// Tier 3: binary64 evaluation with Shewchuk's orient2d error bound
// ccwerrboundA = (3 + 16 eps) eps, eps = 2^-53.  Differences and products of
// binary32 values cannot underflow or overflow in binary64, so the bound
// holds; undecided cases go to tier 4.
static __device__ __noinline__ int orient_d(float ax, float ay, float bx, float by, float cx, float cy)
{
    // orient2d(pa = a, pb = b, pc = c)
    double detleft = __dmul_rn(__dsub_rn((double)ax, (double)cx), __dsub_rn((double)by, (double)cy));
    double detright = __dmul_rn(__dsub_rn((double)ay, (double)cy), __dsub_rn((double)bx, (double)cx));
    double det = __dsub_rn(detleft, detright);
    double detsum;
    if (detleft > 0.0) {
        if (detright <= 0.0) return det > 0.0 ? 1 : (det < 0.0 ? -1 : 0);
        detsum = __dadd_rn(detleft, detright);
    } else if (detleft < 0.0) {
        if (detright >= 0.0) return det > 0.0 ? 1 : (det < 0.0 ? -1 : 0);
        detsum = __dsub_rn(-detleft, detright);
    } else {
        return det > 0.0 ? 1 : (det < 0.0 ? -1 : 0);
    }
    const double errA = (3.0 + 16.0 * 0x1p-53) * 0x1p-53;   // exact in binary64
    double eb = __dmul_ru(errA, detsum);
    if (det >= eb) return 1;
    if (-det >= eb) return -1;
    return orient_exact(ax, ay, bx, by, cx, cy);
}

// Tier 1: binary32 evaluation with a dynamic bound.  The expression has
// Shewchuk's orient2d shape (four differences, two products, one
// subtraction), whose rounding error is below (3 + 16 eps) eps * detsum with
// eps = 2^-24 when nothing under- or overflows; 4 eps * detsum leaves room
// for the rounding of the bound itself, and 2^-140 absorbs the absolute
// error of products that fall into the subnormal range.  Undecided cases
// go on to tier 2.
// The binary32 tier alone, branch-free: the sign when the bound proves it,
// 2 otherwise.
__device__ __forceinline__ int orient_f32(float ax, float ay, float bx, float by, float cx, float cy)
{
    float detleft = __fmul_rn(__fsub_rn(ax, cx), __fsub_rn(by, cy));
    float detright = __fmul_rn(__fsub_rn(ay, cy), __fsub_rn(bx, cx));
    float det = __fsub_rn(detleft, detright);
    float detsum = __fadd_rn(fabsf(detleft), fabsf(detright));
    float eb = __fmaf_ru(detsum, 2.384185791015625e-07f /* 2^-22 */, 7.174648137343064e-43f /* 2^-140 */);
    const int o = det > eb ? 1 : (-det > eb ? -1 : 2);
    return detsum <= 3.0e38f ? o : 2;
}

// A product r = fl(a b) whose rounding error fma(a, b, -r) is exact, as it
// cannot underflow (or r is an exact zero).
__device__ __forceinline__ bool exact_product(float a, float b, float r)
{
    return a == 0.0f || b == 0.0f || (fabsf(r) >= 0x1p-100f && fabsf(r) <= 3.0e38f);
}

// Tier 2: the differences as exact pairs (two-diff), the products and their
// rounding errors (FMA), everything of second order added up in binary32: the
// sign when the bound proves it, 2 otherwise.  With eps = 2^-24 the second-
// order terms are below 6 eps detsum in sum, so their ten roundings and the
// omitted product of two low parts cost less than 64 eps^2 detsum = 2^-42
// detsum, and 2^-138 absorbs products in the subnormal range.  Where the four
// differences are exact (points near one another or of a grid) the products
// p + pe, q + qe are too: rounding is monotone, so p > q implies p + pe > q +
// qe, and for p == q the sign is that of pe - qe, which survives its rounding;
// so points that are exactly collinear are settled as well, a third of the
// neighbours' turns where a ring is dense (3 10^7 points, the chain kernel 1020
// us with these left to the next tier, 864 so).  It settles
// nearly every near-collinear triple of a ring's neighbours.  In binary64 (at
// a 64th of the rate here, some 70 cycles an instruction) one such lane held
// its warp for a thousand cycles.
__device__ __forceinline__ int orient_pair(float ax, float ay, float bx, float by, float cx, float cy)
{
    float u, ul, v, vl, w, wl, z, zl;
    two_diff(ax, cx, u, ul);
    two_diff(by, cy, v, vl);
    two_diff(ay, cy, w, wl);
    two_diff(bx, cx, z, zl);
    const float p = __fmul_rn(u, v), q = __fmul_rn(w, z);
    const float pe = __fmaf_rn(u, v, -p), qe = __fmaf_rn(w, z, -q);
    const float pl = __fmaf_rn(u, vl, __fmul_rn(ul, v)), ql = __fmaf_rn(w, zl, __fmul_rn(wl, z));
    float s, sl;
    two_diff(p, q, s, sl);
    const float t = __fadd_rn(__fadd_rn(__fsub_rn(pe, qe), __fsub_rn(pl, ql)), sl);
    const uint32_t low = (__float_as_uint(ul) | __float_as_uint(vl) | __float_as_uint(wl) | __float_as_uint(zl)) << 1;
    if (low == 0u && exact_product(u, v, p) && exact_product(w, z, q)) {
        const float d = p != q ? __fsub_rn(p, q) : __fsub_rn(pe, qe);
        return d > 0.0f ? 1 : (d < 0.0f ? -1 : 0);
    }
    const float det = __fadd_rn(s, t), detsum = __fadd_rn(fabsf(p), fabsf(q));
    const float eb = __fmaf_ru(detsum, 0x1p-42f, 0x1p-138f);
    const int o = det > eb ? 1 : (-det > eb ? -1 : 2);
    return detsum <= 3.0e38f ? o : 2;
}

// Whether a b == c d, proven.
__device__ __forceinline__ bool same_product(float a, float b, float c, float d)
{
    const float r = __fmul_rn(a, b), s = __fmul_rn(c, d);
    return exact_product(a, b, r) && exact_product(c, d, s) && r == s && __fmaf_rn(a, b, -r) == __fmaf_rn(c, d, -s);
}

// The tiers after that: the exactly collinear triples of points on a side of
// the box, of grids and of lines y = 2^k x, then binary64, then expansions
// (whose 200 binary64 steps are some 15000 cycles).
//  - A difference that is zero is exact, so a product with one is zero
//    whatever its other factor (equal points, points on an axis-parallel
//    edge).
//  - The determinant is zero when its expanded products cancel in pairs.
// In binary64 they took most of the time of such sets: 60 sets of 150001
// points on a square's sides 3345 us (1102 so), of a diagonal 4856 (931).
static __device__ __noinline__ int orient_last(float ax, float ay, float bx, float by, float cx, float cy)
{
    if (ax == bx && ay == by) return 0;
    float u, ul, v, vl, w, wl, z, zl;
    two_diff(ax, cx, u, ul);
    two_diff(by, cy, v, vl);
    two_diff(ay, cy, w, wl);
    two_diff(bx, cx, z, zl);
    if ((u == 0.0f || v == 0.0f) && (w == 0.0f || z == 0.0f)) return 0;
    if (same_product(u, v, w, z) && same_product(ul, vl, wl, zl) &&
        ((same_product(u, vl, w, zl) && same_product(ul, v, wl, z)) ||
         (same_product(u, vl, wl, z) && same_product(ul, v, w, zl))))
        return 0;
    return orient_d(ax, ay, bx, by, cx, cy);
}

__device__ __forceinline__ int orient_rest(float ax, float ay, float bx, float by, float cx, float cy)
{
    const int o = orient_pair(ax, ay, bx, by, cx, cy);
    return o != 2 ? o : orient_last(ax, ay, bx, by, cx, cy);
}

__device__ __forceinline__ int orient(float ax, float ay, float bx, float by, float cx, float cy)
{
    const int o = orient_f32(ax, ay, bx, by, cx, cy);
    return o != 2 ? o : orient_rest(ax, ay, bx, by, cx, cy);
}

// ---------------------------------------------------------------------------
// packed binary32 pairs and three-operand minima (sm_100 and later): one
// instruction for two differences or FMAs, each rounded as on its own
// ---------------------------------------------------------------------------
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float a, float b)
{
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c)
{
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    f32x2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pack2(a.x, a.y)), "l"(pack2(b.x, b.y)));
    return unpack2(r);
}
// NaN-propagating minima
__device__ __forceinline__ float min_nan(float a, float b)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ float min_nan(float a, float b, float c)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// ---------------------------------------------------------------------------
// TMA bulk prefetch into L2
// ---------------------------------------------------------------------------
// Asks the TMA unit to bring `bytes` (a multiple of 16, from a 16-byte
// aligned address) into L2.  A hint: nothing waits on it.
__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// The line holding `p` into L2 (one lane's hint; nothing waits on it).
__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// ---------------------------------------------------------------------------
// programmatic dependent launch
// ---------------------------------------------------------------------------
// First statement of every kernel: waits until the kernels before this one
// have completed and their writes are visible.  A kernel launched with
// launch_next (launch.h) is put on the SMs when the blocks of the kernel before
// it have left them, without waiting for its end to be signalled to the front
// end first.  Every thread passes here, before any return, so a kernel's
// completion implies that of all kernels before it.  A call's pipeline holds
// up to a dozen kernels that find nothing to do for a given set, each 2.8 us
// when launched the ordinary way: ch_hull of 1000 points 62 -> 42 us, of 2^20
// normal points 105 -> 68, of 10^8 circle points 970 -> 928.  No kernel lets the
// next one in earlier (launch_dependents): its blocks would then fill the
// first SMs to become free, and grids of fewer blocks than the chip holds
// would run on half of it (circle 1057, 2^20 normal points 75).
__device__ __forceinline__ void kernel_entry()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------------------
// error reporting and bounded waits
// ---------------------------------------------------------------------------
__device__ __forceinline__ void set_error(void *ws, const Layout &L, uint32_t code, uint32_t site)
{
    Persist *p = at<Persist>(ws, L.persist);
    if (atomicCAS(&p->error, 0u, code) == 0u) atomicExch(&p->error_site, site);
}

__device__ __forceinline__ bool error_set(void *ws, const Layout &L)
{
    return *(volatile uint32_t *)&at<Persist>(ws, L.persist)->error != 0u;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u64(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint32_t ld_relaxed_u32(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_u32(uint32_t *p, uint32_t v)
{
    asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Decoupled look-back (Merrill & Garland, "Single-pass Parallel Prefix Scan
// with Decoupled Look-back", 2016) over 64-bit status words, run by one
// full warp.  Returns the exclusive prefix of tile `tile`.  Waits are
// bounded: when a predecessor never publishes, the error word is set and
// the wait stops (the prefix is then meaningless, the call reports
// CH_ERR_TIMEOUT).
__device__ __forceinline__ unsigned long long lookback_u64(unsigned long long *status, int64_t tile,
                                                           void *ws, const Layout &L, uint32_t site)
{
    const uint32_t lane = lane_id();
    unsigned long long excl = 0;
    int64_t base = tile - 1;
    uint32_t spins = 0;
    while (base >= 0) {
        int64_t idx = base - (int64_t)lane;
        unsigned long long s = idx >= 0 ? ld_acquire_u64(status + idx) : kFlagP;
        while (__any_sync(0xffffffffu, (s >> 62) == 0)) {
            if (++spins > kSpinLimit || (spins > 1024 && error_set(ws, L))) {
                if (lane == 0) set_error(ws, L, kErrTimeout, site);
                return 0;
            }
            if (spins > 64) __nanosleep(100);
            if ((s >> 62) == 0) s = ld_acquire_u64(status + idx);
        }
        uint32_t pmask = __ballot_sync(0xffffffffu, (s >> 62) == 2);
        uint32_t stop = pmask ? (uint32_t)(__ffs(pmask) - 1) : 31u;
        unsigned long long v = lane <= stop ? (s & kValMask) : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        excl += v;
        if (pmask) break;
        base -= 32;
    }
    return excl;
}

}  // namespace ch
