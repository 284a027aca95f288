// filter.cu -- Sec. 3.2 of Carrasco et al.: buildingFilter (is a point
// strictly inside the eight-vertex polygon?) and compactingFilteredPoints
// (stable compaction of the kept points).
//
// The paper writes an n-entry flag vector, scans it (tensor-core segmented
// scan, Thrust or CUB) and scatters.  Flags never reach memory here; two
// variants are built:
//
//  * two-pass (default): a streaming count pass tests 4096-point tiles and
//    writes keep bits and one survivor count per tile, each block over a
//    contiguous range of tiles, plus the block's total; a scatter pass with
//    the same grid finds each tile's output offset from the block totals
//    and an in-block scan of its range, visits only the tiles that have
//    survivors, loads only the kept points and writes them in ascending
//    index order.  No block waits on another, so both passes stream at
//    memory speed; when almost everything is discarded (normal data) the
//    points are read once, when nothing is (circle) they are read twice.
//  * single-pass: one persistent kernel takes tiles in ticket order, tests
//    them, publishes the tile count, gets its offset by decoupled look-back
//    and writes its survivors; points are read once, but each tile waits on
//    its predecessors.
//
// The test: the quick-discard rectangle, then all edges at once by affine
// forms with a proven error (octtest.cuh), exact signs for the few points
// they leave undecided.
//
// ch_hull runs neither pass (kgon.cu tests and writes the survivors of the
// octagon and of its fan in one), unless a second polygon reads the count
// pass's keep bits in between.
//
// Memory traffic: 8 bytes per point read (twice for tiles with survivors in
// the two-pass variant), 12 bytes per kept point written.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "launch.h"
#include "octtest.cuh"

namespace ch {

namespace {

constexpr int NW = kFiltThreads / 32;

// Copies the polygon to shared memory; false when the call was aborted
// (non-finite input or a bad vertex index).
__device__ __forceinline__ bool load_octagon(OctSmem &so, void *ws, const Layout &L)
{
    fill_octagon(so, at<Octagon>(ws, L.oct));
    __syncthreads();
    return !so.abort;
}

// Of eight points (live: bits of those that exist), the ones to keep; those
// the affine forms left undecided are among them, and the result says
// whether there may be any.  The quick-discard rectangle comes first: it
// holds nearly every point of a normal cloud, and a warp whose points are
// all in it is done.
template <bool BOX>
__device__ __forceinline__ bool test8(const OctSmem &so, const float (&px)[8], const float (&py)[8], uint32_t live,
                                      uint32_t &keep)
{
    const float xl = so.xl, xh = so.xh, yl = so.yl, yh = so.yh;
    uint32_t rect = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
        if ((px[q] >= xl) & (px[q] <= xh) & (py[q] >= yl) & (py[q] <= yh)) rect |= 1u << q;
    keep = live & ~rect;
    if (!__any_sync(0xffffffffu, keep != 0u) || !so.has_edges) return false;
    uint32_t outside = 0;
    if constexpr (BOX) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (outside_box<true>(so, px[q], py[q])) outside |= 1u << q;
    }
    uint32_t k8;
    const bool near = oct_decide<8>(so, px, py, k8);
    keep &= k8 | outside;
    return near;
}

// Exact decisions for the kept ones (load(q) reads point q), some of which
// the affine forms left undecided.
template <bool BOX, class Load>
__device__ __forceinline__ uint32_t settle_near(const OctSmem &so, uint32_t keep, Load load)
{
#pragma unroll 1
    for (uint32_t m = keep; m; m &= m - 1u) {
        const float2 p = load(__ffs(m) - 1);
        if (!keep_point<BOX>(so, p.x, p.y)) keep &= ~(m & (0u - m));
    }
    return keep;
}

// Loads and tests one tile, eight of the thread's 16 points at a time (all
// 16 at once would spill).  Returns the keep bits; positions past n are not
// kept.
template <int G, bool BOX>
__device__ __forceinline__ uint32_t load_test(const float *__restrict__ pts, int64_t n, int64_t base, const OctSmem &so)
{
    const uint32_t tid = threadIdx.x;
    uint32_t keep = 0;
    bool near = false;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
        float px[8], py[8];
        uint32_t live = 0xffu, k8;
        if (base + kFiltTile <= n) load_part<G, 8>(pts, base, tid, half, px, py);
        else live = load_part_ragged<G, 8>(pts, n, base, tid, half, so.cx, so.cy, px, py);
        near |= test8<BOX>(so, px, py, live, k8);
        keep |= k8 << (8 * half);
    }
    return near ? settle_near<BOX>(so, keep, [&](int q) { return input_point(pts, item_point<G>(base, tid, q)); }) : keep;
}

// The block writes the kept points of one tile in point order from the
// threads' keep bits (out_off: the tile's first output position): a row is
// one load of every thread, kFiltThreads * G consecutive points.  The loads
// are under way while the warps count their rows; every warp then scans all
// (row, warp) counts itself, so there is one barrier a tile, and s_cnt
// alternates between two arrays.
// Bound by latency and the writes.  (A warp per tile left three of eight
// warps idle on a block's five tiles: 10^7 displaced points, 9.4 M of them
// written, 62 us; this 45.)
template <int G, bool KEYS>
__device__ __forceinline__ void scatter_tile(const float *__restrict__ pts, int64_t n, uint32_t kb, int64_t base,
                                             uint32_t out_off, uint32_t (&s_cnt)[kFiltItems / G][NW],
                                             uint32_t *surv_idx, float2 *surv_pts, uint32_t *out_keys,
                                             unsigned long long *out_pay)
{
    constexpr int ROWS = kFiltItems / G;
    constexpr uint32_t RM = (1u << G) - 1u;   // a row's bits among a thread's 16
    constexpr int PER = ROWS * NW / 32;
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id(), lt = (1u << lane) - 1u;
    float px[kFiltItems], py[kFiltItems];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const int64_t i = item_point<G>(base, tid, r * G);
        if constexpr (G == 2) {
            float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if ((kb >> (2 * r)) & 3u) {
                if (i + 1 < n) {
                    v = __ldcs(reinterpret_cast<const float4 *>(pts) + i / 2);
                } else {
                    const float2 a = reinterpret_cast<const float2 *>(pts)[i];
                    v = make_float4(a.x, a.y, 0.0f, 0.0f);
                }
            }
            px[2 * r] = v.x;
            py[2 * r] = v.y;
            px[2 * r + 1] = v.z;
            py[2 * r + 1] = v.w;
        } else {
            float2 v = make_float2(0.0f, 0.0f);
            if ((kb >> r) & 1u) v = __ldcs(reinterpret_cast<const float2 *>(pts) + i);
            px[r] = v.x;
            py[r] = v.y;
        }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(kb & (RM << (r * G))));
        if (lane == 0) s_cnt[r][warp] = c;
    }
    __syncthreads();
    // lane l holds the counts l * PER .. of the rows' warps, row-major: the point order
    const uint32_t *flat = &s_cnt[0][0];
    uint32_t loc[PER], sum = 0;
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        loc[k] = sum;
        sum += flat[lane * PER + k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl += u;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) loc[k] += out_off + incl - sum;
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
        const uint32_t e = (uint32_t)r * NW + warp;   // this warp's place among the counts
        uint32_t pos = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            const uint32_t v = __shfl_sync(0xffffffffu, loc[k], e / PER);
            if (e % PER == (uint32_t)k) pos = v;
        }
#pragma unroll
        for (int h = 0; h < G; ++h) pos += __popc(__ballot_sync(0xffffffffu, (kb >> (r * G + h)) & 1u) & lt);
#pragma unroll
        for (int h = 0; h < G; ++h) {
            const int q = r * G + h;
            if (!((kb >> q) & 1u)) continue;
            const uint32_t idx = (uint32_t)item_point<G>(base, tid, q);
            if constexpr (KEYS) {
                out_keys[pos] = ord_key(px[q]);
                out_pay[pos] = ((unsigned long long)ord_key(py[q]) << 32) | idx;
            } else {
                surv_idx[pos] = idx;
                if (surv_pts) surv_pts[pos] = make_float2(px[q], py[q]);
            }
            ++pos;
        }
    }
}

__device__ __forceinline__ void write_count(bool keys, Ctrl *ctrl, uint32_t *surv_count, uint32_t v)
{
    if (keys) ctrl->surv_count = v;
    else *surv_count = v;
}

// ---------------------------------------------------------------------------
// single pass: ticket-ordered tiles with decoupled look-back
// ---------------------------------------------------------------------------
template <int G, bool KEYS, bool BOX>
__global__ void __launch_bounds__(kFiltThreads) filter_kernel(const float *__restrict__ pts, int64_t n,
                                                              void *ws, Layout L, uint32_t *__restrict__ surv_idx,
                                                              float2 *__restrict__ surv_pts,
                                                              uint32_t *__restrict__ surv_count)
{
    kernel_entry();
    __shared__ OctSmem so;
    __shared__ uint32_t s_row[kFiltItems / G][NW];
    __shared__ uint32_t s_w[NW];
    __shared__ uint32_t s_tile;
    __shared__ unsigned long long s_excl;
    __shared__ uint32_t s_total;

    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    unsigned long long *status = at<unsigned long long>(ws, L.filt_status);
    if (!load_octagon(so, ws, L)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) write_count(KEYS, ctrl, surv_count, 0);
        return;
    }
    const int64_t ntiles = ceil_div(n, kFiltTile);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(&ctrl->filt_ticket, 1u);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= ntiles) break;
        const int64_t base = tile * kFiltTile;
        const uint32_t keep = load_test<G, BOX>(pts, n, base, so);
        const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(keep));
        if (lane == 0) s_w[warp] = c;
        __syncthreads();
        if (warp == 0) {
            const uint32_t total = __reduce_add_sync(0xffffffffu, lane < (uint32_t)NW ? s_w[lane] : 0u);
            unsigned long long excl = 0;
            if (tile == 0) {
                if (lane == 0) st_release_u64(status, kFlagP | total);
            } else {
                if (lane == 0) st_release_u64(status + tile, kFlagA | total);
                excl = lookback_u64(status, tile, ws, L, 10);
                if (lane == 0) st_release_u64(status + tile, kFlagP | ((excl + total) & kValMask));
            }
            if (lane == 0) {
                s_excl = excl;
                s_total = total;
                if (tile == ntiles - 1) write_count(KEYS, ctrl, surv_count, (uint32_t)(excl + total));
            }
        }
        __syncthreads();
        if (s_total != 0)
            scatter_tile<G, KEYS>(pts, n, keep, base, (uint32_t)s_excl, s_row, surv_idx, surv_pts,
                                  at<uint32_t>(ws, L.keys[0]), at<unsigned long long>(ws, L.pay[0]));
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// the speculative sweep's candidates (extremes.cu): when the sweep proved
// every other point strictly inside the octagon (Octagon::spec), the count
// and scatter passes test and write only the candidates.  Segment j holds
// (unordered) the candidates of the j-th sweep block's contiguous index
// range, so segments in order, each sorted by index, give the survivors in
// ascending index order.
// ---------------------------------------------------------------------------
// Count pass: the exact test of every candidate; the slots of a segment's
// survivors go to utmp (unordered), their number to skept, and each count
// block's total to the block totals the fan reads.
__device__ void spec_count(const Octagon &so, void *ws, const Layout &L)
{
    SpecCtrl *sc = at<SpecCtrl>(ws, L.spec);
    const float2 *cpt = at<float2>(ws, L.pay[1]);
    uint32_t *kept_slot = at<uint32_t>(ws, L.utmp);
    __shared__ uint32_t s_k;
    __shared__ uint32_t s_pre[kSpecWarps + 1];   // candidates before each slice of the segment
    const uint32_t nseg = sc->nseg, cap = sc->cap;
    uint32_t block_total = 0;
    for (uint32_t j = blockIdx.x; j < nseg; j += gridDim.x) {
        const size_t seg0 = (size_t)j * kSpecWarps * cap;
        __syncthreads();   // s_k and s_pre of the previous segment have been read
        if (threadIdx.x < 32) {
            const uint32_t c = threadIdx.x < (uint32_t)kSpecWarps ? min(sc->scnt[j * kSpecWarps + threadIdx.x], cap) : 0u;
            uint32_t incl = c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (threadIdx.x >= (uint32_t)o) incl += t;
            }
            if (threadIdx.x < (uint32_t)kSpecWarps) s_pre[threadIdx.x + 1] = incl;
            if (threadIdx.x == 0) {
                s_pre[0] = 0u;
                s_k = 0u;
            }
        }
        __syncthreads();
        // the segment's candidates in one sweep: e-th candidate = candidate
        // e - s_pre[w] of the slice of warp w, at slot w * cap + that
        const uint32_t total = s_pre[kSpecWarps];
        for (uint32_t e = threadIdx.x; e < total; e += blockDim.x) {
            uint32_t w = 0;
            while (s_pre[w + 1] <= e) ++w;
            const uint32_t slot = w * cap + (e - s_pre[w]);
            const float2 p = cpt[seg0 + slot];
            if (keep_point<false>(so, p.x, p.y)) kept_slot[seg0 + atomicAdd(&s_k, 1u)] = slot;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            sc->skept[j] = s_k;
            block_total += s_k;
        }
    }
    if (threadIdx.x == 0) at<uint32_t>(ws, L.filt_bsum)[blockIdx.x] = block_total;
}

struct SpecScatterSmem {
    uint32_t idx[kSpecKeptSmem];   // indices of a segment's survivors
    uint32_t red[NW];
};

// Scatter pass: each segment's survivors, ranked by index, at the segment's
// offset (the survivors of the segments before it); block 0 writes the
// count.  A segment with more survivors than shared memory holds is ranked
// from global memory (slower, same result).
__device__ void spec_scatter(SpecScatterSmem &sm, void *ws, const Layout &L, uint32_t *surv_idx, float2 *surv_pts,
                             uint32_t *surv_count)
{
    const SpecCtrl *sc = at<SpecCtrl>(ws, L.spec);
    const uint32_t *cidx = at<uint32_t>(ws, L.keys[1]);
    const float2 *cpt = at<float2>(ws, L.pay[1]);
    const uint32_t *kept_slot = at<uint32_t>(ws, L.utmp);
    const uint32_t nseg = sc->nseg, cap = sc->cap, tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    if (blockIdx.x == 0) {
        uint32_t t = 0;
        for (uint32_t i = tid; i < nseg; i += blockDim.x) t += sc->skept[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) sm.red[warp] = t;
        __syncthreads();
        if (tid == 0) {
            uint32_t total = 0;
#pragma unroll
            for (int w = 0; w < NW; ++w) total += sm.red[w];
            *surv_count = total;
        }
    }
    for (uint32_t j = blockIdx.x; j < nseg; j += gridDim.x) {
        const uint32_t k = sc->skept[j];   // block-uniform
        if (k == 0u) continue;
        // offset: survivors of the segments before j
        uint32_t before = 0;
        for (uint32_t i = tid; i < j; i += blockDim.x) before += sc->skept[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
        __syncthreads();   // sm of the previous segment has been read
        if (lane == 0) sm.red[warp] = before;
        const size_t seg0 = (size_t)j * kSpecWarps * cap;
        const bool in_smem = k <= (uint32_t)kSpecKeptSmem;
        if (in_smem)
            for (uint32_t e = tid; e < k; e += blockDim.x) sm.idx[e] = cidx[seg0 + kept_slot[seg0 + e]];
        __syncthreads();
        uint32_t off = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) off += sm.red[w];
        for (uint32_t e = tid; e < k; e += blockDim.x) {
            const uint32_t slot = kept_slot[seg0 + e];
            const uint32_t mine = cidx[seg0 + slot];
            uint32_t r = 0;
            if (in_smem)
                for (uint32_t q = 0; q < k; ++q) r += sm.idx[q] < mine ? 1u : 0u;
            else
                for (uint32_t q = 0; q < k; ++q) r += cidx[seg0 + kept_slot[seg0 + q]] < mine ? 1u : 0u;
            const float2 p = cpt[seg0 + slot];
            const size_t pos = (size_t)off + r;
            surv_idx[pos] = mine;
            if (surv_pts) surv_pts[pos] = p;
        }
    }
}

// ---------------------------------------------------------------------------
// two passes: count -> scan -> scatter
// ---------------------------------------------------------------------------
// filt_status[t] receives the survivor count of tile t (low 32 bits); the
// scan turns it into (offset << 32 | count).  Each thread's 16 keep bits go
// to keep_bits, so the scatter pass does not test again.
// Per-tile survivor counts of a window of kCountRing tiles, added up in
// shared memory by the warps as they finish each tile, written to
// filt_status when the window is done.  Schedule, chosen by each block
// from its first tile: where it keeps under a quarter of its points (the
// rectangle settles most of them: bound by memory) the warps meet at a
// barrier after every tile, so that they read each tile together (a warp's
// share is 512 B of every 4 KB row; warps spread over tiles lose DRAM row
// locality: 0.66 against 0.89 of the copy peak on 10^9 normal points);
// elsewhere (every point takes the edge test: bound by issue) they run
// free and one warp's deferred points do not hold the others.
constexpr int kCountRing = 256;

// Block-wide sum to thread 0 (s_w: one slot per warp).
__device__ __forceinline__ uint32_t block_sum_to0(uint32_t v, uint32_t (&s_w)[NW])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane_id() == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    uint32_t t = 0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < NW; ++w) t += s_w[w];
    }
    return t;
}

// kdev (ch_hull_learned, else NULL): the device's choice of K; 8 means that
// no second polygon will read the keep bits, and the pass is not needed.
template <int G, bool BOX>
__global__ void __launch_bounds__(kFiltThreads, 4) filter_count_kernel(const float *__restrict__ pts, int64_t n,
                                                                    void *ws, Layout L,
                                                                    const int32_t *kdev)
{
    kernel_entry();
    __shared__ OctSmem so;
    __shared__ uint32_t s_cnt[kCountRing];
    __shared__ uint32_t s_w[NW];
    for (int i = threadIdx.x; i < kCountRing; i += kFiltThreads) s_cnt[i] = 0u;
    if (kdev && *kdev == 8) return;
    if (!load_octagon(so, ws, L)) return;   // (its barrier also covers s_cnt)
    if constexpr (!BOX) {
        if (so.spec) {   // the speculative sweep proved all but its candidates inside
            spec_count(so, ws, L);
            return;
        }
    }
    unsigned long long *status = at<unsigned long long>(ws, L.filt_status);
    uint16_t *bits = at<uint16_t>(ws, L.keep_bits);
    const int64_t ntiles = ceil_div(n, kFiltTile);
    const uint32_t lane = lane_id();
    // a contiguous range of tiles per block, so the scatter pass finds
    // every tile's output offset from the block totals and its own range
    const int64_t t0 = first_tile(ntiles, gridDim.x, blockIdx.x), t1 = first_tile(ntiles, gridDim.x, blockIdx.x + 1);
    uint32_t part = 0;   // this thread's share of the block total
    bool first = true, lockstep = true;
    for (int64_t w0 = t0; w0 < t1; w0 += kCountRing) {
        const int64_t w1 = min(t1, w0 + kCountRing);
        for (int64_t tile = w0; tile < w1; ++tile) {
            if (threadIdx.x == 0 && tile + 1 < t1) {   // the next tile streams into L2 meanwhile
                const int64_t nb = (tile + 1) * kFiltTile;
                const uint32_t nn = (uint32_t)std::min<int64_t>(kFiltTile, n - nb);
                if (((reinterpret_cast<uintptr_t>(pts + 2 * nb)) & 15u) == 0)
                    bulk_prefetch_l2(pts + 2 * nb, (nn * 8u) & ~15u);
            }
            const uint32_t keep = load_test<G, BOX>(pts, n, tile * kFiltTile, so);
            bits[tile * kFiltThreads + threadIdx.x] = (uint16_t)keep;
            uint32_t c = __popc(keep);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
            if (lane == 0 && c) atomicAdd(&s_cnt[tile - w0], c);
            if (first) {   // the block's first tile decides (block-uniform: read after the barrier)
                __syncthreads();
                lockstep = s_cnt[tile - w0] < (uint32_t)(kFiltTile / 4);
                first = false;
            } else if (lockstep) {
                __syncthreads();
            }
        }
        __syncthreads();   // every warp's counts of the window are in
        for (int64_t i = threadIdx.x; i < w1 - w0; i += kFiltThreads) {
            const uint32_t v = s_cnt[i];
            status[w0 + i] = v;
            s_cnt[i] = 0u;
            part += v;
        }
        __syncthreads();
    }
    const uint32_t total = block_sum_to0(part, s_w);
    if (threadIdx.x == 0) at<uint32_t>(ws, L.filt_bsum)[blockIdx.x] = total;
}

// Second pass, launched with the count pass's grid: block b owns the same
// tile range.  Its output offset is the sum of the earlier blocks' totals;
// an in-block scan of its tiles' counts gives each tile's offset, and only
// tiles with survivors are visited.  Block 0 writes the survivor count.
template <int G, bool KEYS>
__global__ void __launch_bounds__(kFiltThreads, 3) filter_scatter_kernel(const float *__restrict__ pts, int64_t n,
                                                                      void *ws, Layout L,
                                                                      uint32_t *__restrict__ surv_idx,
                                                                      float2 *__restrict__ surv_pts,
                                                                      uint32_t *surv_count, int allow_spec)
{
    kernel_entry();
    __shared__ uint32_t s_abort;
    __shared__ uint32_t s_red[2][NW];
    __shared__ uint32_t s_list[kFiltThreads];    // non-empty tiles of a chunk: offset in chunk
    __shared__ uint32_t s_loff[kFiltThreads];    // and their output offsets
    __shared__ uint32_t s_nlist;
    __shared__ uint32_t s_row[2][kFiltItems / G][NW];
    __shared__ uint32_t s_spec;
    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    if (threadIdx.x == 0) {
        const Octagon *oct = at<Octagon>(ws, L.oct);
        s_abort = oct->abort;
        s_spec = allow_spec ? oct->spec : 0u;   // a polygon the octagon record does not describe: never
    }
    __syncthreads();
    if (s_abort) {
        if (blockIdx.x == 0 && threadIdx.x == 0) write_count(KEYS, ctrl, surv_count, 0);
        return;
    }
    if constexpr (!KEYS) {   // (the hull step takes the candidates itself)
        __shared__ SpecScatterSmem s_sp;
        if (s_spec) {   // only the speculative sweep's candidates can survive
            spec_scatter(s_sp, ws, L, surv_idx, surv_pts, surv_count);
            return;
        }
    }
    const unsigned long long *status = at<unsigned long long>(ws, L.filt_status);
    const uint32_t *bsum = at<uint32_t>(ws, L.filt_bsum);
    const uint16_t *bits = at<uint16_t>(ws, L.keep_bits);
    uint32_t *out_keys = at<uint32_t>(ws, L.keys[0]);
    unsigned long long *out_pay = at<unsigned long long>(ws, L.pay[0]);
    const int64_t ntiles = ceil_div(n, kFiltTile);
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    // offset of this block's range, and the total
    uint32_t before = 0, total = 0;
    for (uint32_t i = tid; i < gridDim.x; i += kFiltThreads) {
        const uint32_t v = bsum[i];
        total += v;
        if (i < blockIdx.x) before += v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        before += __shfl_xor_sync(0xffffffffu, before, o);
        total += __shfl_xor_sync(0xffffffffu, total, o);
    }
    if (lane == 0) {
        s_red[0][warp] = before;
        s_red[1][warp] = total;
    }
    __syncthreads();
    before = total = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        before += s_red[0][w];
        total += s_red[1][w];
    }
    if (blockIdx.x == 0 && tid == 0) write_count(KEYS, ctrl, surv_count, total);
    __syncthreads();   // s_red is reused below
    const int64_t r0 = first_tile(ntiles, gridDim.x, blockIdx.x), r1 = first_tile(ntiles, gridDim.x, blockIdx.x + 1);
    uint32_t run = before;
    for (int64_t c0 = r0; c0 < r1; c0 += kFiltThreads) {
        // this chunk's tile counts: exclusive scan and the non-empty ones
        const int64_t t = c0 + tid;
        const uint32_t cnt = t < r1 ? (uint32_t)(status[t] & 0xffffffffull) : 0u;
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += u;
        }
        const uint32_t nz = __ballot_sync(0xffffffffu, cnt != 0u);
        if (lane == 31) {
            s_red[0][warp] = incl;
            s_red[1][warp] = __popc(nz);
        }
        __syncthreads();
        uint32_t wbefore = 0, chunk_total = 0, lbefore = 0, nlist = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w < (int)warp) {
                wbefore += s_red[0][w];
                lbefore += s_red[1][w];
            }
            chunk_total += s_red[0][w];
            nlist += s_red[1][w];
        }
        if (cnt != 0u) {
            const uint32_t slot = lbefore + __popc(nz & ((1u << lane) - 1u));
            s_list[slot] = tid;
            s_loff[slot] = run + wbefore + incl - cnt;
        }
        if (tid == 0) s_nlist = nlist;
        __syncthreads();
        const uint32_t nl = s_nlist;
        uint32_t kb = nl ? bits[(c0 + s_list[0]) * kFiltThreads + tid] : 0u;
        for (uint32_t li = 0; li < nl; ++li) {
            const uint32_t mine = kb;
            if (li + 1 < nl) kb = bits[(c0 + s_list[li + 1]) * kFiltThreads + tid];
            scatter_tile<G, KEYS>(pts, n, mine, (c0 + s_list[li]) * kFiltTile, s_loff[li], s_row[li & 1u], surv_idx,
                                  surv_pts, out_keys, out_pay);
        }
        __syncthreads();   // s_list, s_loff, s_row and s_red are written again for the next chunk
        run += chunk_total;
    }
}

template <class K>
int occupancy(K kernel, int threads)
{
    int v = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, kernel, threads, 0);
    return v > 0 ? v : 1;
}

template <int G, bool KEYS>
cudaError_t launch_single(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *surv_idx,
                          float *surv_pts, uint32_t *surv_count, cudaStream_t st)
{
    // the hull step (KEYS) filters with the data's own extremes; ch_filter's
    // caller-supplied vertices need the bounding-box check
    static int per_sm = occupancy(filter_kernel<G, KEYS, !KEYS>, kFiltThreads);
    const int64_t ntiles = ceil_div(n, kFiltTile);
    int64_t blocks = std::min<int64_t>((int64_t)sm_count() * per_sm, ntiles);
    launch_next(filter_kernel<G, KEYS, !KEYS>, (unsigned)std::max<int64_t>(blocks, 1), kFiltThreads, 0, st, pts, n,
                ws, L, surv_idx, reinterpret_cast<float2 *>(surv_pts), surv_count);
    note_kernels(CH_K_FILTER, 1);
    return cudaGetLastError();
}

template <int G, bool BOX>
int64_t count_blocks(int64_t n)
{
    static const int per_sm = occupancy(filter_count_kernel<G, BOX>, kFiltThreads);
    return std::max<int64_t>(1, std::min<int64_t>(std::min<int64_t>((int64_t)sm_count() * per_sm, kFiltMaxBlocks),
                                                  ceil_div(n, kFiltTile)));
}

// BOX: the polygon's vertices were supplied by the caller (ch_filter), so
// points outside their box must be kept first; otherwise they are the
// data's extremes, and the scatter may take the speculative sweep's
// candidates (Octagon::spec)
template <int G, bool BOX>
cudaError_t launch_two_pass(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *surv_idx,
                            float *surv_pts, uint32_t *surv_count, cudaStream_t st)
{
    // both passes use the same grid (block b owns the same tile range),
    // the count pass's resident blocks
    const int64_t bc = count_blocks<G, BOX>(n);
    launch_next(filter_count_kernel<G, BOX>, (unsigned)bc, kFiltThreads, 0, st, pts, n, ws, L, nullptr);
    launch_next(filter_scatter_kernel<G, false>, (unsigned)bc, kFiltThreads, 0, st, pts, n, ws, L, surv_idx,
                reinterpret_cast<float2 *>(surv_pts), surv_count, BOX ? 0 : 1);
    note_kernels(CH_K_FILTER, 2);
    return cudaGetLastError();
}

// 0: two passes, 1: single pass with look-back; process-wide, read once per
// call when its kernels are enqueued (an atomic, so setting it from another
// host thread is not a data race)
std::atomic<int> g_filter_variant{0};

template <int G>
cudaError_t launch_variant(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *surv_idx,
                           float *surv_pts, uint32_t *surv_count, cudaStream_t st, int variant, bool data_extremes)
{
    if (variant == 1) return launch_single<G, false>(pts, n, ws, L, surv_idx, surv_pts, surv_count, st);
    if (data_extremes) return launch_two_pass<G, false>(pts, n, ws, L, surv_idx, surv_pts, surv_count, st);
    return launch_two_pass<G, true>(pts, n, ws, L, surv_idx, surv_pts, surv_count, st);
}

}  // namespace

int filter_variant() { return g_filter_variant.load(std::memory_order_relaxed); }

cudaError_t launch_filter(const float *pts, int64_t n, void *ws, const Layout &L, uint32_t *surv_idx,
                          float *surv_pts, uint32_t *surv_count, cudaStream_t st, int variant, bool data_extremes)
{
    const int v = variant < 0 ? g_filter_variant.load(std::memory_order_relaxed) : variant;
    const bool vec = (reinterpret_cast<uintptr_t>(pts) & 15u) == 0;
    probe_before(CH_K_FILTER, st);
    const cudaError_t e = vec ? launch_variant<2>(pts, n, ws, L, surv_idx, surv_pts, surv_count, st, v, data_extremes)
                              : launch_variant<1>(pts, n, ws, L, surv_idx, surv_pts, surv_count, st, v, data_extremes);
    probe_after(CH_K_FILTER, st);
    return e;
}

cudaError_t launch_filter_keys_single(const float *pts, int64_t n, void *ws, const Layout &L, cudaStream_t st)
{
    const bool vec = (reinterpret_cast<uintptr_t>(pts) & 15u) == 0;
    probe_before(CH_K_FILTER, st);
    const cudaError_t e = vec ? launch_single<2, true>(pts, n, ws, L, nullptr, nullptr, nullptr, st)
                              : launch_single<1, true>(pts, n, ws, L, nullptr, nullptr, nullptr, st);
    probe_after(CH_K_FILTER, st);
    return e;
}

cudaError_t launch_filter_count(const float *pts, int64_t n, const int32_t *kdev, void *ws, const Layout &L,
                                cudaStream_t st)
{
    const bool vec = (reinterpret_cast<uintptr_t>(pts) & 15u) == 0;
    const int64_t bc = vec ? count_blocks<2, false>(n) : count_blocks<1, false>(n);
    probe_before(CH_K_FILTER, st);
    if (vec) launch_next(filter_count_kernel<2, false>, (unsigned)bc, kFiltThreads, 0, st, pts, n, ws, L, kdev);
    else launch_next(filter_count_kernel<1, false>, (unsigned)bc, kFiltThreads, 0, st, pts, n, ws, L, kdev);
    note_kernels(CH_K_FILTER, 1);
    probe_after(CH_K_FILTER, st);
    return cudaGetLastError();
}

cudaError_t launch_filter_scatter(const float *pts, int64_t n, int64_t grid, void *ws, const Layout &L,
                                  uint32_t *surv_idx, float *surv_pts, uint32_t *surv_count, bool keys_mode,
                                  cudaStream_t st)
{
    const bool vec = (reinterpret_cast<uintptr_t>(pts) & 15u) == 0;
    float2 *sp = reinterpret_cast<float2 *>(surv_pts);
    const unsigned g = (unsigned)std::max<int64_t>(1, grid);
    if (keys_mode) {
        if (vec) launch_next(filter_scatter_kernel<2, true>, g, kFiltThreads, 0, st, pts, n, ws, L, nullptr, nullptr, nullptr, 0);
        else launch_next(filter_scatter_kernel<1, true>, g, kFiltThreads, 0, st, pts, n, ws, L, nullptr, nullptr, nullptr, 0);
    } else {
        if (vec) launch_next(filter_scatter_kernel<2, false>, g, kFiltThreads, 0, st, pts, n, ws, L, surv_idx, sp, surv_count, 0);
        else launch_next(filter_scatter_kernel<1, false>, g, kFiltThreads, 0, st, pts, n, ws, L, surv_idx, sp, surv_count, 0);
    }
    note_kernels(CH_K_FILTER, 1);
    return cudaGetLastError();
}

}  // namespace ch

extern "C" ch_status ch_filter_variant(int32_t variant)
{
    if (variant != 0 && variant != 1) return CH_ERR_ARG;
    ch::g_filter_variant.store(variant, std::memory_order_relaxed);
    return CH_OK;
}
