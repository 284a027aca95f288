// chain.cu -- Sec. 3.3 of Carrasco et al. (convexHull_algorithm), kept on
// the device: Andrew's monotone chain over the survivors sorted by x.
//
// The paper copies the candidates to the host and calls CGAL; its
// conclusion names a fully device-resident hull as the next step.  Here:
//
//  0. runs: the survivors arrive sorted by x (equal x in any order), or are
//     so few that the block sorts them itself.  In a run of equal x only the
//     lowest point can be a vertex of the lower chain and only the highest
//     one of the upper chain, because the others lie strictly above (below)
//     it on the same vertical.  The exceptions are the first x, whose lowest
//     point starts both chains and whose highest point follows it on the
//     upper chain, and the last x, whose highest point ends both chains after
//     its lowest point on the lower chain.  Each run is reduced to those
//     representatives (on ties the lowest index, which also collapses equal
//     points).  A block owns the runs starting in its 4096-point
//     super-chunk and looks ahead (block-parallel) when its last run
//     continues past the super-chunk.
//  1. elimination: of the points between a side's two ends only those
//     strictly beyond the segment joining the ends stay, and then parallel
//     passes drop every point whose turn with its current neighbours is not
//     strict (for the lower chain: on or above the segment joining them).
//     Such a point lies on or above a segment between two points of the set,
//     so it is not a strict vertex of the lower hull and the sequential
//     chain would pop it too; a sequence where every turn is strict is its
//     own monotone chain.  Half of the block's warps take each side: a pass
//     over the whole sequence, passes inside each warp's share, and again
//     until a whole pass drops nothing.  The sequence is written out as the
//     super-chunk's chain.
//  2. fallback, when the passes do not converge within their cap: what is
//     left is cut into leaves; one thread runs the sequential monotone
//     chain on each, and the leaf chains are merged pairwise up a binary
//     tree inside the block (shared memory, one level per barrier).
//     Across super-chunks a second kernel merges the chains up a tree in
//     global memory, where the second child to finish merges the pair (no
//     thread ever waits).  Two x-ordered lower chains A | B merge by walking
//     the common tangent: the cursor b on B moves right while B's next
//     vertex is on or below line(a, b); the cursor a on A moves left while
//     A's previous vertex is on or below line(a, b); repeat until neither
//     moves.  The merged chain is A up to a followed by B from b, which is
//     what the sequential chain produces (same pops, same collinear
//     exclusion).  Each chunk keeps the surviving range [lo, hi] of its
//     chain; chunks whose range empties are unlinked from a list of live
//     chunks.  Upper chains are handled the same way with the predicate
//     mirrored.
//  3. emit: one pass finds the live ranges' output offsets (decoupled
//     look-back over super-chunk counts), and the final kernel copies them
//     to the hull: the lower chain, then the upper chain reversed and
//     without its end points: counter-clockwise from the lexicographically
//     smallest point.
#include <algorithm>

#include "common.cuh"
#include "launch.h"

namespace ch {

namespace {

// Threads per block, and leaves per super-chunk: one set has few super-chunks,
// and 512 threads finish one sooner (10^6 circle points: 163 us the hull with
// 256, 154 so); many sets fill the chip, and 256 wait less for one another (4096
// sets: 1.8 % less than with 512).
constexpr int kOneThreads = 512;
constexpr int kBxThreads = kChainThreads;
constexpr int SC = kChainC;         // points per super-chunk
constexpr int CS = kChainStride;    // chain slots per super-chunk
constexpr int NL = SC + 2;          // sequence capacity: SC points + 2 look-ahead slots
constexpr int SY = NL + 6;
constexpr int kCopyParts = 18;                 // a range is shared by so many warps (4: 3 us more on 10^6 circle points)
constexpr int kCopyLen = CS / kCopyParts;      // entries per part
static_assert(CS % kCopyParts == 0, "parts cover a super-chunk's slots");

// pop / advance test: lower chains drop a vertex when the turn is not
// strictly counter-clockwise, upper chains when it is not strictly clockwise
__device__ __forceinline__ bool drop(int side, const float2 &a, const float2 &b, const float2 &c)
{
    const int o = orient(a.x, a.y, b.x, b.y, c.x, c.y);
    return side == 0 ? o <= 0 : o >= 0;
}

// One strict-turn elimination pass of a warp over the sequence
// src[0 .. len) of point indices: the kept entries go to dst in order;
// returns how many.  Its two ends stay unless there is a neighbour before
// (left) or after (right) them.  Two 32-entry chunks per step, binary32 tier
// of both tests first, so their latencies overlap.  (Inlined once a kernel, and the block's loops are not unrolled: a
// block runs most of this code a few times, and fetching it counts.  A call
// would lose the address space of its arguments.)
__device__ __forceinline__ int warp_elim_pass(const float2 *pts, const uint16_t *src, uint16_t *dst, int len,
                                              int side, int lane, uint32_t lt, bool left = false, bool right = false)
{
    int kept = 0;
    for (int c0 = 0; c0 < len; c0 += 64) {
        int j[2];
        bool test[2];
        float2 a[2], b[2], c[2];
        int o[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            j[u] = c0 + 32 * u + lane;
            test[u] = (j[u] > 0 || left) && (j[u] < len - 1 || (right && j[u] < len));
            const int jj = min(j[u], len - 1);   // (no test: any readable neighbours)
            b[u] = pts[src[jj]];
            a[u] = test[u] ? pts[src[jj - 1]] : b[u];
            c[u] = test[u] ? pts[src[jj + 1]] : b[u];
            o[u] = orient_f32(a[u].x, a[u].y, b[u].x, b[u].y, c[u].x, c[u].y);
        }
        if (__any_sync(0xffffffffu, (test[0] && o[0] == 2) || (test[1] && o[1] == 2))) {
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (o[u] == 2) o[u] = orient_pair(a[u].x, a[u].y, b[u].x, b[u].y, c[u].x, c[u].y);
#pragma unroll 1
            for (int u = 0; u < 2; ++u) {
                const float2 A = u ? a[1] : a[0], B = u ? b[1] : b[0], C = u ? c[1] : c[0];
                if ((u ? test[1] && o[1] == 2 : test[0] && o[0] == 2)) {
                    const int r = orient_last(A.x, A.y, B.x, B.y, C.x, C.y);
                    o[0] = u ? o[0] : r;
                    o[1] = u ? r : o[1];
                }
            }
        }
        uint32_t m[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const bool drop_it = test[u] && (side == 0 ? o[u] <= 0 : o[u] >= 0);
            const bool k = j[u] < len && !drop_it;
            m[u] = __ballot_sync(0xffffffffu, k);
            if (k) dst[kept + __popc(m[u] & lt)] = src[j[u]];
            kept += __popc(m[u]);
        }
    }
    __syncwarp();
    return kept;
}

// ---------------------------------------------------------------------------
// tangent walk of the in-block merge (the global one: MergeSide)
// ---------------------------------------------------------------------------
// Acc provides lo/hi/prv/nxt get+set per chunk and point(side, chunk, k).
template <class Acc>
__device__ void merge_walk(Acc &A, int side, int fa, int la, int fb, int lb)
{
    int ca = la, ka = A.hi(side, ca);
    int cb = fb, kb = A.lo(side, cb);
    int loa = A.lo(side, ca), hib = A.hi(side, cb);
    float2 pa = A.point(side, ca, ka);
    float2 pb = A.point(side, cb, kb);
    for (;;) {
        bool moved = false;
        for (;;) {   // advance b
            int nc = cb, nk = kb + 1, nhi = hib;
            if (kb >= hib) {
                if (cb == lb) break;
                nc = A.nxt(side, cb);
                nk = A.lo(side, nc);
                nhi = A.hi(side, nc);
            }
            const float2 q = A.point(side, nc, nk);
            if (!drop(side, pa, pb, q)) break;
            if (nc != cb) {   // chunk cb is now entirely removed
                A.set_range(side, cb, 1, 0);
                cb = nc;
                hib = nhi;
            }
            kb = nk;
            pb = q;
            moved = true;
        }
        for (;;) {   // retreat a
            int pc = ca, pk = ka - 1, plo = loa;
            if (ka <= loa) {
                if (ca == fa) break;
                pc = A.prv(side, ca);
                plo = A.lo(side, pc);
                pk = A.hi(side, pc);
            }
            const float2 q = A.point(side, pc, pk);
            if (!drop(side, q, pa, pb)) break;
            if (pc != ca) {
                A.set_range(side, ca, 1, 0);
                ca = pc;
                loa = plo;
            }
            ka = pk;
            pa = q;
            moved = true;
        }
        if (!moved) break;
    }
    A.set_hi(side, ca, ka);
    A.set_lo(side, cb, kb);
    A.link(side, ca, cb);
}

// ---------------------------------------------------------------------------
// in-block state
// ---------------------------------------------------------------------------
template <int LT>
__device__ __forceinline__ void side_barrier(int side)   // of the warps that work on one side
{
    __syncwarp();   // (whole warps arrive)
    asm volatile("bar.sync %0, %1;" ::"r"(1 + side), "n"(LT / 2) : "memory");
}

template <int LT>
struct ChainSmem {
    static constexpr int NWB = LT / 32;                              // warps per block
    static constexpr int LWMAX = ((NL + NWB - 1) / NWB + 31) / 32;   // longest leaf
    float2 pts[NL];               // staged points; [SC], [SC+1]: look-ahead lowest / highest
    union {
        struct {
            // from 0: the two sides' sequences one after the other (a point
            // between the ends is on one side at most: up to SC + 4 entries);
            // from SY: lowest / highest point of the run that ends at a point,
            // then the passes' other buffer
            uint16_t seq[SY + 2 * NL];
            uint8_t stk[LWMAX * LT];      // leaf stacks: entry j of leaf t at [j * LT + t]
            int16_t lb[LT];               // leaf t's first entry in the flat list array
            int16_t lo[LT], hi[LT], prv[LT], nxt[LT], first[LT], last[LT];
        };
        unsigned long long tmp[SC];       // local_sort's second buffer (pts is its first)
    };
    uint16_t perm[SC];            // unsorted set: staged point -> its place in the input
    uint32_t wsum[LT / 32];
    uint32_t total;
    float red_y[2][LT / 32];      // look-ahead reduction scratch
    unsigned long long red_q[2][LT / 32];
    uint32_t ext_pos[2];          // global positions of the look-ahead lowest / highest
    uint32_t ext_idx[2];          // and their point indices
    float prev_x;
    int has_prev;
    int seq_len[2];               // per side: its length, and whether every turn is strict
    int strict[2];
    int run[4];                   // lowest, highest point of the set's first run, of its last
};

// leaf c's entries start at flat[lb[c]]; its stack holds offsets from there
template <int LT>
struct SmemAcc {
    ChainSmem<LT> &s;
    const uint16_t *flat;
    __device__ int lo(int, int c) const { return s.lo[c]; }
    __device__ int hi(int, int c) const { return s.hi[c]; }
    __device__ int prv(int, int c) const { return s.prv[c]; }
    __device__ int nxt(int, int c) const { return s.nxt[c]; }
    __device__ void set_range(int, int c, int l, int h) const
    {
        s.lo[c] = (int16_t)l;
        s.hi[c] = (int16_t)h;
    }
    __device__ void set_lo(int, int c, int l) const { s.lo[c] = (int16_t)l; }
    __device__ void set_hi(int, int c, int h) const { s.hi[c] = (int16_t)h; }
    __device__ void link(int, int a, int b) const
    {
        s.nxt[a] = (int16_t)b;
        s.prv[b] = (int16_t)a;
    }
    __device__ float2 point(int, int c, int k) const { return s.pts[flat[s.lb[c] + s.stk[k * LT + c]]]; }
};

// Exclusive scan of one count per thread over the block; the total goes to
// s.total.  Contains two barriers.
template <int LT>
__device__ __forceinline__ uint32_t block_scan(ChainSmem<LT> &s, uint32_t v)
{
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    uint32_t incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
    }
    if (lane == 31) s.wsum[warp] = incl;
    __syncthreads();
    uint32_t before = 0, total = 0;
#pragma unroll
    for (int w = 0; w < LT / 32; ++w) {
        const uint32_t u = s.wsum[w];
        if (w < warp) before += u;
        total += u;
    }
    if (t == 0) s.total = total;
    __syncthreads();
    return before + incl - v;
}

// ---------------------------------------------------------------------------
// global state (one "chunk" = one super-chunk)
// ---------------------------------------------------------------------------
struct ChainPtrs {
    const uint32_t *keys;             // sorted ord(x)
    const unsigned long long *pay;    // sorted ord(y) << 32 | index
    uint32_t *pos0, *pos1;            // chain vertices: sorted positions, super-chunk c at [c * CS, ...)
    float2 *pt0, *pt1;                // chain vertices: coordinates
    int32_t *chunk;                   // per side lo, hi (the surviving range), then per side prv, nxt, n_chunks each
    int64_t n_chunks;
    int32_t *node;                    // 4 ints per tree node: firstL lastL firstU lastU
    int32_t *node_cnt;                // arrivals per node and side (zeroed at the start of each call)

    // (no arrays: an index known only at run time would put them in local memory)
    __device__ uint32_t *pos(int side) const { return side ? pos1 : pos0; }
    __device__ float2 *pt(int side) const { return side ? pt1 : pt0; }
    __device__ int32_t *lo(int side) const { return chunk + 2 * side * n_chunks; }
    __device__ int32_t *hi(int side) const { return chunk + (2 * side + 1) * n_chunks; }
    __device__ int32_t *prv(int side) const { return chunk + (4 + 2 * side) * n_chunks; }
    __device__ int32_t *nxt(int side) const { return chunk + (5 + 2 * side) * n_chunks; }
};

__device__ __forceinline__ ChainPtrs chain_ptrs(void *ws, const Layout &L, uint32_t buf)
{
    return {buf ? at<uint32_t>(ws, L.keys[1]) : at<uint32_t>(ws, L.keys[0]),
            buf ? at<unsigned long long>(ws, L.pay[1]) : at<unsigned long long>(ws, L.pay[0]),
            at<uint32_t>(ws, L.chain_pos[0]), at<uint32_t>(ws, L.chain_pos[1]),
            at<float2>(ws, L.chain_pt[0]), at<float2>(ws, L.chain_pt[1]),
            at<int32_t>(ws, L.chunk), L.n_chunks, at<int32_t>(ws, L.node), at<int32_t>(ws, L.node_cnt)};
}

__device__ __forceinline__ float2 sorted_point(const ChainPtrs &P, int64_t q)
{
    return make_float2(key_float(__ldg(P.keys + q)), key_float((uint32_t)(__ldg(P.pay + q) >> 32)));
}

// The common tangent of two neighbouring chains, by one warp: the merge_walk of
// chunks fa..la | fb..lb.  Values written by other blocks are read through L2
// (ld.cg): this thread's L1 may hold stale lines.
// The walk's steps are dependent loads, some 0.6 us each, and a merge takes
// tens of them.  Trees on the way (one thread per node): 10^8 ellipse points
// 154 us, 39 so; 10^6 circle points 68, 28.
// Here the lanes test 32 vertices at once, the next 32 in a row first, then 32
// spread over the rest of the chunk: as seen from a point beside it, the
// vertices of a strictly convex chain that the walk passes come before those
// it does not.
struct MergeSide {
    const float2 *pt;
    int32_t *lo, *hi, *prv, *nxt;
    int side;
    __device__ float2 point(int c, int k) const { return __ldcg(pt + (int64_t)c * CS + k); }

    // From vertex k of chunk c on (step d = 1: up to e, -1: down to e): the
    // number of vertices that are passed, 0 .. |e - k|, as seen from `from`;
    // p, vertex k, becomes the vertex reached.
    __device__ int passed(int c, int k, int e, int d, const float2 &from, float2 &p) const
    {
        const int lane = (int)lane_id(), n = d > 0 ? e - k : k - e;
        int i = 0, stride = 1;
        while (i < n) {
            const int l = i + lane * stride;
            bool pass = false;
            float2 u = p, v = p;
            if (l < n) {
                u = point(c, k + d * l);
                v = point(c, k + d * (l + 1));
                pass = d > 0 ? drop(side, from, u, v) : drop(side, v, u, from);
            }
            const int f = __ffs(~__ballot_sync(0xffffffffu, pass)) - 1;   // the first that stays (-1: none)
            if (f == 0) break;
            // passed for sure: all before and at the last lane that passed
            const int last = f < 0 ? 31 : f - 1;
            i += last * stride + 1;
            p.x = __shfl_sync(0xffffffffu, v.x, last);
            p.y = __shfl_sync(0xffffffffu, v.y, last);
            if (f > 0 && stride == 1) break;
            stride = max(1, (n - i + 31) / 32);
            if (f > 0) stride = 1;
        }
        return i;
    }

    __device__ void merge(int fa, int la, int fb, int lb) const
    {
        const int lane = (int)lane_id();
        int ca = la, cb = fb;
        int loa = __ldcg(lo + ca), ka = __ldcg(hi + ca), kb = __ldcg(lo + cb), hib = __ldcg(hi + cb);
        float2 pa = point(ca, ka), pb = point(cb, kb);
        for (;;) {
            bool moved = false;
            for (;;) {   // advance b
                const int m = passed(cb, kb, hib, 1, pa, pb);
                moved |= m > 0;
                kb += m;
                if (kb < hib || cb == lb) break;
                const int nc = __ldcg(nxt + cb), nk = __ldcg(lo + nc);
                const float2 q = point(nc, nk);
                if (!drop(side, pa, pb, q)) break;
                if (lane == 0) lo[cb] = 1, hi[cb] = 0;   // that chunk is gone
                cb = nc;
                kb = nk;
                hib = __ldcg(hi + nc);
                pb = q;
                moved = true;
            }
            for (;;) {   // retreat a
                const int m = passed(ca, ka, loa, -1, pb, pa);
                moved |= m > 0;
                ka -= m;
                if (ka > loa || ca == fa) break;
                const int pc = __ldcg(prv + ca), pk = __ldcg(hi + pc);
                const float2 q = point(pc, pk);
                if (!drop(side, q, pa, pb)) break;
                if (lane == 0) lo[ca] = 1, hi[ca] = 0;
                ca = pc;
                ka = pk;
                loa = __ldcg(lo + pc);
                pa = q;
                moved = true;
            }
            if (!moved) break;
        }
        if (lane == 0) {
            hi[ca] = ka;
            lo[cb] = kb;
            nxt[ca] = cb;
            prv[cb] = ca;
        }
    }
};

// One warp climbs one side of a set's merge tree from its super-chunk c (0 <=
// c < nsc; leaves at coff, nodes at noff): the second child to arrive at a
// node merges its two children and continues upward (no warp ever waits).
__device__ void climb(const ChainPtrs &P, int side, int64_t c, int64_t nsc, int64_t coff, int64_t noff)
{
    const MergeSide M{P.pt(side), P.lo(side), P.hi(side), P.prv(side), P.nxt(side), side};
    const uint32_t lane = lane_id();
    int64_t node = c, w = nsc, nb_child = 0, nb = 0;   // nb: base of the level above
    int level = 0;
    // first and last live super-chunk (absolute; -1: none) of child j of this level
    const auto ends = [&](int64_t j) {
        if (level == 0) {
            const int ci = (int)(coff + j);
            return __ldcg(M.hi + ci) >= __ldcg(M.lo + ci) ? make_int2(ci, ci) : make_int2(-1, -1);
        }
        const int32_t *r = P.node + (noff + nb_child + j) * 4 + 2 * side;
        return make_int2(__ldcg(r), __ldcg(r + 1));
    };
    while (w > 1) {
        const int64_t parent = node >> 1, pw = (w + 1) / 2;
        int2 rec;
        if ((node ^ 1) >= w) {
            rec = ends(node);
        } else {
            int before = 0;
            if (lane == 0) {
                __threadfence();
                before = atomicAdd(P.node_cnt + noff + nb + parent, side ? 0x10000 : 1) >> (side ? 16 : 0);
                __threadfence();
            }
            if ((__shfl_sync(0xffffffffu, before, 0) & 0xffff) == 0) return;   // first to arrive: the sibling merges
            const int2 A = ends(parent * 2), B = ends(parent * 2 + 1);
            if (A.y < 0) rec = B;
            else if (B.x < 0) rec = A;
            else {
                M.merge(A.x, A.y, B.x, B.y);
                rec = make_int2(A.x, B.y);
            }
        }
        if (lane == 0) {
            int32_t *r = P.node + (noff + nb + parent) * 4 + 2 * side;
            r[0] = rec.x;
            r[1] = rec.y;
        }
        __syncwarp();
        node = parent;
        nb_child = nb;
        nb += pw;
        w = pw;
        ++level;
    }
}

// Block reduction of (y, index << 32 | position) pairs: the lowest (highest)
// y, ties to the lowest index.  Contains two barriers.
template <int LT>
__device__ __forceinline__ void block_extreme_y(ChainSmem<LT> &s, float ylo, unsigned long long qlo, float yhi,
                                                unsigned long long qhi, float &out_ylo, unsigned long long &out_qlo,
                                                float &out_yhi, unsigned long long &out_qhi)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float y1 = __shfl_xor_sync(0xffffffffu, ylo, o);
        const unsigned long long q1 = __shfl_xor_sync(0xffffffffu, qlo, o);
        if (y1 < ylo || (y1 == ylo && q1 < qlo)) {
            ylo = y1;
            qlo = q1;
        }
        const float y2 = __shfl_xor_sync(0xffffffffu, yhi, o);
        const unsigned long long q2 = __shfl_xor_sync(0xffffffffu, qhi, o);
        if (y2 > yhi || (y2 == yhi && q2 < qhi)) {
            yhi = y2;
            qhi = q2;
        }
    }
    if (lane == 0) {
        s.red_y[0][warp] = ylo;
        s.red_q[0][warp] = qlo;
        s.red_y[1][warp] = yhi;
        s.red_q[1][warp] = qhi;
    }
    __syncthreads();
    out_ylo = s.red_y[0][0];
    out_qlo = s.red_q[0][0];
    out_yhi = s.red_y[1][0];
    out_qhi = s.red_q[1][0];
    for (int w = 1; w < LT / 32; ++w) {
        if (s.red_y[0][w] < out_ylo || (s.red_y[0][w] == out_ylo && s.red_q[0][w] < out_qlo)) {
            out_ylo = s.red_y[0][w];
            out_qlo = s.red_q[0][w];
        }
        if (s.red_y[1][w] > out_yhi || (s.red_y[1][w] == out_yhi && s.red_q[1][w] < out_qhi)) {
            out_yhi = s.red_y[1][w];
            out_qhi = s.red_q[1][w];
        }
    }
    __syncthreads();
}

// Stages the m <= SC unsorted survivors at `base` in the order of x (equal x
// in any order): pts and perm.  Each warp sorts 32 keys at a time in registers
// (a bitonic network), then runs are merged in pairs by merge path (Odeh, Green
// et al. 2012): a thread finds by binary search where its stretch of the
// output begins in both runs and merges that stretch.
// Bound by latency.  A set that fits one block need not be written back
// between digits: the histogram and four passes over global memory take 57 us
// on 4200 survivors, this 27 on 4096.  (Every key by a binary search in the
// other run instead of the serial merge: 40.)
template <int LT>
__device__ void local_sort(ChainSmem<LT> &sm, const ChainPtrs &P, int64_t base, int m)
{
    const int t = threadIdx.x, lane = t & 31;
    const int C = ((m + LT - 1) / LT) | 1;   // outputs per thread and round; odd: no bank conflicts in the stores
    unsigned long long *src = reinterpret_cast<unsigned long long *>(sm.pts), *dst = sm.tmp;
    for (int i0 = t - lane; i0 < m; i0 += LT) {
        const int i = i0 + lane;
        unsigned long long v = i < m ? ((unsigned long long)__ldg(P.keys + base + i) << 32) | (uint32_t)i : ~0ull;
#pragma unroll
        for (int g = 2; g <= 32; g <<= 1) {
#pragma unroll
            for (int h = g >> 1; h > 0; h >>= 1) {
                const unsigned long long o = __shfl_xor_sync(0xffffffffu, v, h);
                if ((o < v) == (((lane & g) == 0) == ((lane & h) == 0))) v = o;
            }
        }
        if (i < m) src[i] = v;
    }
    __syncthreads();
    for (int w = 32; w < m; w <<= 1) {
        int o = t * C, pair = o & ~(2 * w - 1);
        const int end = min(o + C, m);
        if (o < end) {
            // places a and b in the pair's two runs before output o
            int la = min(w, m - pair), lb = min(w, max(0, m - pair - w));
            int lo = max(0, o - pair - lb), hi = min(o - pair, la);
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (src[pair + mid] < src[pair + w + (o - pair) - 1 - mid]) lo = mid + 1;
                else hi = mid;
            }
            int a = lo, b = o - pair - lo;
            unsigned long long ka = a < la ? src[pair + a] : ~0ull, kb = b < lb ? src[pair + w + b] : ~0ull;
            for (;;) {
                const int stop = min(end, pair + 2 * w);
                for (; o < stop; ++o) {
                    const bool first = ka < kb;
                    dst[o] = first ? ka : kb;
                    a += first ? 1 : 0;
                    b += first ? 0 : 1;
                    const bool more = first ? a < la : b < lb;
                    const unsigned long long next = more ? src[pair + (first ? a : w + b)] : ~0ull;
                    ka = first ? next : ka;
                    kb = first ? kb : next;
                }
                if (o == end) break;
                pair = o;   // the next pair
                la = min(w, m - pair);
                lb = min(w, max(0, m - pair - w));
                a = b = 0;
                ka = src[pair];
                kb = lb > 0 ? src[pair + w] : ~0ull;
            }
        }
        __syncthreads();
        unsigned long long *u = src;
        src = dst;
        dst = u;
    }
    unsigned long long v[SC / LT];
#pragma unroll
    for (int k = 0; k < SC / LT; ++k)
        if (t + k * LT < m) v[k] = src[t + k * LT];
    __syncthreads();
#pragma unroll
    for (int k = 0; k < SC / LT; ++k) {
        const int i = t + k * LT;
        if (i >= m) continue;
        const uint32_t e = (uint32_t)v[k];
        sm.pts[i] = make_float2(key_float((uint32_t)(v[k] >> 32)), key_float((uint32_t)(__ldg(P.pay + base + e) >> 32)));
        sm.perm[i] = (uint16_t)e;
    }
}

// The chains of one super-chunk: sorted positions [base, base + m) of a set
// occupying [sbeg, send); results go to chain slot j.  local: the super-chunk
// is a whole set and not sorted yet.  Called by all threads of the block.
template <int LT>
__device__ __forceinline__ void superchunk(ChainSmem<LT> &sm, const ChainPtrs &P, int64_t j, int64_t base, int m,
                                           int64_t sbeg, int64_t send, bool local)
{
    constexpr int NWB = LT / 32, NWS = NWB / 2;   // warps per block, per side
    const auto place = [&](int e) { return base + (local ? (int)sm.perm[e] : e); };   // of a staged point
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t lt = (1u << lane) - 1u;
    const float kInf = __int_as_float(0x7f800000);
    const int64_t sc = j;
    {
        // ---- stage the super-chunk (coalesced), decoded to points
        if (local) local_sort(sm, P, base, m);
        else
            for (int i = t; i < m; i += LT) sm.pts[i] = sorted_point(P, base + i);
        if (t == 0) {
            sm.has_prev = base > sbeg;
            sm.prev_x = base > sbeg ? key_float(__ldg(P.keys + base - 1)) : 0.0f;
        }
        __syncthreads();

        const float xr = sm.pts[m - 1].x;
        const bool cont = sm.has_prev && sm.pts[0].x == sm.prev_x;   // it starts inside a run
        if (cont && xr == sm.prev_x) {   // the whole super-chunk continues an earlier run
            if (t == 0)
                for (int side = 0; side < 2; ++side) {
                    P.lo(side)[sc] = 0;
                    P.hi(side)[sc] = -1;
                }
            __syncthreads();
            return;
        }
        // ---- look ahead when the last run continues past the super-chunk
        const bool ext = base + m < send && key_float(__ldg(P.keys + base + m)) == xr;
        int64_t run_end = base + m;
        if (ext) {
            float ylo = kInf, yhi = -kInf;
            unsigned long long qlo = ~0ull, qhi = ~0ull;   // index << 32 | position
            for (int64_t q0 = base + m;; q0 += LT) {
                const int64_t q = q0 + t;
                const bool in_run = q < send && key_float(__ldg(P.keys + q)) == xr;
                if (in_run) {
                    const unsigned long long pv = __ldg(P.pay + q), iq = (pv << 32) | (uint32_t)q;
                    const float y = key_float((uint32_t)(pv >> 32));
                    if (y < ylo || (y == ylo && iq < qlo)) {
                        ylo = y;
                        qlo = iq;
                    }
                    if (y > yhi || (y == yhi && iq < qhi)) {
                        yhi = y;
                        qhi = iq;
                    }
                }
                // the keys are sorted, so the run's positions are contiguous
                const int n_in = __syncthreads_count(in_run);
                if (n_in < LT) {
                    run_end = q0 + n_in;
                    break;
                }
            }
            float oyl, oyh;
            unsigned long long oql, oqh;
            block_extreme_y(sm, ylo, qlo, yhi, qhi, oyl, oql, oyh, oqh);
            if (t == 0) {
                sm.pts[SC] = make_float2(xr, oyl);
                sm.pts[SC + 1] = make_float2(xr, oyh);
                sm.ext_pos[0] = (uint32_t)oql;
                sm.ext_pos[1] = (uint32_t)oqh;
                sm.ext_idx[0] = (uint32_t)(oql >> 32);
                sm.ext_idx[1] = (uint32_t)(oqh >> 32);
            }
        }
        const bool holds_last = run_end == send;
        __syncthreads();
        const auto index_of = [&](int e) {
            return e < SC ? (uint32_t)__ldg(P.pay + place(e)) : sm.ext_idx[e - SC];
        };
        const auto lower = [&](float y, int e, float y0, int e0) {
            return y < y0 || (y == y0 && e != e0 && index_of(e) < index_of(e0));
        };
        const auto higher = [&](float y, int e, float y0, int e0) {
            return y > y0 || (y == y0 && e != e0 && index_of(e) < index_of(e0));
        };
        // ---- runs, their lowest and highest points, and the sides' sequences
        // in one sweep.  A warp takes a segment of the points and the runs that
        // start in it, 32 points at a time (a scan over the lanes of a run;
        // equal points: the lowest index).  Lower: the lowest of every run, then
        // the highest of the very last run; upper: the lowest of the very first
        // run, then the highest of every run.  Of the points beside the first
        // and last x only those strictly below (above) the segment joining two
        // points there can be vertices (a ring's chunk holds both arcs by
        // turns).  Bound by latency, like all of this kernel on few chunks:
        // runs, representatives and sequences in steps of their own (a thread
        // per run) took 24000 to 48000 cycles on a ring's chunk, this 16000 to 36000.
        uint16_t *const low = sm.seq + SY, *const high = low + NL;
        int n0, n1;
        {
            const float2 A = sm.pts[0], B = sm.pts[m - 1];
            const int S = (((m + NWB - 1) / NWB) + 31) & ~31, j0 = min(warp * S, m), j1 = min(j0 + S, m);
            const bool starts = j0 == 0 ? !cont : j0 < m && sm.pts[j0].x != sm.pts[j0 - 1].x;   // with a run of its own
            const bool crosses = j1 < m && j1 > j0 && sm.pts[j1].x == sm.pts[j1 - 1].x;         // its last run goes on
            uint32_t masks0 = 0, masks1 = 0, c01 = 0;   // lane c: the kept ones of the c-th 32 points; both counts
            bool owned = starts;                        // the run open at the 32 points' start, and its state
            float cylo = 0.0f, cyhi = 0.0f;
            int clo = 0, chi = 0;
#pragma unroll 1
            for (int c = 0; j0 + c * 32 < j1; ++c) {
                const int i = min(j0 + c * 32 + lane, j1 - 1);
                const bool in = j0 + c * 32 + lane < j1;
                const float2 p = sm.pts[i];
                const bool head = in && (i == j0 ? starts : sm.pts[i - 1].x != p.x);
                const bool tail = in && (i == j1 - 1 || sm.pts[i + 1].x != p.x);
                const uint32_t hm = __ballot_sync(0xffffffffu, head), vm = __ballot_sync(0xffffffffu, in);
                int lo = i, hi = i;
                float ylo = p.y, yhi = p.y;
                bool mine = true;
                if (hm != vm) {
                    uint32_t ilo = (uint32_t)__ldg(P.pay + place(i)), ihi = ilo;   // equal points: by index
                    const auto take = [&](float y1, uint32_t i1, int e1, float y2, uint32_t i2, int e2) {
                        if (y1 < ylo || (y1 == ylo && i1 < ilo)) {
                            ylo = y1;
                            ilo = i1;
                            lo = e1;
                        }
                        if (y2 > yhi || (y2 == yhi && i2 < ihi)) {
                            yhi = y2;
                            ihi = i2;
                            hi = e2;
                        }
                    };
                    const uint32_t upto = hm & (lt | (1u << lane));
                    const int start = upto ? 31 - __clz(upto) : 0;
                    // (runs are short: 1053 -> 1020 us on those points)
                    const int reach = (int)__reduce_max_sync(0xffffffffu, in ? (uint32_t)(lane - start) : 0u);
#pragma unroll 1
                    for (int o = 1; o <= reach; o <<= 1) {
                        const float y1 = __shfl_up_sync(0xffffffffu, ylo, o), y2 = __shfl_up_sync(0xffffffffu, yhi, o);
                        const uint32_t i1 = __shfl_up_sync(0xffffffffu, ilo, o), i2 = __shfl_up_sync(0xffffffffu, ihi, o);
                        const int e1 = __shfl_up_sync(0xffffffffu, lo, o), e2 = __shfl_up_sync(0xffffffffu, hi, o);
                        if (lane - o >= start) take(y1, i1, e1, y2, i2, e2);
                    }
                    if (upto == 0u) {
                        mine = owned;
                        if (c > 0)   // the run open before these points
                            take(cylo, (uint32_t)__ldg(P.pay + place(clo)), clo, cyhi,
                                 (uint32_t)__ldg(P.pay + place(chi)), chi);
                    }
                }
                int end_of_run = i + 1;
                if (crosses && j0 + c * 32 + 32 >= j1) {   // the run of the segment's last point goes on
                    const int last = j1 - 1 - (j0 + c * 32);
                    float ay = __int_as_float(0x7f800000), by = -ay;
                    int ae = -1, be = -1, q = j1 + lane;
                    for (; q < m && sm.pts[q].x == sm.pts[j1 - 1].x; q += 32) {
                        const float y = sm.pts[q].y;
                        if (ae < 0 || lower(y, q, ay, ae)) {
                            ay = y;
                            ae = q;
                        }
                        if (be < 0 || higher(y, q, by, be)) {
                            by = y;
                            be = q;
                        }
                    }
                    __syncwarp();
                    const int stop = (int)__reduce_min_sync(0xffffffffu, (uint32_t)min(q, m));   // the first past the run
#pragma unroll 1
                    for (int o = 16; o > 0; o >>= 1) {
                        const float y1 = __shfl_xor_sync(0xffffffffu, ay, o), y2 = __shfl_xor_sync(0xffffffffu, by, o);
                        const int e1 = __shfl_xor_sync(0xffffffffu, ae, o), e2 = __shfl_xor_sync(0xffffffffu, be, o);
                        if (e1 >= 0 && (ae < 0 || lower(y1, e1, ay, ae))) {
                            ay = y1;
                            ae = e1;
                        }
                        if (e2 >= 0 && (be < 0 || higher(y2, e2, by, be))) {
                            by = y2;
                            be = e2;
                        }
                    }
                    if (lane == last) {
                        if (lower(ay, ae, ylo, lo)) {
                            ylo = ay;
                            lo = ae;
                        }
                        if (higher(by, be, yhi, hi)) {
                            yhi = by;
                            hi = be;
                        }
                        end_of_run = stop;
                    }
                }
                const bool rep = tail && mine;
                int o0 = 0, o1 = 0;
                const bool end = p.x == A.x || p.x == B.x;
                if (rep) {
                    if (ext && end_of_run == m) {   // and past the super-chunk
                        if (lower(sm.pts[SC].y, SC, ylo, lo)) lo = SC;
                        if (higher(sm.pts[SC + 1].y, SC + 1, yhi, hi)) hi = SC + 1;
                    }
                    low[i] = (uint16_t)lo;
                    high[i] = (uint16_t)hi;
                    if (p.x == A.x) {
                        sm.run[0] = lo;
                        sm.run[1] = hi;
                    }
                    if (p.x == B.x) {
                        sm.run[2] = lo;
                        sm.run[3] = hi;
                    }
                    if (!end) {
                        const float2 u = sm.pts[lo];
                        o0 = o1 = orient(A.x, A.y, u.x, u.y, B.x, B.y);
                        if (hi != lo) {
                            const float2 v = sm.pts[hi];
                            o1 = orient(A.x, A.y, v.x, v.y, B.x, B.y);
                        }
                    }
                }
                const uint32_t m0 = __ballot_sync(0xffffffffu, rep && (end || o0 > 0));
                const uint32_t m1 = __ballot_sync(0xffffffffu, rep && (end || o1 < 0));
                if (lane == c) {
                    masks0 = m0;
                    masks1 = m1;
                }
                c01 += __popc(m0) + (__popc(m1) << 16);
                cylo = __shfl_sync(0xffffffffu, ylo, 31);
                cyhi = __shfl_sync(0xffffffffu, yhi, 31);
                clo = __shfl_sync(0xffffffffu, lo, 31);
                chi = __shfl_sync(0xffffffffu, hi, 31);
                owned = __shfl_sync(0xffffffffu, mine ? 1 : 0, 31) != 0;
            }
            if (lane == 0) sm.wsum[warp] = c01;
            __syncthreads();
            const bool last_two = holds_last && sm.pts[sm.run[3]].y > sm.pts[sm.run[2]].y;
            const bool first_two = base == sbeg && sm.pts[sm.run[1]].y > sm.pts[sm.run[0]].y;
            uint32_t before = 0, total = 0;
#pragma unroll
            for (int w = 0; w < NWB; ++w) {
                const uint32_t u = sm.wsum[w];
                if (w < warp) before += u;
                total += u;
            }
            n0 = (int)(total & 0xffffu) + (last_two ? 1 : 0);
            n1 = (int)(total >> 16) + (first_two ? 1 : 0);
            int at0 = (int)(before & 0xffffu), at1 = n0 + (int)(before >> 16) + (first_two ? 1 : 0);
#pragma unroll 2
            for (int c = 0; j0 + c * 32 < j1; ++c) {
                const int j = j0 + c * 32 + lane;
                const uint32_t m0 = __shfl_sync(0xffffffffu, masks0, c), m1 = __shfl_sync(0xffffffffu, masks1, c);
                if ((m0 >> lane) & 1u) sm.seq[at0 + __popc(m0 & lt)] = low[j];
                if ((m1 >> lane) & 1u) sm.seq[at1 + __popc(m1 & lt)] = high[j];
                at0 += __popc(m0);
                at1 += __popc(m1);
            }
            if (t == 0) {
                if (last_two) sm.seq[n0 - 1] = (uint16_t)sm.run[3];
                if (first_two) sm.seq[n0] = (uint16_t)sm.run[0];
            }
            __syncthreads();
        }

        // ---- elimination, half of the block per side: rounds of one pass over
        // the whole sequence, each warp its share, then passes inside the
        // shares (their ends stay), then the shares closed up again; done when
        // the first pass of a round drops nothing.  Many super-chunks are bound
        // by issue, so a share is whole steps of a pass, and of a short sequence
        // fewer warps have one (3 10^7 unfiltered circle points, this kernel:
        // 1242 us with even shares, 1053 so)
        {
            const int side = warp / NWS, gw = warp % NWS;
            uint16_t *const X = sm.seq + (side ? n0 : 0), *const Y = X + SY;
            int len = side ? n1 : n0, w0 = 0, wl = 0, pass = 0, round = 0;
            bool strict = len <= 2, whole = true, in_y = false;
#pragma unroll 1
            while (!strict) {
                if (whole) {
                    const int S = ((len + NWS - 1) / NWS + 63) & ~63;
                    w0 = min(gw * S, len);
                    wl = min(S, len - w0);
                    in_y = false;
                }
                const int kept = warp_elim_pass(sm.pts, (in_y ? Y : X) + w0, (in_y ? X : Y) + w0, wl, side, lane, lt,
                                                whole && w0 > 0, whole && w0 + wl < len);
                in_y = !in_y;
                bool closed = kept <= 2;
                if (whole) {
                    if (lane == 0) sm.wsum[warp] = (uint32_t)kept;
                    side_barrier<LT>(side);
                    int total = 0;
#pragma unroll
                    for (int w = 0; w < NWS; ++w) total += (int)sm.wsum[side * NWS + w];
                    if (total == len) {
                        strict = true;
                        break;
                    }
                    whole = false;
                    pass = 0;
                } else {
                    closed |= kept == wl || ++pass == kElimPasses;
                }
                wl = kept;
                if (!closed) continue;
                if (!in_y) {
                    for (int i = lane; i < wl; i += 32) Y[w0 + i] = X[w0 + i];
                }
                side_barrier<LT>(side);   // wsum has been read
                if (lane == 0) sm.wsum[warp] = (uint32_t)wl;
                side_barrier<LT>(side);
                int at = 0;
                len = 0;
#pragma unroll
                for (int w = 0; w < NWS; ++w) {
                    const int u = (int)sm.wsum[side * NWS + w];
                    if (w < gw) at += u;
                    len += u;
                }
                for (int i = lane; i < wl; i += 32) X[at + i] = Y[w0 + i];
                side_barrier<LT>(side);
                strict = len <= 2;
                if (++round == kElimRounds) break;
                whole = true;
            }
            if (gw == 0 && lane == 0) {
                sm.seq_len[side] = len;
                sm.strict[side] = strict ? 1 : 0;
            }
        }
        __syncthreads();

        for (int side = 0; side < 2; ++side) {
            const int o = side ? n0 : 0, blen = sm.seq_len[side];
            const uint16_t *flat = sm.seq + o;
            if (sm.strict[side]) {   // its own chain
                uint32_t *dpos = P.pos(side) + sc * CS;
                float2 *dpt = P.pt(side) + sc * CS;
                for (int q = t; q < blen; q += LT) {
                    const int e = flat[q];
                    dpos[q] = e < SC ? (uint32_t)place(e) : sm.ext_pos[e - SC];
                    dpt[q] = sm.pts[e];
                }
                if (t == 0) {
                    P.lo(side)[sc] = 0;
                    P.hi(side)[sc] = blen - 1;
                }
                continue;
            }
            // not yet a chain: leaves and merges over the block's sequence
            const int S2 = (blen + NWB - 1) / NWB, w0 = warp * S2;
            const int wl = max(0, min(S2, blen - w0));
            // ---- leaf chains: lane l takes [l * LW, l * LW + LW) of the warp's list
            const int LW = (wl + 31) / 32;
            const int lbase = w0 + lane * LW;
            const int cnt = max(0, min(LW, wl - lane * LW));
            sm.lb[t] = (int16_t)lbase;
            int h = 0;
            float2 t1 = make_float2(0.0f, 0.0f), t2 = t1;   // top and second of the stack
            for (int k = 0; k < cnt; ++k) {
                const float2 p = sm.pts[flat[lbase + k]];
                while (h >= 2 && drop(side, t2, t1, p)) {
                    --h;
                    t1 = t2;
                    if (h >= 2) t2 = sm.pts[flat[lbase + sm.stk[(h - 2) * LT + t]]];
                }
                sm.stk[h * LT + t] = (uint8_t)k;
                ++h;
                t2 = t1;
                t1 = p;
            }
            sm.lo[t] = 0;
            sm.hi[t] = (int16_t)(h - 1);
            sm.first[t] = sm.last[t] = (int16_t)(h > 0 ? t : -1);
            __syncwarp();
            // ---- merge tree: five levels inside the warp, then three (256 threads) or four (512) across warps
            const SmemAcc<LT> A{sm, flat};
            for (int w = 1; w < 32; w *= 2) {
                if (lane < 32 / (2 * w)) {
                    const int a0 = warp * 32 + 2 * lane * w, b0 = a0 + w;
                    const int fa = sm.first[a0], la = sm.last[a0];
                    const int fb = sm.first[b0], lb = sm.last[b0];
                    if (la >= 0 && fb >= 0) merge_walk(A, side, fa, la, fb, lb);
                    sm.first[a0] = (int16_t)(la >= 0 ? fa : fb);
                    sm.last[a0] = (int16_t)(fb >= 0 ? lb : la);
                }
                __syncwarp();
            }
            __syncthreads();
            for (int w = 32; w < LT; w *= 2) {
                if (t < LT / (2 * w)) {
                    const int a0 = 2 * t * w, b0 = a0 + w;
                    const int fa = sm.first[a0], la = sm.last[a0];
                    const int fb = sm.first[b0], lb = sm.last[b0];
                    if (la >= 0 && fb >= 0) merge_walk(A, side, fa, la, fb, lb);
                    sm.first[a0] = (int16_t)(la >= 0 ? fa : fb);
                    sm.last[a0] = (int16_t)(fb >= 0 ? lb : la);
                }
                __syncthreads();
            }

            // ---- write the super-chunk's chain contiguously
            const int l = sm.lo[t], hh = sm.hi[t];
            const int c = hh >= l ? hh - l + 1 : 0;
            const int off = (int)block_scan(sm, (uint32_t)c);
            uint32_t *dpos = P.pos(side) + sc * CS + off;
            float2 *dpt = P.pt(side) + sc * CS + off;
            for (int q = 0; q < c; ++q) {
                const int e = flat[lbase + sm.stk[(l + q) * LT + t]];
                dpos[q] = e < SC ? (uint32_t)place(e) : sm.ext_pos[e - SC];
                dpt[q] = sm.pts[e];
            }
            if (t == 0) {
                P.lo(side)[sc] = 0;
                P.hi(side)[sc] = (int)sm.total - 1;
            }
            __syncthreads();
        }
        __syncthreads();   // sm is staged again
    }
}

__device__ __forceinline__ void copy_chain_part(const ChainPtrs &P, int side, int64_t c, int part, uint32_t off0,
                                                uint32_t hl, uint32_t hu, uint32_t *out, int64_t limit);

// At most SC survivors (the sort has left them alone): one block sorts them
// and writes the hull itself, and the later kernels have nothing to do.
__global__ void __launch_bounds__(kOneThreads) chain_kernel(void *ws, Layout L, uint32_t *hull_idx, uint32_t *hull_count)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ChainSmem<kOneThreads> &sm = *reinterpret_cast<ChainSmem<kOneThreads> *>(smem_raw);
    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    const Octagon *oct = at<Octagon>(ws, L.oct);
    const uint32_t s = hull_stage_count(ctrl, oct);
    if (s == 0) return;
    const bool local = s <= (uint32_t)SC;   // not sorted yet
    const ChainPtrs P = chain_ptrs(ws, L, local ? ctrl->sort_in : ctrl->final_buf);
    const int64_t nsc = ceil_div((int64_t)s, SC);
    for (int64_t sc = blockIdx.x; sc < nsc; sc += gridDim.x) {
        // the block's next super-chunk streams into L2 meanwhile
        const int64_t nxt = sc + gridDim.x;
        if (threadIdx.x == 0 && nxt < nsc) {
            const uint32_t nn = (uint32_t)min((int64_t)SC, (int64_t)s - nxt * SC);
            bulk_prefetch_l2(P.keys + nxt * SC, (nn * 4u) & ~15u);
            bulk_prefetch_l2(P.pay + nxt * SC, (nn * 8u) & ~15u);
        }
        superchunk(sm, P, sc, sc * SC, (int)min((int64_t)SC, (int64_t)s - sc * SC), 0, s, local);
    }
    if (!local || blockIdx.x != 0) return;
    const uint32_t hl = (uint32_t)__ldcg(P.hi(0)) + 1u, hu = (uint32_t)__ldcg(P.hi(1)) + 1u;   // (behind a barrier)
    for (int it = (int)(threadIdx.x >> 5); it < 2 * kCopyParts; it += kOneThreads / 32)
        copy_chain_part(P, it & 1, 0, it >> 1, 0u, hl, hu, hull_idx, L.n);
    if (threadIdx.x == 0) {
        *hull_count = hl + (hu >= 2 ? hu - 2 : 0u);
        ctrl->small_done = 1u;
    }
}

// Global merge tree over the super-chunks: a warp per super-chunk and side.
constexpr int kMergeThreads = 128;

__global__ void __launch_bounds__(kMergeThreads) chain_merge_kernel(void *ws, Layout L)
{
    kernel_entry();
    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    const Octagon *oct = at<Octagon>(ws, L.oct);
    const uint32_t s = hull_stage_count(ctrl, oct);
    if (s == 0) return;
    const ChainPtrs P = chain_ptrs(ws, L, ctrl->final_buf);
    const int64_t nsc = ceil_div((int64_t)s, SC), step = (int64_t)gridDim.x * (kMergeThreads / 32);
    for (int64_t i = ((int64_t)blockIdx.x * kMergeThreads + threadIdx.x) >> 5; i < 2 * nsc; i += step)
        climb(P, (int)(i & 1), i >> 1, nsc, 0, 0);
}

// ---- many sets: super-chunks never span two sets; each set has its own
// merge tree; the sorted arrays end up in buffer 0 (four passes)
__global__ void __launch_bounds__(kBxThreads) bx_chain_kernel(void *ws, Layout L, BatchLayout BL)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    ChainSmem<kBxThreads> &sm = *reinterpret_cast<ChainSmem<kBxThreads> *>(smem_raw);
    const BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t *sc_set = at<uint32_t>(ws, BL.sc_set);
    const ChainPtrs P = chain_ptrs(ws, L, 0);
    const int64_t nsc = bc->nsc;
    for (int64_t j = blockIdx.x; j < nsc; j += gridDim.x) {
        const uint32_t b = sc_set[j];
        const int64_t sb = (int64_t)sets[b].surv_base, n = sets[b].s;
        const int64_t local = j - sets[b].sc_base;
        superchunk(sm, P, j, sb + local * SC, (int)min((int64_t)SC, n - local * SC), sb, sb + n,
                   n <= (int64_t)kBxLocalMax);
    }
}

__global__ void __launch_bounds__(kMergeThreads) bx_merge_kernel(void *ws, Layout L, BatchLayout BL)
{
    kernel_entry();
    const BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t *sc_set = at<uint32_t>(ws, BL.sc_set);
    const ChainPtrs P = chain_ptrs(ws, L, 0);
    const int64_t nsc = bc->nsc_sort, step = (int64_t)gridDim.x * (kMergeThreads / 32);   // (the others are alone)
    for (int64_t i = ((int64_t)blockIdx.x * kMergeThreads + threadIdx.x) >> 5; i < 2 * nsc; i += step) {
        const int64_t j = i >> 1;
        const SetInfo &S = sets[sc_set[j]];
        climb(P, (int)(i & 1), j - S.sc_base, S.nsc, S.sc_base, S.node_base);
    }
}

// blocks for the merge tree of up to n super-chunks
unsigned merge_grid(int64_t n)
{
    return (unsigned)std::min<int64_t>(ceil_div(2 * n, kMergeThreads / 32), (int64_t)sm_count() * 8);
}

// Output offsets of the live chain ranges of super-chunks [0, nc), per side:
// thread = super-chunk, look-back over tiles of kEmitThreads super-chunks.
// sc_off[side][c] receives the entries of the ranges before c,
// sc_off[side][nc] and h_total the side's total.
struct EmitArgs {
    uint32_t *sc_off[2];
    uint32_t *ticket;
    uint32_t *h_total[2];
};

__device__ void emit_body(void *ws, const Layout &L, const ChainPtrs &P, int64_t nc, const EmitArgs &E)
{
    const int64_t ntiles = ceil_div(nc, kEmitThreads);
    unsigned long long *status[2] = {at<unsigned long long>(ws, L.emit_status[0]),
                                     at<unsigned long long>(ws, L.emit_status[1])};
    constexpr int NW = kEmitThreads / 32;
    __shared__ uint32_t s_tile;
    __shared__ uint32_t s_wsum[2][NW];
    __shared__ unsigned long long s_excl[2];
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = lane_id();
    for (;;) {
        if (tid == 0) s_tile = atomicAdd(E.ticket, 1u);
        __syncthreads();
        const int64_t tile = s_tile;
        if (tile >= ntiles) break;
        const int64_t c = tile * kEmitThreads + tid;
        int32_t cnt[2] = {0, 0};
        if (c < nc) {
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const int32_t lo = __ldcg(P.lo(side) + c), hi = __ldcg(P.hi(side) + c);
                cnt[side] = hi >= lo ? hi - lo + 1 : 0;
            }
        }
        uint32_t pre[2];
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            uint32_t incl = (uint32_t)cnt[side];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += t;
            }
            pre[side] = incl - (uint32_t)cnt[side];
            if (lane == 31) s_wsum[side][warp] = incl;
        }
        __syncthreads();
        if (warp < 2) {
            const int side = (int)warp;
            uint32_t wv = lane < (uint32_t)NW ? s_wsum[side][lane] : 0u;
            uint32_t incl = wv;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= (uint32_t)o) incl += t;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
            if (lane < (uint32_t)NW) s_wsum[side][lane] = incl - wv;
            unsigned long long excl = 0;
            if (tile == 0) {
                if (lane == 0) st_release_u64(status[side], kFlagP | total);
            } else {
                if (lane == 0) st_release_u64(status[side] + tile, kFlagA | total);
                excl = lookback_u64(status[side], tile, ws, L, 30 + side);
                if (lane == 0) st_release_u64(status[side] + tile, kFlagP | ((excl + total) & kValMask));
            }
            if (lane == 0) {
                s_excl[side] = excl;
                if (tile == ntiles - 1) {
                    *E.h_total[side] = (uint32_t)(excl + total);
                    E.sc_off[side][nc] = (uint32_t)(excl + total);
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int side = 0; side < 2; ++side)
            if (c < nc) E.sc_off[side][c] = (uint32_t)(s_excl[side] + s_wsum[side][warp] + pre[side]);
        // (the loop's first barrier orders the next tile's shared writes)
    }
}

// One warp copies a part of super-chunk c's live range of one side to its
// place in the hull: chain entry g of the side (off0: its entries before
// this super-chunk) goes to position g on the lower side; the upper chain
// (hu entries) follows the hl lower ones reversed and without its two ends.
// The warp knows where its range goes, so no position is searched for and
// the chains are copied once.  limit: positions the hull may fill (only a
// look-back that gave up could pass it).

__device__ __forceinline__ void copy_chain_part(const ChainPtrs &P, int side, int64_t c, int part, uint32_t off0,
                                                uint32_t hl, uint32_t hu, uint32_t *out, int64_t limit)
{
    const int32_t lo = __ldcg(P.lo(side) + c), cnt = __ldcg(P.hi(side) + c) - lo + 1;
    const int32_t k1 = min(cnt, (part + 1) * kCopyLen);
    const uint32_t *chain = P.pos(side) + c * CS + lo;
    constexpr int U = 4;   // entries per lane in flight
    for (int32_t k0 = part * kCopyLen + (int32_t)lane_id(); k0 < k1; k0 += 32 * U) {
        uint32_t sp[U], ix[U];
#pragma unroll
        for (int u = 0; u < U; ++u) sp[u] = k0 + 32 * u < k1 ? __ldcg(chain + k0 + 32 * u) : 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) ix[u] = k0 + 32 * u < k1 ? (uint32_t)__ldg(P.pay + sp[u]) : 0u;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (k0 + 32 * u >= k1) continue;
            const uint32_t g = off0 + (uint32_t)(k0 + 32 * u);
            if (side == 1 && (g == 0u || g + 1u >= hu)) continue;   // the ends are the lower chain's
            const int64_t p = side == 0 ? (int64_t)g : (int64_t)hl + (hu - 2u - g);
            if (p < limit) out[p] = ix[u];
        }
    }
}

__global__ void __launch_bounds__(kEmitThreads) emit_kernel(void *ws, Layout L)
{
    kernel_entry();
    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    const Octagon *oct = at<Octagon>(ws, L.oct);
    const uint32_t s = hull_stage_count(ctrl, oct);
    if (s <= (uint32_t)(kEmitThreads * SC)) return;   // hull_copy_kernel adds so few ranges up itself
    const ChainPtrs P = chain_ptrs(ws, L, ctrl->final_buf);
    EmitArgs E{{at<uint32_t>(ws, L.emit_off[0]), at<uint32_t>(ws, L.emit_off[1])},
               &ctrl->emit_ticket[0],
               {&ctrl->h_lower, &ctrl->h_upper}};
    emit_body(ws, L, P, ceil_div((int64_t)s, SC), E);
}

// The hull and its vertex count: the chains' surviving ranges (original
// indices, the low half of the payload) straight to their positions, a warp
// per part of a super-chunk's range.  Up to kEmitThreads super-chunks each
// block adds their lengths up itself, which costs it less than a launch in
// between.
__global__ void __launch_bounds__(kEmitThreads) hull_copy_kernel(void *ws, Layout L, uint32_t *hull_idx,
                                                                 uint32_t *hull_count)
{
    kernel_entry();
    __shared__ uint32_t s_off[2][kEmitThreads], s_w[2][kEmitThreads / 32];
    const Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    if (ctrl->small_done) return;
    const uint32_t s = hull_stage_count(ctrl, at<Octagon>(ws, L.oct));
    if (s == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) *hull_count = 0u;
        return;
    }
    const ChainPtrs P = chain_ptrs(ws, L, ctrl->final_buf);
    const int64_t nsc = ceil_div((int64_t)s, SC);
    const bool few = nsc <= kEmitThreads;
    uint32_t hl = ctrl->h_lower, hu = ctrl->h_upper;
    if (few) {
        const int c = (int)threadIdx.x, lane = c & 31;
        uint32_t n[2] = {0u, 0u}, incl[2];
        if (c < nsc) {
#pragma unroll
            for (int side = 0; side < 2; ++side)
                n[side] = (uint32_t)max(0, __ldcg(P.hi(side) + c) - __ldcg(P.lo(side) + c) + 1);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            incl[side] = n[side];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t u = __shfl_up_sync(0xffffffffu, incl[side], o);
                if (lane >= o) incl[side] += u;
            }
            if (lane == 31) s_w[side][c >> 5] = incl[side];
        }
        __syncthreads();
        uint32_t total[2];
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            uint32_t before = 0;
            total[side] = 0u;
#pragma unroll
            for (int w = 0; w < kEmitThreads / 32; ++w) {
                if (w < c >> 5) before += s_w[side][w];
                total[side] += s_w[side][w];
            }
            s_off[side][c] = before + incl[side] - n[side];
        }
        hl = total[0];
        hu = total[1];
        __syncthreads();
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *hull_count = hl == 0 ? 0u : hl + (hu >= 2 ? hu - 2 : 0u);
    const int64_t items = nsc * 2 * kCopyParts, warps = (int64_t)gridDim.x * (kEmitThreads / 32);
    for (int64_t it = ((int64_t)blockIdx.x * kEmitThreads + threadIdx.x) >> 5; it < items; it += warps) {
        const int64_t c = it / (2 * kCopyParts);
        const int side = (int)(it / kCopyParts) & 1;
        const uint32_t off = few ? s_off[side][c] : __ldg(at<uint32_t>(ws, side ? L.emit_off[1] : L.emit_off[0]) + c);
        copy_chain_part(P, side, c, (int)(it % kCopyParts), off, hl, hu, hull_idx, L.n);
    }
}

// all sets at once: the offsets of every super-chunk's ranges
__global__ void __launch_bounds__(kEmitThreads) bx_emit_kernel(void *ws, Layout L, BatchLayout BL)
{
    kernel_entry();
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    const int64_t nc = bc->nsc;
    if (nc == 0) return;
    const ChainPtrs P = chain_ptrs(ws, L, 0);
    EmitArgs E{{at<uint32_t>(ws, BL.sc_off[0]), at<uint32_t>(ws, BL.sc_off[1])},
               &bc->emit_ticket,
               {&bc->h_lower, &bc->h_upper}};
    emit_body(ws, L, P, nc, E);
}

// The sets' hulls: as hull_copy_kernel, every set's part of the output at
// its hull_offsets entry (a set's hull has at most as many vertices as the
// set has points).
__global__ void __launch_bounds__(kEmitThreads) bx_assemble_kernel(void *ws, Layout L, BatchLayout BL,
                                                                   const int64_t *__restrict__ hull_offsets,
                                                                   uint32_t *hull_idx)
{
    kernel_entry();
    const BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t *sc_set = at<uint32_t>(ws, BL.sc_set);
    const uint32_t *off[2] = {at<uint32_t>(ws, BL.sc_off[0]), at<uint32_t>(ws, BL.sc_off[1])};
    const ChainPtrs P = chain_ptrs(ws, L, 0);
    const int64_t items = (int64_t)bc->nsc * 2 * kCopyParts;
    const int64_t warps = (int64_t)gridDim.x * (kEmitThreads / 32);
    for (int64_t it = ((int64_t)blockIdx.x * kEmitThreads + threadIdx.x) >> 5; it < items; it += warps) {
        const int64_t j = it / (2 * kCopyParts);
        const int side = (int)(it / kCopyParts) & 1;
        const SetInfo &S = sets[sc_set[j]];
        const int64_t ho = hull_offsets[sc_set[j]];
        const uint32_t l0 = off[0][S.sc_base], u0 = off[1][S.sc_base];
        copy_chain_part(P, side, j, (int)(it % kCopyParts), off[side][j] - (side ? u0 : l0),
                        off[0][S.sc_base + S.nsc] - l0, off[1][S.sc_base + S.nsc] - u0, hull_idx + ho,
                        S.pt_begin + S.n - ho);
    }
}

// Few survivors (at most kSmallHull): one block sorts them by (x, y, index)
// -- a bitonic network with one point per thread, exchanged by shuffles
// within a warp -- drops repeated points (the first, of the lowest index,
// stays), and two warps run the strict-turn elimination passes of the chain
// kernel, one per side, until nothing changes: a sequence with only strict
// turns is its own monotone chain.  The later sort and chain kernels then
// stop at once.  More survivors: it does nothing.
// Bound by latency.  One thread's sequential chain took 60 of this kernel's
// 67 us on the 69 survivors of 10^8 normal points (three dependent shared
// loads and an orientation per step); the passes look at every point at
// once and there are few of them.
constexpr int kSmallHull = 512;

struct SmallSmem {
    unsigned long long sk[kSmallHull];   // ord(x) << 32 | ord(y)
    uint32_t si[kSmallHull];             // point index
    float2 pt[kSmallHull];
    uint16_t list[2][2][kSmallHull];     // per side: the sequence and the pass's output
    uint32_t wsum[kSmallHull / 32];
    int len[2], cur[2];
};

__global__ void __launch_bounds__(kSmallHull) small_hull_kernel(void *ws, Layout L, uint32_t *hull_idx,
                                                                uint32_t *hull_count)
{
    kernel_entry();
    __shared__ SmallSmem sm;
    Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
    const Octagon *oct = at<Octagon>(ws, L.oct);
    const uint32_t s = hull_stage_count(ctrl, oct);
    if (s == 0 && threadIdx.x == 0) *hull_count = 0u;   // (no later kernel may follow)
    if (s == 0 || s > (uint32_t)kSmallHull) return;
    const uint32_t t = threadIdx.x, lane = lane_id(), warp = t >> 5, lt = (1u << lane) - 1u;
    unsigned long long k = ~0ull;   // after every point
    uint32_t ix = ~0u;
    if (t < s) {
        const unsigned long long pv = at<unsigned long long>(ws, L.pay[ctrl->sort_in])[t];
        k = ((unsigned long long)at<uint32_t>(ws, L.keys[ctrl->sort_in])[t] << 32) | (pv >> 32);
        ix = (uint32_t)pv;
    }
    uint32_t m = 32;
    while (m < s) m <<= 1;
    for (uint32_t g = 2; g <= m; g <<= 1) {
        for (uint32_t j = g >> 1; j > 0; j >>= 1) {
            unsigned long long ok;
            uint32_t oi;
            if (j >= 32) {
                sm.sk[t] = k;
                sm.si[t] = ix;
                __syncthreads();
                ok = sm.sk[t ^ j];
                oi = sm.si[t ^ j];
                __syncthreads();
            } else {
                ok = __shfl_xor_sync(0xffffffffu, k, j);
                oi = __shfl_xor_sync(0xffffffffu, ix, j);
            }
            const bool less = k < ok || (k == ok && ix < oi);   // (padding entries are equal: either order)
            if (less != (((t & g) == 0) == ((t & j) == 0))) {
                k = ok;
                ix = oi;
            }
        }
    }
    sm.sk[t] = k;
    __syncthreads();
    // equal points: the first stays
    const bool first = t < s && (t == 0 || sm.sk[t - 1] != k);
    const uint32_t bal = __ballot_sync(0xffffffffu, first);
    if (lane == 0) sm.wsum[warp] = __popc(bal);
    __syncthreads();
    uint32_t before = 0, u = 0;
#pragma unroll
    for (int w = 0; w < kSmallHull / 32; ++w) {
        if (w < (int)warp) before += sm.wsum[w];
        u += sm.wsum[w];
    }
    if (first) {
        const uint32_t p = before + __popc(bal & lt);
        sm.pt[p] = key_point(k);
        sm.si[p] = ix;
        sm.list[0][0][p] = sm.list[1][0][p] = (uint16_t)p;
    }
    __syncthreads();
    if (warp < 2) {
        int len = (int)u, cur = 0;
        while (len > 2) {   // each pass but the last drops a point
            const int kept = warp_elim_pass(sm.pt, sm.list[warp][cur], sm.list[warp][cur ^ 1], len, (int)warp,
                                            (int)lane, lt);
            cur ^= 1;
            if (kept == len) break;
            len = kept;
        }
        if (lane == 0) {
            sm.len[warp] = len;
            sm.cur[warp] = cur;
        }
    }
    __syncthreads();
    const uint32_t hl = (uint32_t)sm.len[0], hu = (uint32_t)sm.len[1], mid = hu >= 2 ? hu - 2 : 0;
    if (t < hl) hull_idx[t] = sm.si[sm.list[0][sm.cur[0]][t]];
    if (t < mid) hull_idx[hl + t] = sm.si[sm.list[1][sm.cur[1]][hu - 2 - t]];
    if (t == 0) {
        *hull_count = hl + mid;
        ctrl->small_done = 1u;
    }
}

}  // namespace

static cudaError_t launch_small_hull(void *ws, const Layout &L, uint32_t *hull_idx, uint32_t *hull_count, cudaStream_t st)
{
    probe_before(CH_K_CHAIN, st);
    launch_next(small_hull_kernel, 1, kSmallHull, 0, st, ws, L, hull_idx, hull_count);
    note_kernels(CH_K_CHAIN, 1);
    probe_after(CH_K_CHAIN, st);
    return cudaGetLastError();
}

static cudaError_t launch_chain(void *ws, const Layout &L, uint32_t *hull_idx, uint32_t *hull_count, cudaStream_t st)
{
    const int sms = sm_count();
    int64_t cb = L.n_chunks;
    static const int per_sm = [] {   // thread-safe one-time initialisation
        cudaFuncSetAttribute(chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ChainSmem<kOneThreads>));
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, chain_kernel, kOneThreads, sizeof(ChainSmem<kOneThreads>));
        return v > 0 ? v : 1;
    }();
    if (cb > (int64_t)sms * per_sm) cb = (int64_t)sms * per_sm;
    if (cb < 1) cb = 1;
    probe_before(CH_K_CHAIN, st);
    launch_next(chain_kernel, (unsigned)cb, kOneThreads, sizeof(ChainSmem<kOneThreads>), st, ws, L, hull_idx, hull_count);
    if (L.n <= SC) {   // one super-chunk at most: that kernel wrote the hull
        note_kernels(CH_K_CHAIN, 1);
        probe_after(CH_K_CHAIN, st);
        return cudaGetLastError();
    }
    launch_next(chain_merge_kernel, merge_grid(L.n_chunks), kMergeThreads, 0, st, ws, L);
    note_kernels(CH_K_CHAIN, 2);
    probe_after(CH_K_CHAIN, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (L.n_chunks > kEmitThreads) {
        const int64_t eb = std::min<int64_t>(L.emit_tiles, (int64_t)sms * 4);
        probe_before(CH_K_EMIT, st);
        launch_next(emit_kernel, (unsigned)eb, kEmitThreads, 0, st, ws, L);
        note_kernels(CH_K_EMIT, 1);
        probe_after(CH_K_EMIT, st);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    const int64_t fb = std::min<int64_t>(ceil_div(L.n_chunks * 2 * kCopyParts, kEmitThreads / 32), (int64_t)sms * 4);
    probe_before(CH_K_FINISH, st);
    launch_next(hull_copy_kernel, (unsigned)fb, kEmitThreads, 0, st, ws, L, hull_idx, hull_count);
    note_kernels(CH_K_FINISH, 1);
    probe_after(CH_K_FINISH, st);
    return cudaGetLastError();
}

// The hull of the survivors.  Few points need few of the kernels: each idle
// launch is more than 1 us (1000 points: 31 us with all of them, 20 without).
cudaError_t launch_hull_stage(void *ws, const Layout &L, uint32_t *hull_idx, uint32_t *hull_count, cudaStream_t st)
{
    cudaError_t e = launch_small_hull(ws, L, hull_idx, hull_count, st);
    if (e == cudaSuccess && L.n > SC) e = launch_sort(ws, L, st);
    if (e == cudaSuccess && L.n > kSmallHull) e = launch_chain(ws, L, hull_idx, hull_count, st);
    return e;
}

cudaError_t launch_bx_chain(void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st)
{
    const int sms = sm_count();
    static const int per_sm = [] {   // thread-safe one-time initialisation
        cudaFuncSetAttribute(bx_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(ChainSmem<kBxThreads>));
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, bx_chain_kernel, kBxThreads, sizeof(ChainSmem<kBxThreads>));
        return v > 0 ? v : 1;
    }();
    int64_t cb = BL.tiles_max;
    if (cb > (int64_t)sms * per_sm) cb = (int64_t)sms * per_sm;
    if (cb < 1) cb = 1;
    probe_before(CH_K_CHAIN, st);
    launch_next(bx_chain_kernel, (unsigned)cb, kBxThreads, sizeof(ChainSmem<kBxThreads>), st, ws, L, BL);
    launch_next(bx_merge_kernel, merge_grid(BL.tiles_max), kMergeThreads, 0, st, ws, L, BL);
    note_kernels(CH_K_CHAIN, 2);
    probe_after(CH_K_CHAIN, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int64_t eb = ceil_div(BL.tiles_max, kEmitThreads);
    const int emit_per_sm = tune_value(CH_TUNE_BX_EMIT) ? tune_value(CH_TUNE_BX_EMIT) : 4;
    if (eb > (int64_t)sms * emit_per_sm) eb = (int64_t)sms * emit_per_sm;
    if (eb < 1) eb = 1;
    probe_before(CH_K_EMIT, st);
    launch_next(bx_emit_kernel, (unsigned)eb, kEmitThreads, 0, st, ws, L, BL);
    note_kernels(CH_K_EMIT, 1);
    probe_after(CH_K_EMIT, st);
    return cudaGetLastError();
}

cudaError_t launch_bx_assemble(void *ws, const Layout &L, const BatchLayout &BL, const int64_t *hull_offsets,
                               uint32_t *hull_idx, cudaStream_t st)
{
    const int64_t blocks =
        std::min<int64_t>(ceil_div(BL.tiles_max * 2 * kCopyParts, kEmitThreads / 32), (int64_t)sm_count() * 8);
    launch_next(bx_assemble_kernel, (unsigned)blocks, kEmitThreads, 0, st, ws, L, BL, hull_offsets, hull_idx);
    return cudaGetLastError();
}

}  // namespace ch
