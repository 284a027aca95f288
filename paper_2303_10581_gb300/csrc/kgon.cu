// kgon.cu -- the hull step's filter: the octagon test of Sec. 3.2 and a
// second throw-away test against a fan of triangles around an interior
// point, in one pass that writes the survivors of both.
//
// The octagon filter (Sec. 3.1-3.2) removes almost nothing from points near
// a circle, and on a displaced circle 95 % survive it, although the hulls
// have a small fraction of the points as vertices.  The hull step repeats
// the throw-away idea of Sec. 3.1 on a much finer scale.  Let c be the
// centre of the bounding box.  The plane around c is cut into kFanBins
// angular bins (a pseudo-angle, fan.cuh).  The vertex of a bin is the input
// point farthest from c among a sample (the octagon survivors of about
// kFanBinTiles evenly spaced 4096-point tiles of the input), or, where that
// lies well inside the chord of samples to either side of the bin, a point on
// that chord, rounded a little inwards; a bin with neither repeats the vertex
// before it.  Every vertex is a point of the hull.
//
// The test of a point p in bin b, with P, Q, N the vertices of the bins
// b - 1, b, b + 1: if p is proven strictly after Q (left of c -> Q) and
// strictly left of Q -> N, or strictly before Q and strictly left of P -> Q,
// it is dropped.  Signs are proven in binary32 (proven_sign).  Then p lies
// strictly inside the hull:
//  - the pseudo-angle grows with the angle, and its binary32 value is off by
//    less than 0.0049 bins (0.0386 with the second level's eight times as
//    many): in units of eps = 2^-24, t = dy / (|dx| + |dy|) gets 7 |t| (two
//    differences, the sum, at most 2 ulp for the quotient); the scaling is
//    one FMA, which rounds by at most half an ulp of NB, or down to the
//    bin.  A vertex is taken only where its value is at least a margin (1/32;
//    1/8) away from both ends of its bin, so as directions P comes strictly
//    before p and N strictly after it (or N == Q, whose sign is never proven);
//  - consecutive vertices v, w were proven strictly counter-clockwise around
//    c (v != w), less than half a turn apart, so p is in the wedge of (Q, N)
//    or of (P, Q), where strictly left of the edge is the triangle (c, Q, N)
//    or (c, P, Q).  When all of them were, the triangles wind around c once,
//    so c and the triangles' interiors are in the interior of a polygon of
//    hull points.  Where a pair is not proven (a gap of half a turn, seen from
//    c: a cloud with far outliers that no sample met), its first vertex is
//    taken out (NaN, with which nothing is proven), so that only the points of
//    that wedge are kept; then c itself must lie clearly inside the octagon,
//    whose vertices are input points, for the other triangles to lie in the
//    hull, and there is no disk.  (One gap switching the fan off: 10^8 points
//    of a displaced circle and one at ten radii, 49 M of them sorted, 5146 us;
//    131 thousand and 2140 us when each wedge stood alone.);
//  - all of this is done on points times a power of two that brings the set's
//    box near size 1 where it is far from it (fan_space, Octagon::scale), so
//    that nothing overflows; a coordinate moves by 2^-150 at most, which the
//    2^-140 in the signs' bounds covers (points, vertices and c within 2^-148
//    of where they are, in a box of size at most 2^22);
//  - the quotient needs |dx| + |dy| of at least 2^-126: a point closer to c is
//    inside the disk around c that is proven inside the fan (without gaps the
//    fan is off unless its radius exceeds 2^-60) or inside the octagon.
// Nothing else is exact: a sign that is not proven keeps the point, and what
// is kept only costs the sort time.
//
// The disk around c proven inside the fan (a lower bound on the distance
// from c to every fan edge) lets most points of a displaced circle pass
// with one compare.
//
//  fan_bins_kernel    per bin, the farthest sampled octagon survivor
//                     (atomicMax of (far_key << 32 | ~index) into global
//                     slots), and how many of the sample survived
//  fan_vertex_kernel  whether there is a fan; the bins' vertices
//  fan_build_kernel   empty bins filled; the proofs that need consecutive
//                     vertices; the disk
//  hull_filter_kernel both tests of every point; the survivors' sort keys and
//                     payloads, in no particular order (the chain breaks
//                     ties by the index in the payload)
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "fan.cuh"
#include "launch.h"
#include "octtest.cuh"

namespace ch {
namespace {

constexpr int CT = 768;                  // threads per block of the filter pass: groups
constexpr int CG = CT / kFiltThreads;    // groups of kFiltThreads, each with its own tiles
constexpr int kFanTable = (kFanBins + 4) * 8;  // vertices, the last two again before them and the first two after them
constexpr int kQueue = 64;                     // points a warp of the filter pass queues (under 32, and 32 more)
constexpr uint32_t kMany = 128;                // a warp's survivors of a tile that go straight to the list
constexpr int kQueueSmem = CT / 32 * kQueue * 4;
using Level1 = FixedBins<kFanBins>;
using Level2 = FixedBins<kFan2Bins>;
constexpr float kFanMargin = 1.0f / 32.0f;     // of a vertex's pseudo-angle from its bin's ends
constexpr float kFan2Margin = 1.0f / 8.0f;     // second level
static_assert(kFiltItems == 16 && CT % kFiltThreads == 0, "16 items per filter thread");
static_assert(kQueueSmem % 16 == 0 && kFanTable + kQueueSmem <= 227 * 1024 - 1024, "table and queues fit a block's shared memory");

// det = (a - c) x (b - c) from the rounded differences, and a bound: a det
// beyond it in magnitude has the exact sign.  Shewchuk's orient2d error
// (orient_f32) is below 2^-22 (|l| + |r|) with l, r the products; |r| <= |l| +
// |det|, so |det| > 2^-20 |l| implies |det| > 2^-22 (|l| + |r|) (2^-140 for
// products that underflow; fan_space rules out overflow).
__device__ __forceinline__ float det_bound(float2 ac, float2 bc, float &bound)
{
    const float l = __fmul_rn(ac.x, bc.y), r = __fmul_rn(ac.y, bc.x);
    bound = __fmaf_ru(fabsf(l), 0x1p-20f, 0x1p-140f);
    return __fsub_rn(l, r);
}

// The vertices in shared memory, at their bins' biased indices.
struct SharedFan {
    uint32_t base;
    __device__ __forceinline__ explicit SharedFan(const float2 *V)
        : base((uint32_t)__cvta_generic_to_shared(V) - kBinBias * 8u)
    {
    }
    __device__ __forceinline__ uint32_t at(uint32_t biased) const { return base + biased * 8u; }
    __device__ __forceinline__ float2 get(uint32_t a, int d) const   // the vertex d entries on
    {
        float2 v;
        asm("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a + (uint32_t)(8 * d)));
        return v;
    }
};

// The same in global memory.
struct GlobalFan {
    const float2 *V;
    __device__ __forceinline__ const float2 *at(uint32_t biased) const { return V + (int)(biased - kBinBias); }   // (may be -1)
    __device__ __forceinline__ float2 get(const float2 *a, int d) const { return __ldg(a + d); }
};

// Strictly inside the fan, proven (see the top of the file).  F: the
// vertices; before the first come the last two, after the last the first two
// again; d = fl(p - c).  Two vertices are read: in shared memory the reads of
// 32 random bins conflict (six wavefronts each), and a third would bound the
// pass.
template <class Bins, class Fan>
__device__ __forceinline__ bool fan_inside(Bins nb, const Fan &F, float2 c, float2 d, float2 p)
{
    const auto a = F.at(fan_bin_biased(nb, d.x, d.y));   // (a NaN: any vertex; such a point is next to c)
    const float2 Q = F.get(a, 0);
    float e1, e2;
    const float side = det_bound(sub2(Q, c), d, e1);
    const float2 W = F.get(a, side > 0.0f ? 1 : -1);
    const float det = det_bound(sub2(W, Q), sub2(p, Q), e2);
    const float turned = __uint_as_float(__float_as_uint(det) ^ (__float_as_uint(side) & 0x80000000u));
    return (fabsf(side) > e1) & (turned > e2);   // (no branches: the points of a thread interleave)
}

// The bin a point may be the vertex of, -1 when its pseudo-angle is within
// `margin` of the bin's ends (or undefined).
template <class Bins>
__device__ __forceinline__ int vertex_bin(Bins nb, float dx, float dy, float margin)
{
    const float phi = fan_phi(nb, dx, dy);
    const float f = __fadd_rd(phi, 0x1p23f);   // 2^23 + the bin
    const float mid = phi - (f - 0x1p23f) - 0.5f;
    return fabsf(mid) <= 0.5f - margin ? (int)(__float_as_uint(f) - kBinBias) : -1;
}

// c clearly inside the octagon: every edge's affine form at c (its constant)
// is at least 2 where 1 proves it (octtest.cuh), so that the points next to c
// are inside too.
__device__ __forceinline__ bool centre_inside(const Octagon &o)
{
    bool in = true;
#pragma unroll
    for (int k = 0; k < 8; ++k) in &= o.tz[k] >= 2.0f;
    return in;
}

// Whether a fan's proofs hold: its consecutive vertex pairs v != w that are
// proven (edges), whether some are not (gaps), a lower bound on its radius (no gaps) or c
// inside the octagon.
__device__ __forceinline__ bool fan_holds(uint32_t edges, bool gaps, float rho2, bool centre)
{
    return gaps ? edges >= 1u && centre : edges >= 3u && rho2 > 0x1p-120f;
}

// Whether this call has a fan whose proofs hold (after fan_build_kernel).
__device__ __forceinline__ float fan_rho2(const KgonCtrl *kc) { return __uint_as_float(~kc->rho_inv); }
__device__ __forceinline__ bool fan_ready(const KgonCtrl *kc, const Kgon *g)
{
    return g->ok && fan_holds(kc->edges, kc->gaps != 0u, fan_rho2(kc), g->centre != 0u);
}

// ---------------------------------------------------------------------------
// first level: bins and vertices
// ---------------------------------------------------------------------------
constexpr int BI = 4;   // points per thread and step of the bins passes

// The bins' slots raised by a thread's points (live: those that count;
// index(k): point k's index).  A point whose binary32 distance is clearly below
// its slot's needs no exact key.
template <class Bins, class Index>
__device__ __forceinline__ void raise_bins(Bins nb, unsigned long long *slot, const float (&qx)[BI], const float (&qy)[BI],
                                           uint32_t live, float2 c, float r2ref, Index index)
{
    uint32_t top[BI];   // the slots' keys (most points do not raise their bin's)
    int b[BI];
#pragma unroll
    for (int k = 0; k < BI; ++k) {
        b[k] = vertex_bin(nb, __fsub_rn(qx[k], c.x), __fsub_rn(qy[k], c.y), kFanMargin);
        top[k] = 0u;
        if (!((live >> k) & 1u)) b[k] = -1;
        if (b[k] >= 0) top[k] = __ldcg(reinterpret_cast<const uint32_t *>(slot + b[k]) + 1);
    }
#pragma unroll
    for (int k = 0; k < BI; ++k) {
        const float dx = __fsub_rn(qx[k], c.x), dy = __fsub_rn(qy[k], c.y);
        const float r2 = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
        // (an empty slot's key is a NaN: not below)
        if (b[k] >= 0 && !(r2 - r2ref < __fmaf_rn(r2, -0x1p-20f, key_float(top[k])))) {
            const uint32_t key = far_key(qx[k], qy[k], c.x, c.y, r2ref);
            if (key >= top[k]) atomicMax(slot + b[k], ((unsigned long long)key << 32) | (uint32_t)~index(k));
        }
    }
}

__device__ __forceinline__ void to_fan_space(float (&qx)[BI], float (&qy)[BI], float scale)
{
    if (scale == 1.0f) return;   // uniform
#pragma unroll
    for (int k = 0; k < BI; ++k) {
        qx[k] = __fmul_rn(qx[k], scale);
        qy[k] = __fmul_rn(qy[k], scale);
    }
}

// The octagon's vertices raise the bins as well (a warp calls; index(k):
// vertex k's): far points in tiles that are not sampled are among them.
template <class Bins, class Index>
__device__ __forceinline__ void raise_octagon(Bins nb, unsigned long long *slot, const Octagon &o, Index index)
{
    const int first = (int)(lane_id() & 1u) * BI;
    static_assert(2 * BI == 8, "two lanes hold the eight vertices");
    float qx[BI], qy[BI];
#pragma unroll
    for (int k = 0; k < BI; ++k) {
        const float2 v = fan_space(make_float2(o.ax[first + k], o.ay[first + k]), o.scale);
        qx[k] = v.x;
        qy[k] = v.y;
    }
    raise_bins(nb, slot, qx, qy, lane_id() < 2u ? (1u << BI) - 1u : 0u, fan_centre(o), far_ref(o),
               [&](int k) { return index(first + k); });
}

// Every stride-th tile, in quarters (1024 points, four a thread) over a
// persistent grid: the bins' farthest points among the octagon's survivors,
// and how many of the first quarters' points survive it (of all quarters'
// points: the blocks' sums meet at two words, 6 us more on 10^6 circle
// points).  Bound by the latency of the points'
// and then the slots' reads, so the next quarter's points are read while this
// one is binned, and few registers keep five blocks on an SM.  The rectangle
// settles nearly every point of a normal cloud, the octagon's forms those of
// clouds at the ends of their box: seen from its centre in a small angle,
// they meet in few bins, whose slots then bound the pass (3 10^6 points of two
// clusters 266 us the hull, of a Cauchy cloud 229, with the rectangle alone;
// 120 and 61 so).
template <int G>
__global__ void __launch_bounds__(kFiltThreads, 5) fan_bins_kernel(const float *__restrict__ pts, uint32_t n, void *ws,
                                                                   Layout L, uint32_t stride, int use_bits,
                                                                   const int32_t *kdev)
{
    kernel_entry();
    __shared__ OctSmem so;
    const Octagon *oct = at<Octagon>(ws, L.oct);
    if (oct->abort || oct->spec || !oct->has_edges) return;
    fill_octagon(so, oct);
    __syncthreads();
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    const bool bits_mode = use_bits && (!kdev || *kdev != 8);
    const float r2ref = far_ref(so);
    const float2 c = fan_centre(so);
    const uint32_t t = threadIdx.x;
    constexpr uint32_t parts = kFiltItems / BI;
    const uint32_t ntiles = (n + kFiltTile - 1) / kFiltTile, steps = (ntiles + stride - 1) / stride * parts;
    uint32_t seen = 0, kept = 0;   // (n < 2^30)
    float px[BI], py[BI];
    uint32_t live = 0;
    const auto fetch = [&](uint32_t w) {
        const uint32_t base = w / parts * stride * kFiltTile;
        const int part = (int)(w % parts);
        if (base + kFiltTile <= n) {
            load_part<G, BI>(pts, base, t, part, px, py);
            live = (1u << BI) - 1u;
        } else {
            live = load_part_ragged<G, BI>(pts, n, base, t, part, so.cx, so.cy, px, py);
        }
    };
    if (blockIdx.x < steps) fetch(blockIdx.x);
    if (blockIdx.x == gridDim.x - 1 && t < 32u) {
        const uint32_t *ext8 = at<uint32_t>(ws, L.ext8);
        raise_octagon(Level1{}, kc->slot, so, [&](int k) { return ext8[k]; });
    }
    for (uint32_t w = blockIdx.x; w < steps; w += gridDim.x) {
        const uint32_t tile = w / parts * stride, part = w % parts;
        float qx[BI], qy[BI];
        uint32_t mine = live;
#pragma unroll
        for (int k = 0; k < BI; ++k) {
            qx[k] = px[k];
            qy[k] = py[k];
        }
        if (w + gridDim.x < steps) fetch(w + gridDim.x);
        const bool counts = part == 0u || bits_mode;
        if (counts) seen += __popc(mine);
        if (bits_mode) {
            mine &= (uint32_t)at<uint16_t>(ws, L.keep_bits)[tile * kFiltThreads + t] >> (BI * part);
        } else {
#pragma unroll
            for (int k = 0; k < BI; ++k)
                if ((qx[k] >= so.xl) & (qx[k] <= so.xh) & (qy[k] >= so.yl) & (qy[k] <= so.yh)) mine &= ~(1u << k);
            if (!__any_sync(0xffffffffu, mine != 0u)) continue;
            uint32_t out;
            oct_decide<BI>(so, qx, qy, out);   // (undecided points count)
            mine &= out;
        }
        if (counts) kept += __popc(mine);
        if (!__any_sync(0xffffffffu, mine != 0u)) continue;
        to_fan_space(qx, qy, so.scale);
        raise_bins(Level1{}, kc->slot, qx, qy, mine, c, r2ref, [&](int k) {
            return (uint32_t)item_point<G>(tile * kFiltTile, t, (int)(BI * part) + k);
        });
    }
    seen = __reduce_add_sync(0xffffffffu, seen);
    kept = __reduce_add_sync(0xffffffffu, kept);
    if (lane_id() == 0 && seen) {
        atomicAdd(&kc->sample, seen);
        if (kept) atomicAdd(&kc->inside, kept);
    }
}

// One thread per bin (kFanBins / BT blocks).  An empty bin repeats the last
// vertex before it, cyclically: a max-scan of the bins that have one inside
// the block, and for the bins before the block's first, the last one of the
// nearest earlier range of BT bins that has one (searched range by range).
constexpr int BT = 1024;
static_assert(kFanBins % BT == 0, "bins split evenly over the blocks");

__device__ __forceinline__ int block_max(int v, int *s_w)
{
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();   // s_w may still be read from an earlier call
    if (lane_id() == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    return __reduce_max_sync(0xffffffffu, s_w[lane_id()]);   // (32 warps)
}

// The last bin with a vertex of its own at or before bin blockIdx.x * BT +
// threadIdx.x, cyclically (-1: no bin has one; block-uniform then).  Every
// thread of the block calls; has(j): bin j has one.
template <class Has>
__device__ __forceinline__ int vertex_source(Has has, int *s_w, int *s_scan)
{
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const int b = (int)(blockIdx.x * BT + tid);
    int incl = has(b) ? b : -1;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl = max(incl, u);
    }
    if (lane == 31) s_scan[warp] = incl;
    __syncthreads();
    incl = max(incl, __reduce_max_sync(0xffffffffu, lane < warp ? s_scan[lane] : -1));   // (32 warps)
    if (!__syncthreads_or(incl < 0)) return incl;
    int prev = -1;
    for (uint32_t k = 1; k <= gridDim.x && prev < 0; ++k) {   // prev is block-uniform
        const uint32_t rb = (blockIdx.x + gridDim.x - k) % gridDim.x;
        const int j = (int)(rb * BT + tid);
        prev = block_max(has(j) ? j : -1, s_w);
    }
    return prev < 0 ? -1 : (incl >= 0 ? incl : prev);
}

// Lower bound on the squared distance from c to the segment [v, w] (v != w),
// or -1 when (c, v, w) is not proven strictly counter-clockwise.  The
// distance is the one to the nearer end when the foot of the perpendicular
// provably falls outside the segment, else at least the one to the line.
// T: the arithmetic; its rounding (half an ulp) is U.  Sums of two products
// lose at most 4 U of the sum of their magnitudes, squares and the quotient
// 16 U.
template <class T>
__device__ __forceinline__ T edge_bound(float cx, float cy, float2 v, float2 w, T U)
{
    const T ux = (T)cx - (T)v.x, uy = (T)cy - (T)v.y;   // c - v
    const T dv = (ux * ux + uy * uy) * ((T)1 - (T)16 * U);
    const T ex = (T)w.x - (T)v.x, ey = (T)w.y - (T)v.y;   // w - v
    const T t1 = ex * uy, t2 = ey * ux;
    const T lo = (t1 - t2) - (fabs(t1) + fabs(t2)) * ((T)8 * U);   // c strictly left of v -> w
    if (!(lo > (T)0)) return (T)-1;
    const T len2 = ex * ex + ey * ey;
    const T d1 = ex * ux, d2 = ey * uy;
    const T dot = d1 + d2, derr = (fabs(d1) + fabs(d2)) * ((T)8 * U);   // (c - v) . (w - v)
    if (dot < -derr) return dv;   // the foot lies before v
    if (dot > len2 * ((T)1 + (T)16 * U) + derr) {   // after w
        const T zx = (T)cx - (T)w.x, zy = (T)cy - (T)w.y;
        return (zx * zx + zy * zy) * ((T)1 - (T)16 * U);
    }
    return lo * lo / (len2 * ((T)1 + (T)16 * U)) * ((T)1 - (T)16 * U);
}

// In binary32 first (27648 binary64 quotients on 27 SMs would take 15 us),
// in binary64 where that proves nothing: a value in binary32, rounded down.
__device__ __forceinline__ float disk_bound(float cx, float cy, float2 v, float2 w)
{
    const float f = edge_bound<float>(cx, cy, v, w, 0x1p-24f);
    if (f >= 0x1p-100f && f <= 0x1p100f) return f;
    const double d = edge_bound<double>(cx, cy, v, w, 0x1p-53);
    return d < 0.0 ? -1.0f : (d <= 3.0e38 ? __double2float_rd(d) : 3.0e38f);
}

__device__ __forceinline__ bool fan_live(const KgonCtrl *kc, int64_t n)
{
    // (an aborted call, the speculative sweep's candidates, a polygon without
    // edges: the bins pass left no sample)
    const uint32_t sample = kc->sample;
    return sample != 0u && (double)kc->inside / sample * (double)n >= (double)kKgonMinS;
}

// The vertices of 64 consecutive bins, a warp: the samples of the bins and of
// the nearest non-empty bins to either side, then strict-turn elimination
// passes leave their (nearly) convex chain.  A bin whose sample was
// eliminated and lies more than 2^-18 inside the chord over it, or that has
// none, gets the point of the chord in the direction of its middle, moved
// inwards by 2^-20 and rounded; it is used only when it is proven inside the
// triangle of c and the chord's ends (exact signs, its bin's margins), hence
// in the hull.  On a displaced circle with few samples per bin the farthest
// sample of a bin lies deep: of 10^8 points 338428 reached the sort with the
// samples alone, and the disk around c missed a fourteenth of the points.
constexpr int VB = 64;                   // bins per warp
constexpr int VT = 256;                  // threads per block
constexpr int kVertexPasses = 16;
static_assert(kFanBins % (VB * VT / 32) == 0, "bins split evenly over the warps");

struct VertexSmem {
    float2 p[2][VB + 2];
    int bin[2][VB + 2];                  // unwrapped: below 0 / beyond NB across the ends
};

// The nearest non-empty bin before `from` (dir = -1) or from `from` on (dir =
// 1), unwrapped, among `reach` of them (a multiple of 32); kNoBin when there is
// none.  The first 32 nearly always hold one; of the others four times 32 are
// read at once.
constexpr int kNoBin = INT_MIN;

__device__ __forceinline__ int nearest_bin(int NB, const unsigned long long *slot, int from, int dir, int reach)
{
    const int lane = (int)lane_id();
    const auto filled = [&](int k) {   // of the 32 bins after the first k
        const int j = dir > 0 ? from + k + lane : from - 1 - k - lane;
        const int w = j < 0 ? j + NB : (j >= NB ? j - NB : j);
        return k < reach && __ldcg(slot + w) != 0ull;
    };
    const auto place = [&](int k, uint32_t m) { return dir > 0 ? from + k + __ffs(m) - 1 : from - k - __ffs(m); };
    const uint32_t m0 = __ballot_sync(0xffffffffu, filled(0));
    if (m0) return place(0, m0);
    for (int k = 32; k < reach; k += 128) {
        bool f[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) f[u] = filled(k + 32 * u);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const uint32_t m = __ballot_sync(0xffffffffu, f[u]);
            if (m) return place(k + 32 * u, m);
        }
    }
    return kNoBin;
}

// Bins [b0, b0 + VB) of a fan; point(i) reads input point i
// (clamped to the input); V receives the vertices, x = NaN for none.  The
// neighbours of the range are looked for within an eighth of the turn and 288
// bins: a chord over more empty bins adds nothing that the wedge over them
// does not have, and walking the empty bins of a set that is seen from its
// centre in a small angle (an arc, far outliers, a line) 32 at a time took
// 117 to 362 us.
template <class Bins, class Point>
__device__ __forceinline__ void make_vertices(Bins nb, VertexSmem &sm, const unsigned long long *slot, int b0, float2 c,
                                              Point point, float2 *V)
{
    const int NB = (int)nb.count();
    const int lane = (int)lane_id();
    const uint32_t lt = (1u << lane) - 1u;
    const int reach = min(288, NB / 8 & ~31);
    const int before = nearest_bin(NB, slot, b0, -1, reach), after = nearest_bin(NB, slot, b0 + VB, 1, reach);
    const int head = before != kNoBin ? 1 : 0;
    bool has[VB / 32];
    float2 own[VB / 32];
    int len = head;
#pragma unroll
    for (int h = 0; h < VB / 32; ++h) {
        const unsigned long long v = __ldcg(slot + b0 + 32 * h + lane);
        has[h] = v != 0ull;
        own[h] = has[h] ? point(~(uint32_t)v) : c;
        const uint32_t m = __ballot_sync(0xffffffffu, has[h]);
        if (has[h]) {
            sm.p[0][len + __popc(m & lt)] = own[h];
            sm.bin[0][len + __popc(m & lt)] = b0 + 32 * h + lane;
        }
        len += __popc(m);
    }
    if (lane < 2) {
        const int j = lane ? after : before;
        if (j != kNoBin) {
            const int w = j < 0 ? j + NB : (j >= NB ? j - NB : j);
            const int at = lane ? len : 0;
            sm.p[0][at] = point(~(uint32_t)__ldcg(slot + w));
            sm.bin[0][at] = j;
        }
    }
    len += after != kNoBin ? 1 : 0;
    __syncwarp();
    int cur = 0;
    for (int pass = 0; pass < kVertexPasses; ++pass) {
        int kept = 0;
        for (int i0 = 0; i0 < len; i0 += 32) {
            const int i = i0 + lane;
            bool keep = i < len;
            if (keep && i > 0 && i < len - 1) {
                const float2 a = sm.p[cur][i - 1], q = sm.p[cur][i], d = sm.p[cur][i + 1];
                keep = (a.x - q.x) * (d.y - q.y) - (a.y - q.y) * (d.x - q.x) < 0.0f;   // right of the chord
            }
            const uint32_t m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                sm.p[cur ^ 1][kept + __popc(m & lt)] = sm.p[cur][i];
                sm.bin[cur ^ 1][kept + __popc(m & lt)] = sm.bin[cur][i];
            }
            kept += __popc(m);
        }
        __syncwarp();
        cur ^= 1;
        const bool done = kept == len;
        len = kept;
        if (done) break;
    }
#pragma unroll
    for (int h = 0; h < VB / 32; ++h) {
        const int b = b0 + 32 * h + lane;
        int lo = -1, hi = len;   // the last entry at or before bin b (-1: none), the first after it (len: none)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (sm.bin[cur][mid] <= b) lo = mid;
            else hi = mid;
        }
        float2 v = own[h];
        bool ok = has[h];
        if (lo >= 0 && hi < len && sm.bin[cur][lo] != b) {
            const float2 Lp = sm.p[cur][lo], Rp = sm.p[cur][hi];
            const float lx = Lp.x - c.x, ly = Lp.y - c.y, ex = Rp.x - Lp.x, ey = Rp.y - Lp.y;
            const float num = lx * ey - ly * ex;
            const float own_den = (v.x - c.x) * ey - (v.y - c.y) * ex;
            if (!ok || num > own_den * (1.0f + 0x1p-18f)) {   // (own_den > 0: the sample is on the chord's side of c)
                const float2 d = fan_direction(nb, (float)b + 0.5f);
                const float s = num / (d.x * ey - d.y * ex) * (1.0f - 0x1p-20f);
                const float2 q = make_float2(__fmaf_rn(s, d.x, c.x), __fmaf_rn(s, d.y, c.y));
                if (fabsf(q.x) <= 3.0e38f && fabsf(q.y) <= 3.0e38f &&
                    vertex_bin(nb, __fsub_rn(q.x, c.x), __fsub_rn(q.y, c.y), kFanMargin) == b &&
                    orient(Lp.x, Lp.y, Rp.x, Rp.y, q.x, q.y) > 0 && orient(Lp.x, Lp.y, Rp.x, Rp.y, c.x, c.y) > 0) {
                    v = q;
                    ok = true;
                }
            }
        }
        V[b] = ok ? v : make_float2(__int_as_float(0x7fc00000), 0.0f);
    }
}

__global__ void __launch_bounds__(VT) fan_vertex_kernel(const float *__restrict__ pts, int64_t n, void *ws, Layout L)
{
    kernel_entry();
    __shared__ VertexSmem sm[VT / 32];
    const Octagon *oct = at<Octagon>(ws, L.oct);
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    if (!fan_live(kc, n)) return;
    const int warp = (int)(threadIdx.x >> 5);
    const int b0 = (int)(blockIdx.x * (VT / 32) + warp) * VB;
    make_vertices(
        Level1{}, sm[warp], kc->slot, b0, fan_centre(*oct),
        [&](uint32_t i) { return fan_space(input_point(pts, (int64_t)i < n ? i : 0u), oct->scale); },
        at<float2>(ws, L.pay[1]));
}

__global__ void __launch_bounds__(BT) fan_build_kernel(int64_t n, void *ws, Layout L)
{
    kernel_entry();
    __shared__ int s_w[BT / 32];
    __shared__ int s_scan[BT / 32];
    const Octagon *oct = at<Octagon>(ws, L.oct);
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    Kgon *g = at<Kgon>(ws, L.kgon);
    const float2 *raw = at<float2>(ws, L.pay[1]);
    const uint32_t tid = threadIdx.x;
    const bool live = fan_live(kc, n);
    const int b = (int)(blockIdx.x * BT + tid);
    int src = -1;
    if (live) src = vertex_source([&](int j) { return raw[j].x == raw[j].x; }, s_w, s_scan);   // block-uniform
    if (src < 0) {
        if (blockIdx.x == 0 && tid == 0) g->ok = 0u;
        return;
    }
    const float2 c = fan_centre(*oct);
    float2 v = raw[src];
    const float2 next = raw[b + 1 == kFanBins ? 0 : b + 1];
    // the next bin's vertex: its own point, or this one's again
    const float2 w = next.x == next.x ? next : v;
    float r = __int_as_float(0x7f800000);
    const bool edge = v.x != w.x || v.y != w.y;
    bool gap = false;
    if (edge) {
        r = disk_bound(c.x, c.y, v, w);
        gap = r < 0.0f;
        if (gap) v.x = __int_as_float(0x7fc00000);
    }
    g->v[b] = v;
    uint32_t inv = ~__float_as_uint(fmaxf(r, 0.0f));
    inv = __reduce_max_sync(0xffffffffu, inv);
    const uint32_t edges = __popc(__ballot_sync(0xffffffffu, edge && !gap));
    gap = __any_sync(0xffffffffu, gap);
    if (lane_id() == 0) {
        atomicMax(&kc->rho_inv, inv);
        if (edges) atomicAdd(&kc->edges, edges);
        if (gap) kc->gaps = 1u;
    }
    if (blockIdx.x == 0 && tid == 0) {
        g->cx = c.x;
        g->cy = c.y;
        g->ok = 1u;
        g->centre = centre_inside(*oct) ? 1u : 0u;
    }
}

// ---------------------------------------------------------------------------
// the filter pass
// ---------------------------------------------------------------------------
// Where survivors go: sort keys, payloads and their number.
struct Sink {
    uint32_t *count, *keys;
    unsigned long long *pay;
    __device__ __forceinline__ void put(uint32_t pos, float2 p, uint32_t i) const
    {
        keys[pos] = ord_key(p.x);
        pay[pos] = ((unsigned long long)ord_key(p.y) << 32) | i;
    }
};

// What a filter pass has in shared memory beside its queues and vertices.
struct FilterSmem {
    OctSmem so;
    Sink sink;
    uint32_t octs;
    uint32_t item;
};

// The warp's kept points (mask: this lane's items among N; get(q): the point
// and its index) to the end of the survivor list, item by item, so that the
// lanes' writes (and the points they read again) are neighbours.
template <int N, class Get>
__device__ __forceinline__ void append_survivors(uint32_t mask, uint32_t total, const Sink &sink, Get get)
{
    const uint32_t lt = (1u << lane_id()) - 1u;
    uint32_t pos = 0;
    if (lane_id() == 0) pos = atomicAdd(sink.count, total);
    pos = __shfl_sync(0xffffffffu, pos, 0);
#pragma unroll N > 4 ? 4 : N
    for (int q = 0; q < N; ++q) {
        const bool mine = (mask >> q) & 1u;
        const uint32_t m = __ballot_sync(0xffffffffu, mine);
        if (mine) {
            uint32_t i;
            const float2 p = get(q, i);
            sink.put(pos + __popc(m & lt), p, i);
        }
        pos += __popc(m);
    }
}

// The speculative sweep's candidates (extremes.cu; every other point is
// proven inside the octagon): a warp per slice, the exact test.
__device__ __forceinline__ uint32_t filter_candidates(const FilterSmem &fs, void *ws, const Layout &L)
{
    const SpecCtrl *sc = at<SpecCtrl>(ws, L.spec);
    const uint32_t *cidx = at<uint32_t>(ws, L.keys[1]);
    const float2 *cpt = at<float2>(ws, L.pay[1]);
    const uint32_t slices = sc->nseg * kSpecWarps, cap = sc->cap, lane = lane_id();
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    uint32_t mine = 0;
    for (uint32_t j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); j < slices; j += warps) {
        const uint32_t c = min(sc->scnt[j], cap);
        const size_t s0 = (size_t)j * cap;
        for (uint32_t e0 = 0; e0 < c; e0 += 32) {   // warp-uniform
            float2 p = make_float2(0.0f, 0.0f);
            bool keep = e0 + lane < c;
            if (keep) {
                p = cpt[s0 + e0 + lane];
                keep = keep_point<false>(fs.so, p.x, p.y);
            }
            mine += keep ? 1u : 0u;
            const uint32_t total = __popc(__ballot_sync(0xffffffffu, keep));
            if (total)
                append_survivors<1>(keep ? 1u : 0u, total, fs.sink, [&](int, uint32_t &i) {
                    i = cidx[s0 + e0 + lane];
                    return p;
                });
        }
    }
    return mine;
}

// A warp's queue of point indices (shared memory): survivors on their way to
// the list, or (candidates) points outside the disk that still need the fan
// test.  Full batches of 32 leave it, read their points again (L2) and do the
// fan test of scattered points and the list's atomics and writes as a whole
// warp.
struct PointQueue {
    uint32_t *i;
    uint32_t n;   // warp-uniform
};

// SCALED: the set's scale is not 1.  (A variant of its own: the loop is bound
// by issue.)
template <class Bins_, bool SCALED>
struct FanView {
    using Bins = Bins_;
    bool fan;       // there is one
    Bins nb;
    SharedFan F;
    float2 c;       // scaled
    float rho2t;    // r2 < rho2t proves |p - c| below the disk's radius
    bool disk;      // try the disk first
    float scale;
    __device__ __forceinline__ float2 space(float x, float y) const
    {
        if constexpr (SCALED) return fan_space(make_float2(x, y), scale);
        return make_float2(x, y);
    }
};

// An index with this bit (n < 2^30) is a point the octagon's forms may have
// left undecided: the exact test first, and then the fan test.
constexpr uint32_t kUnsettled = 0x80000000u;

// Whether point p (i: its index and kUnsettled) survives; octs counts the
// octagon survivors among the unsettled ones.  test: a candidate.
template <class View>
__device__ __forceinline__ bool settle(const OctSmem &so, const View &f, bool test, uint32_t i, float2 p,
                                       uint32_t &octs)
{
    bool keep = true;
    if (i & kUnsettled) {
        keep = keep_point<false>(so, p.x, p.y);
        octs += keep ? 1u : 0u;
    }
    if (test || ((i & kUnsettled) && f.fan)) {
        const float2 q = f.space(p.x, p.y);
        keep = keep && !fan_inside(f.nb, f.F, f.c, sub2(q, f.c), q);
    }
    return keep;
}

// The last (up to) 32 points of the queue: the survivors to the list.
template <class View>
__device__ __forceinline__ void queue_drain(PointQueue &q, const FilterSmem &fs, const View &f, bool test,
                                            const float *__restrict__ pts, uint32_t &octs)
{
    const uint32_t lane = lane_id(), m = min(q.n, 32u);
    q.n -= m;
    bool keep = lane < m;
    const uint32_t e = q.i[q.n + (keep ? lane : 0u)], i = e & ~kUnsettled;
    const float2 p = input_point(pts, i);
    __syncwarp();   // the slots may be filled again
    if (keep) keep = settle(fs.so, f, test, e, p, octs);
    const uint32_t b = __ballot_sync(0xffffffffu, keep);
    if (!b) return;
    uint32_t pos = 0;
    if (lane == 0) pos = atomicAdd(fs.sink.count, (uint32_t)__popc(b));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(b & ((1u << lane) - 1u));
    if (keep) fs.sink.put(pos, p, i);
}

// Tiles tile, tile + step, ... below t1 of the set pts (n points), by a group
// of kFiltThreads threads whose warps have queues of their own: a thread tests
// its 16 points of a tile eight at a time: the octagon's affine forms, then
// (fan) the fan test, branch-free -- or, in a warp where the disk holds most
// points, the disk test, the others going to the queue.  bits: a second
// polygon has refined the count pass's keep bits, which then stand for the
// octagon test.  octs counts the octagon survivors.
template <int G, class View>
__device__ __forceinline__ void filter_tiles(const FilterSmem &fs, const View &f, uint32_t *queue,
                                             const float *__restrict__ pts, uint32_t n, uint32_t tile, uint32_t t1,
                                             uint32_t step, const uint16_t *bits, uint32_t &octs)
{
    const uint32_t t = threadIdx.x % kFiltThreads, lt = (1u << lane_id()) - 1u;
    const bool edges = !bits && fs.so.has_edges;
    PointQueue q{queue, 0u};
    bool use_disk = f.fan && f.disk;   // (then the queue holds candidates)
    for (; tile < t1; tile += step) {
        const uint32_t base = tile * kFiltTile;
        if (t == 0 && tile + step < t1) {   // the next tile streams into L2 meanwhile
            const uint32_t nb = base + step * kFiltTile;
            const uintptr_t next = reinterpret_cast<uintptr_t>(pts + 2 * (size_t)nb);
            const uint32_t head = (uint32_t)(next & 8u);   // (a set may start 8 bytes past a 16-byte boundary)
            const uint32_t bytes = (min((uint32_t)kFiltTile, n - nb) * 8u - head) & ~15u;
            if (bytes) bulk_prefetch_l2(reinterpret_cast<const void *>(next + head), bytes);
        }
        // kept: octagon survivors; drop: those of them inside the disk or the
        // fan; near: some may be undecided, and all of this lane's are settled
        // when they leave the queue (rare: next to the octagon)
        uint32_t kept = 0xffffu, drop = 0;
        bool near = false;
        if (bits) kept = bits[tile * kFiltThreads + t];
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
            float px[8], py[8];
            if (base + kFiltTile <= n) load_part<G, 8>(pts, base, t, half, px, py);
            else kept &= ~(0xffu << (8 * half)) |
                         load_part_ragged<G, 8>(pts, n, base, t, half, fs.so.cx, fs.so.cy, px, py) << (8 * half);
            if (edges) {
                uint32_t out8;
                near |= oct_decide<8>(fs.so, px, py, out8);
                kept &= ~(0xffu << (8 * half)) | out8 << (8 * half);
            }
            if (!f.fan) continue;
            uint32_t in = 0;
            if (use_disk) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float2 p = f.space(px[k], py[k]);
                    const float dx = __fsub_rn(p.x, f.c.x), dy = __fsub_rn(p.y, f.c.y);
                    if (__fmaf_rn(dx, dx, __fmul_rn(dy, dy)) < f.rho2t) in |= 1u << k;
                }
            } else if (__any_sync(0xffffffffu, ((kept >> (8 * half)) & 0xffu) != 0u)) {
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    if (k % 4 == 0) asm volatile("" ::: "memory");   // four points at a time (more would spill)
                    const float2 p = f.space(px[k], py[k]);
                    if (fan_inside(f.nb, f.F, f.c, sub2(p, f.c), p)) in |= 1u << k;
                }
            }
            drop |= in << (8 * half);
        }
        uint32_t live = near ? kept : kept & ~drop;
        if (!near) octs += __popc(kept);
        const uint32_t total = __reduce_add_sync(0xffffffffu, __popc(live));
        if (use_disk) {   // a warp that finds under a quarter of a tile's points in the disk stops testing it
            const uint32_t tried = __reduce_add_sync(0xffffffffu, __popc(kept));
            if (4u * total > 3u * tried) {
                while (q.n) queue_drain(q, fs, f, true, pts, octs);
                if (!near) octs -= __popc(kept);
                use_disk = false;
                tile -= step;   // once more, with the fan
                continue;
            }
        }
        if (total == 0u) continue;
        if (total <= kMany) {
            // (a ballot per round: a lane has few points)
            uint32_t m;
            while ((m = __ballot_sync(0xffffffffu, live != 0u)) != 0u) {
                if (live)
                    q.i[q.n + __popc(m & lt)] = (uint32_t)item_point<G>(base, t, __ffs(live) - 1) | (near ? kUnsettled : 0u);
                live &= live - 1u;
                q.n += __popc(m);
                __syncwarp();
                if (q.n >= 32u) queue_drain(q, fs, f, use_disk, pts, octs);
            }
        } else {   // many at once: the points are read again
            if ((use_disk || near) && live) {   // (the next point is on its way meanwhile)
                uint32_t m = live, i = (uint32_t)item_point<G>(base, t, __ffs(m) - 1);
                float2 p = input_point(pts, i);
#pragma unroll 1
                while (m) {
                    const uint32_t bit = m & (0u - m), mine = i;
                    m ^= bit;
                    float2 next = p;
                    if (m) next = input_point(pts, i = (uint32_t)item_point<G>(base, t, __ffs(m) - 1));
                    if (!settle(fs.so, f, use_disk, mine | (near ? kUnsettled : 0u), p, octs)) live ^= bit;
                    p = next;
                }
            }
            const uint32_t left = __reduce_add_sync(0xffffffffu, __popc(live));
            if (left)
                append_survivors<kFiltItems>(live, left, fs.sink, [&](int k, uint32_t &i) {
                    i = (uint32_t)item_point<G>(base, t, k);
                    return input_point(pts, i);
                });
        }
    }
    while (q.n) queue_drain(q, fs, f, use_disk, pts, octs);
}

// The vertices in shared memory, with the repeated ends.
__device__ __forceinline__ void load_fan(float2 *sv, const float2 *V, int nb)
{
    // (both 16-byte aligned, nb even; four loads in flight)
    const float4 *src = reinterpret_cast<const float4 *>(V);
    float4 *dst = reinterpret_cast<float4 *>(sv);
#pragma unroll 4
    for (int i = threadIdx.x; i < nb / 2; i += blockDim.x) dst[i] = __ldg(src + i);
    if (threadIdx.x == 0) {
        sv[-2] = __ldg(V + nb - 2);
        sv[-1] = __ldg(V + nb - 1);
        sv[nb] = __ldg(V);
        sv[nb + 1] = __ldg(V + 1);
    }
}

// (2^-20 covers the rounding of a point's binary32 squared distance)
__device__ __forceinline__ float disk_limit(float rho2) { return __fmul_rd(rho2, 1.0f - 0x1p-20f); }

// The tiles go in contiguous ranges to groups of kFiltThreads threads.  One
// block of 768 threads per SM: the vertices and the queues take its shared
// memory, and what its registers do not hold would go to L2.  Bound by issue
// and the vertices' bank conflicts on circle-like sets (about 18 instructions
// for the octagon, 27 for the fan and two vertex reads per point) and by the
// points' latency on others.  Testing and writing in one pass replaces a
// count pass, a fan pass and a scatter that each read the points again: 274 +
// 455 + 214 us on 10^8 points of the unit circle.
template <int G>
__global__ void __launch_bounds__(CT, 1) hull_filter_kernel(const float *__restrict__ pts, uint32_t n, void *ws, Layout L,
                                                            int has_fan, int use_bits, const int32_t *kdev)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ FilterSmem fs;
    const Octagon *oct = at<Octagon>(ws, L.oct);
    if (oct->abort) return;
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    fill_octagon(fs.so, oct);
    if (threadIdx.x == 0) {
        fs.octs = 0u;
        fs.sink = Sink{&at<Ctrl>(ws, L.ctrl)->surv_count, at<uint32_t>(ws, L.keys[0]),
                       at<unsigned long long>(ws, L.pay[0])};
    }
    const Kgon *g = at<Kgon>(ws, L.kgon);
    const bool fan = has_fan && !oct->spec && fan_ready(kc, g);
    float2 *sv = reinterpret_cast<float2 *>(smem_raw + kQueueSmem) + 2;
    if (fan) load_fan(sv, g->v, kFanBins);
    __syncthreads();
    uint32_t octs = 0;   // octagon survivors of this thread
    if (oct->spec) {
        octs = filter_candidates(fs, ws, L);
    } else {
        const uint32_t ntiles = (n + kFiltTile - 1) / kFiltTile;   // (n < 2^30)
        const uint32_t gi = blockIdx.x * CG + threadIdx.x / kFiltThreads;
        const uint32_t per = (ntiles + gridDim.x * CG - 1) / (gridDim.x * CG);
        uint32_t *const queue = reinterpret_cast<uint32_t *>(smem_raw) + (threadIdx.x >> 5) * kQueue;
        const uint16_t *const bits = use_bits && (!kdev || *kdev != 8) ? at<uint16_t>(ws, L.keep_bits) : nullptr;
        const float scale = fs.so.scale, rho2t = fan ? disk_limit(fan_rho2(kc)) : 0.0f;
        const float2 c = fan_centre(fs.so);
        const bool disk = fan && kc->gaps == 0u;
        const uint32_t t0 = gi * per, t1 = min(ntiles, (gi + 1) * per);
        if (fan && scale != 1.0f)
            filter_tiles<G>(fs, FanView<Level1, true>{fan, Level1{}, SharedFan(sv), c, rho2t, disk, scale}, queue, pts, n,
                            t0, t1, 1u, bits, octs);
        else
            filter_tiles<G>(fs, FanView<Level1, false>{fan, Level1{}, SharedFan(sv), c, rho2t, disk, 1.0f}, queue, pts, n,
                            t0, t1, 1u, bits, octs);
    }
    octs = __reduce_add_sync(0xffffffffu, octs);
    if (lane_id() == 0 && octs) atomicAdd(&fs.octs, octs);
    __syncthreads();
    if (threadIdx.x == 0 && fs.octs) atomicAdd(&kc->s_oct, fs.octs);
}

// ---------------------------------------------------------------------------
// second level, over the first level's survivors.  On the unit circle the
// binary32 points scatter about 10^-7 around the circle while a chord of
// the first fan sags 6 10^-9 below it, so a fan vertex, the farthest
// sampled point of its bin, leaves the points near the top of that scatter
// outside its triangles: about a sixteenth of 10^8 points.  The same test
// with kFan2Sub times as many bins, each vertex the farthest survivor of
// its sub-bin (every survivor, not a sample), drops most of those.
//
//  fan2_max_kernel      whether the level runs (a fan whose proofs hold, and
//                       at least kFan2MinS points, or the tuned minimum,
//                       survived); per sub-bin the farthest survivor
//  fan2_build_kernel    the vertex of every sub-bin (the previous non-empty
//                       one for an empty sub-bin, cyclically); where the next
//                       one is not proven counter-clockwise from it: none
//                       (the first level's proofs put c inside the hull)
//  fan2_test_kernel     the test of every survivor; the kept ones go to the
//                       sort's second buffers, which the sort then reads
// ---------------------------------------------------------------------------
constexpr int F2T = 256;
constexpr int F2I = 8;   // survivors per thread and step of the test
static_assert(kFan2Bins % BT == 0, "sub-bins split evenly over the build blocks");

__device__ __forceinline__ float2 surv_point(const uint32_t *keys, const unsigned long long *pay, uint32_t i, float scale)
{
    return fan_space(make_float2(key_float(keys[i]), key_float((uint32_t)(pay[i] >> 32))), scale);
}

__global__ void __launch_bounds__(F2T) fan2_max_kernel(void *ws, Layout L, uint32_t min_s)
{
    kernel_entry();
    const Octagon *oct = at<Octagon>(ws, L.oct);
    const Kgon *g = at<Kgon>(ws, L.kgon);
    const uint32_t m = at<Ctrl>(ws, L.ctrl)->surv_count;
    const bool on = !oct->abort && !oct->spec && m >= min_s && fan_ready(at<KgonCtrl>(ws, L.kgon_ctrl), g);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        Fan2Ctrl *f2 = at<Fan2Ctrl>(ws, L.fan2);
        f2->on = on ? 1u : 0u;
        f2->count_in = on ? m : 0u;
    }
    if (!on) return;
    const uint32_t *keys = at<uint32_t>(ws, L.keys[0]);
    const unsigned long long *pay = at<unsigned long long>(ws, L.pay[0]);
    unsigned long long *slot = at<unsigned long long>(ws, L.fan2_slot);
    const float cx = g->cx, cy = g->cy, r2ref = far_ref(*oct), scale = oct->scale;
    for (uint32_t i = blockIdx.x * F2T + threadIdx.x; i < m; i += gridDim.x * F2T) {
        const float2 p = surv_point(keys, pay, i, scale);
        const int b = vertex_bin(Level2{}, __fsub_rn(p.x, cx), __fsub_rn(p.y, cy), kFan2Margin);
        if (b < 0) continue;
        const unsigned long long v = ((unsigned long long)far_key(p.x, p.y, cx, cy, r2ref) << 32) | (uint32_t)~i;
        if (v > __ldcg(&slot[b])) atomicMax(&slot[b], v);   // the read only saves atomics
    }
}

// One thread per sub-bin, as fan_build_kernel; the table's ends are repeated
// at V[-2], V[-1] and V[kFan2Bins], V[kFan2Bins + 1].
__global__ void __launch_bounds__(BT) fan2_build_kernel(void *ws, Layout L)
{
    kernel_entry();
    __shared__ int s_w[BT / 32];
    __shared__ int s_scan[BT / 32];
    Fan2Ctrl *f2 = at<Fan2Ctrl>(ws, L.fan2);
    if (!f2->on) return;
    const unsigned long long *slot = at<unsigned long long>(ws, L.fan2_slot);
    const uint32_t *keys = at<uint32_t>(ws, L.keys[0]);
    const unsigned long long *pay = at<unsigned long long>(ws, L.pay[0]);
    const Kgon *g = at<Kgon>(ws, L.kgon);
    float2 *V = at<float2>(ws, L.fan2_v) + 2;
    const int b = (int)(blockIdx.x * BT + threadIdx.x);
    const int src = vertex_source([&](int j) { return slot[j] != 0ull; }, s_w, s_scan);
    if (src < 0) {   // no survivor reached a slot: keep everything
        if (threadIdx.x == 0) f2->bad = 1u;
        return;
    }
    const float scale = at<Octagon>(ws, L.oct)->scale;
    float2 v = surv_point(keys, pay, ~(uint32_t)slot[src], scale);
    const unsigned long long nextp = slot[b + 1 == kFan2Bins ? 0 : b + 1];
    const float2 w = nextp != 0ull ? surv_point(keys, pay, ~(uint32_t)nextp, scale) : v;
    const bool edge = v.x != w.x || v.y != w.y;
    // c strictly left of v -> w, proven in binary32 or exactly
    const bool gap = edge && orient(v.x, v.y, w.x, w.y, g->cx, g->cy) <= 0;
    if (gap) v.x = __int_as_float(0x7fc00000);
    V[b] = v;
    if (b < 2) V[kFan2Bins + b] = v;
    if (b >= kFan2Bins - 2) V[b - kFan2Bins] = v;
    const uint32_t edges = __popc(__ballot_sync(0xffffffffu, edge && !gap));
    if (lane_id() == 0 && edges) atomicAdd(&f2->edges, edges);
}

// Bound by the latency of the 1.8 MB table in L2: eight survivors per thread
// keep their reads in flight together, and only binary32 signs are taken.
// The order of the survivors is not kept, so the kept ones are appended and
// need no second pass (test and ordered compaction took 105 + 39 us for the
// 6.4 M first-level survivors of 10^8 circle points).
__global__ void __launch_bounds__(F2T) fan2_test_kernel(void *ws, Layout L)
{
    kernel_entry();
    Fan2Ctrl *f2 = at<Fan2Ctrl>(ws, L.fan2);
    if (!f2->on) return;
    const uint32_t m = f2->count_in;
    const bool test = !f2->bad && f2->edges != 0u;
    const Kgon *g = at<Kgon>(ws, L.kgon);
    const float2 c = make_float2(g->cx, g->cy);
    const float scale = at<Octagon>(ws, L.oct)->scale;
    const GlobalFan F{at<float2>(ws, L.fan2_v) + 2};
    const uint32_t *keys = at<uint32_t>(ws, L.keys[0]);
    const unsigned long long *pay = at<unsigned long long>(ws, L.pay[0]);
    uint32_t *okeys = at<uint32_t>(ws, L.keys[1]);
    unsigned long long *opay = at<unsigned long long>(ws, L.pay[1]);
    const uint32_t lane = lane_id();
    for (uint32_t base = blockIdx.x * (F2T * F2I); base < m; base += gridDim.x * (F2T * F2I)) {
        uint32_t kv[F2I];
        unsigned long long pv[F2I];
        uint32_t keep = 0;
#pragma unroll
        for (int k = 0; k < F2I; ++k) {
            const uint32_t i = base + k * F2T + threadIdx.x;
            kv[k] = 0u;
            pv[k] = 0ull;
            if (i < m) {
                kv[k] = __ldcs(keys + i);
                pv[k] = __ldcs(pay + i);
                keep |= 1u << k;
            }
        }
        if (test) {
            uint32_t in = 0;
#pragma unroll
            for (int k = 0; k < F2I; ++k) {
                const float2 p = fan_space(make_float2(key_float(kv[k]), key_float((uint32_t)(pv[k] >> 32))), scale);
                if (fan_inside(Level2{}, F, c, sub2(p, c), p)) in |= 1u << k;
            }
            keep &= ~in;
        }
        uint32_t incl = __popc(keep);
        const uint32_t cnt = incl;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += u;
        }
        uint32_t pos = 0;
        if (lane == 31 && incl) pos = atomicAdd(&f2->kept, incl);
        pos = __shfl_sync(0xffffffffu, pos, 31) + incl - cnt;
#pragma unroll
        for (int k = 0; k < F2I; ++k) {
            if ((keep >> k) & 1u) {
                okeys[pos] = kv[k];
                opay[pos] = pv[k];
                ++pos;
            }
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        if (atomicAdd(&f2->done, 1u) == gridDim.x - 1) {   // every block's survivors are counted
            Ctrl *ctrl = at<Ctrl>(ws, L.ctrl);
            ctrl->surv_count = atomicAdd(&f2->kept, 0u);
            ctrl->sort_in = 1u;
        }
    }
}

template <int G>
cudaError_t launch_hull_filter_g(const float *pts, int64_t n, void *ws, const Layout &L, int use_bits,
                                 const int32_t *kdev, cudaStream_t st)
{
    const int sms = sm_count();
    static const bool attr = [] {   // thread-safe one-time initialisation
        cudaFuncSetAttribute(hull_filter_kernel<G>, cudaFuncAttributeMaxDynamicSharedMemorySize, kQueueSmem + kFanTable);
        return true;
    }();
    (void)attr;
    const int64_t ntiles = ceil_div(n, kFiltTile);
    const int has_fan = n >= (int64_t)kKgonMinS ? 1 : 0;   // (fewer points: fewer survivors)
    if (has_fan) {
        const int64_t stride = fan_sample_stride(ntiles);
        const int64_t bb = std::min<int64_t>(ceil_div(ntiles, stride) * (kFiltItems / BI), (int64_t)sms * 5);
        probe_before(CH_K_KGON, st);
        launch_next(fan_bins_kernel<G>, (unsigned)bb, kFiltThreads, 0, st, pts, (uint32_t)n, ws, L, (uint32_t)stride,
                    use_bits, kdev);
        launch_next(fan_vertex_kernel, kFanBins / (VB * VT / 32), VT, 0, st, pts, n, ws, L);
        launch_next(fan_build_kernel, kFanBins / BT, BT, 0, st, n, ws, L);
        note_kernels(CH_K_KGON, 3);
        probe_after(CH_K_KGON, st);
    }
    probe_before(CH_K_FILTER, st);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ceil_div(ntiles, (int64_t)CG), sms));
    launch_next(hull_filter_kernel<G>, (unsigned)grid, CT, kQueueSmem + (has_fan ? kFanTable : 0), st, pts,
                (uint32_t)n, ws, L, has_fan, use_bits, kdev);
    note_kernels(CH_K_FILTER, 1);
    probe_after(CH_K_FILTER, st);
    cudaError_t e = cudaGetLastError();
    // a set too small for the second level, or of fewer than four times as
    // many points as it asks for: a first level that leaves a quarter of them
    // is looking at vertices, and three idle launches are 6 % of a call on 2^20
    // points
    const int lg = tune_value(CH_TUNE_FAN2_MIN_LOG2);
    const uint32_t min_s = lg ? (uint32_t)(1ull << lg) : kFan2MinS;
    if (e != cudaSuccess || L.fan2_bins == 0 || n < 4 * (int64_t)min_s) return e;
    probe_before(CH_K_KGON, st);
    launch_next(fan2_max_kernel, sms * 8, F2T, 0, st, ws, L, min_s);
    launch_next(fan2_build_kernel, kFan2Bins / BT, BT, 0, st, ws, L);
    const int64_t tb = std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, (int64_t)F2T * F2I), (int64_t)sms * 8));
    launch_next(fan2_test_kernel, (unsigned)tb, F2T, 0, st, ws, L);
    note_kernels(CH_K_KGON, 3);
    probe_after(CH_K_KGON, st);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_hull_filter(const float *pts, int64_t n, void *ws, const Layout &L, const KgonStage *kg,
                               cudaStream_t st)
{
    const bool bits = kg && (kg->kdev || kg->K != 8);   // the second polygon's keep bits
    if (bits) {
        cudaError_t e = launch_filter_count(pts, n, kg->kdev, ws, L, st);
        if (e == cudaSuccess) e = launch_kx_sv(pts, n, kg->dirs, kg->kdev, kg->K, kg->ext_out, ws, L, st);
        if (e != cudaSuccess) return e;
    }
    const int32_t *kdev = bits ? kg->kdev : nullptr;
    return (reinterpret_cast<uintptr_t>(pts) & 15u) == 0
               ? launch_hull_filter_g<2>(pts, n, ws, L, bits ? 1 : 0, kdev, st)
               : launch_hull_filter_g<1>(pts, n, ws, L, bits ? 1 : 0, kdev, st);
}

namespace {

// ---------------------------------------------------------------------------
// many sets (ch_hull_batched): the same filter per set.  A set's survivors go
// to its own stretch of the sort arrays (from its first point's position), so
// no scan over tiles places them.  Sets of at least kBxFanMinN points with
// enough octagon survivors in a sample get a fan of up to kBxTileBins bins per
// tile, smoothed as the single set's; one whose fan drops less than an eighth
// of a sample goes without.
// ---------------------------------------------------------------------------
constexpr int64_t kBxTightMinN = 65536;
constexpr int kBxSample = 256;        // points of a set's estimates
static_assert(kFanBins % kBxBinRun == 0 && kBxTileBins % kBxBinRun == 0 && kBxBinRun == VB * VT / 32, "whole runs of bins");

// A fan's bins and sample, by what limits it.  Points of a circle (tight)
// differ in radius by the rounding of their coordinates: only short chords lie
// above enough of them, so as many bins as shared memory holds and every or
// every second tile (fewer than 65536 points: nearly all are vertices, no
// fan).  Elsewhere the farthest of few samples in a wide sector do: a bin per
// 16 points, at most 8192, and a sample of about 65536 points.  (With the
// circle's choice for all sets, 4096 sets' bins, vertices and vertex tables
// took 1.7 ms more.)
__device__ __forceinline__ uint32_t bx_bins(uint32_t ntiles, bool tight)
{
    return tight ? min(ntiles * kBxTileBins, (uint32_t)kFanBins)
                 : min((ntiles * 256u + kBxBinRun - 1u) / kBxBinRun * kBxBinRun, 8192u);
}
__device__ __forceinline__ uint32_t bx_stride(int64_t n, bool tight)
{
    return tight ? 1u : (uint32_t)max(1ll, min(8ll, (long long)(n >> 16)));
}

// One warp per set: whether it gets a fan -- at least 2048 octagon survivors,
// estimated from kBxSample evenly spaced points.
__global__ void __launch_bounds__(256) bx_fan_want_kernel(const float *__restrict__ pts, void *ws, BatchLayout BL)
{
    kernel_entry();
    const int64_t b = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (b >= BL.num_sets) return;
    const SetInfo &S = at<SetInfo>(ws, BL.sets)[b];
    const Octagon &o = at<Octagon>(ws, BL.octs)[b];
    FanInfo &f = at<FanInfo>(ws, BL.fan)[b];
    uint32_t out = 0;
    float lo = __int_as_float(0x7f800000), hi = 0.0f;   // squared distances
    const bool may = !at<BatchCtrl>(ws, BL.bctrl)->abort && !o.abort && o.has_edges && S.n >= kBxFanMinN;   // warp-uniform
    if (may) {
        const float2 *p = reinterpret_cast<const float2 *>(pts) + S.pt_begin;
        float2 v[kBxSample / 32];
#pragma unroll
        for (int r = 0; r < kBxSample / 32; ++r) v[r] = __ldg(p + S.n * (r * 32 + (int)lane_id()) / kBxSample);
#pragma unroll
        for (int r = 0; r < kBxSample / 32; ++r) {
            const float x = __fsub_rn(v[r].x, o.cx), y = __fsub_rn(v[r].y, o.cy);
            const float2 d = fan_space(make_float2(x, y), o.scale);
            float m = __int_as_float(0x7f800000);
#pragma unroll
            for (int k = 0; k < 8; ++k) m = min_nan(m, __fmaf_rn(o.tx[k], x, __fmaf_rn(o.ty[k], y, o.tz[k])));
            out += m > 1.0f ? 0u : 1u;
            const float r2 = __fmaf_rn(d.x, d.x, __fmul_rn(d.y, d.y));
            lo = fminf(lo, r2);
            hi = fmaxf(hi, r2);
        }
        out = __reduce_add_sync(0xffffffffu, out);
        // (non-negative: their bits order as they do)
        lo = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(lo)));
        hi = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(hi)));
    }
    if (lane_id() == 0) {
        const bool tight = hi - lo <= hi * 0x1p-16f;
        f.tight = tight ? 1u : 0u;
        f.nb = bx_bins(S.ntiles, tight);
        f.want = may && (int64_t)out * S.n >= (int64_t)2048 * kBxSample && (!tight || S.n >= kBxTightMinN) ? 1u : 0u;
    }
}

// One block: the lists of the fan sets and of all work items (runs of `chunk`
// tiles of a fan set, of kBxPlainChunk tiles of another, of kBxBinRun bins).
__global__ void __launch_bounds__(1024) bx_fan_select_kernel(void *ws, BatchLayout BL, uint32_t chunk)
{
    kernel_entry();
    __shared__ uint32_t s_w[4][32];
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    FanInfo *fan = at<FanInfo>(ws, BL.fan);
    uint2 *fi = at<uint2>(ws, BL.fan_items), *pi = at<uint2>(ws, BL.plain_items), *bi = at<uint2>(ws, BL.bin_items);
    const int64_t B = BL.num_sets;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const int64_t per = ceil_div(B, (int64_t)blockDim.x);
    const int64_t b0 = min((int64_t)threadIdx.x * per, B), b1 = min(b0 + per, B);
    uint32_t c[4] = {0, 0, 0, 0};   // fan sets, fan items, plain items, bin runs
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t nt = sets[b].ntiles;
        if (fan[b].want) {
            c[0] += 1u;
            c[1] += (nt + chunk - 1) / chunk;
            c[3] += fan[b].nb / kBxBinRun;
        } else {
            c[2] += (nt + kBxPlainChunk - 1) / kBxPlainChunk;
        }
    }
    uint32_t run[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        uint32_t incl = c[q];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl += u;
        }
        if (lane == 31) s_w[q][warp] = incl;
        run[q] = incl - c[q];
    }
    __syncthreads();
    uint32_t tot[4] = {0, 0, 0, 0};
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (w < warp) run[q] += s_w[q][w];
            tot[q] += s_w[q][w];
        }
    }
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t nt = sets[b].ntiles;
        if (fan[b].want) {
            const uint32_t nb = fan[b].nb;
            fan[b].ready = 0u;
            at<uint32_t>(ws, BL.fan_set)[run[0]++] = (uint32_t)b;
            for (uint32_t t = 0; t < nt; t += chunk) fi[run[1]++] = make_uint2((uint32_t)b, t);
            for (uint32_t k = 0; k < nb; k += kBxBinRun) bi[run[3]++] = make_uint2((uint32_t)b, k);
        } else {
            for (uint32_t t = 0; t < nt; t += kBxPlainChunk) pi[run[2]++] = make_uint2((uint32_t)b, t);
        }
    }
    if (threadIdx.x == 0) {
        bc->nfan = tot[0];
        bc->nfan_items = tot[1];
        bc->nplain_items = tot[2];
        bc->nbin_items = tot[3];
    }
}

// A set's slots, vertices (in the same place once the slots are read) and
// vertices before empty bins are filled (BatchLayout::fan_tab; 16-byte
// aligned, nb is even).
__device__ __forceinline__ unsigned long long *bx_slots(void *ws, const BatchLayout &BL, const SetInfo &S)
{
    return at<unsigned long long>(ws, BL.fan_tab) + ((S.pt_begin + 1) & ~(int64_t)1);
}
__device__ __forceinline__ float2 *bx_raw(void *ws, const BatchLayout &BL, const SetInfo &S, uint32_t nb)
{
    return reinterpret_cast<float2 *>(bx_slots(ws, BL, S) + nb);
}

__global__ void __launch_bounds__(256) bx_fan_zero_kernel(void *ws, BatchLayout BL)
{
    kernel_entry();
    const uint2 *bi = at<uint2>(ws, BL.bin_items);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t n = at<BatchCtrl>(ws, BL.bctrl)->nbin_items;
    for (uint32_t w = blockIdx.x; w < n; w += gridDim.x) {
        unsigned long long *slot = bx_slots(ws, BL, sets[bi[w].x]) + bi[w].y;
        for (int k = threadIdx.x; k < kBxBinRun; k += 256) slot[k] = 0ull;
    }
}

// Per work item of a fan set, every stride-th tile (counted from the set's
// first; 0: the built-in choice): the bins' farthest points, as
// fan_bins_kernel.
__global__ void __launch_bounds__(kFiltThreads, 5) bx_fan_bins_kernel(const float *__restrict__ pts, void *ws, BatchLayout BL,
                                                                      uint32_t chunk, uint32_t stride)
{
    kernel_entry();
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint2 *items = at<uint2>(ws, BL.fan_items);
    const uint32_t nitems = at<BatchCtrl>(ws, BL.bctrl)->nfan_items, t = threadIdx.x;
    constexpr uint32_t parts = kFiltItems / BI;
    // (eight tiles of an item at a time: the set's data are looked up once)
    const uint32_t units = chunk / kBxFanChunkMin;
    for (uint32_t w = blockIdx.x; w < nitems * units; w += gridDim.x) {
        const uint2 item = items[w / units];
        const SetInfo &S = sets[item.x];
        const FanInfo &info = at<FanInfo>(ws, BL.fan)[item.x];
        const uint32_t st = stride ? stride : bx_stride(S.n, info.tight);
        const uint32_t first = (item.y + w % units * kBxFanChunkMin + st - 1) / st * st;
        const uint32_t end = min(item.y + (w % units + 1) * kBxFanChunkMin, S.ntiles);
        if (first >= end) continue;   // block-uniform
        const Octagon &o = octs[item.x];
        const SetBins nb{info.nb};
        const float r2ref = far_ref(o), scale = o.scale;
        const float2 c = fan_centre(o);
        const float *p2 = pts + 2 * S.pt_begin;
        unsigned long long *slot = bx_slots(ws, BL, S);
        const uint32_t n = (uint32_t)S.n, steps = ((end - first + st - 1) / st) * parts;   // parts of every st-th tile
        float px[BI], py[BI];
        uint32_t live = 0;
        const auto fetch = [&](uint32_t u) {
            const uint32_t base = (first + u / parts * st) * kFiltTile;
            const int part = (int)(u % parts);
            if (base + kFiltTile <= n) {
                load_part<1, BI>(p2, base, t, part, px, py);
                live = (1u << BI) - 1u;
            } else {
                live = load_part_ragged<1, BI>(p2, n, base, t, part, o.cx, o.cy, px, py);
            }
        };
        fetch(0);
        if (first == 0u && t < 32u) {
            const unsigned long long *ext = at<unsigned long long>(ws, BL.ext_slot) + (size_t)item.x * 8;
            raise_octagon(nb, slot, o, [&](int k) { return ~(uint32_t)ext[k]; });
        }
        for (uint32_t u = 0; u < steps; ++u) {
            float qx[BI], qy[BI];
            const uint32_t mine = live;
#pragma unroll
            for (int k = 0; k < BI; ++k) {
                qx[k] = px[k];
                qy[k] = py[k];
            }
            if (u + 1 < steps) fetch(u + 1);
            to_fan_space(qx, qy, scale);
            raise_bins(nb, slot, qx, qy, mine, c, r2ref, [&](int k) {
                return (uint32_t)item_point<1>((first + u / parts * st) * kFiltTile, t, (int)(BI * (u % parts)) + k);
            });
        }
    }
}

// A block per run of kBxBinRun bins: the vertices (make_vertices).
__global__ void __launch_bounds__(VT) bx_fan_vertex_kernel(const float *__restrict__ pts, void *ws, BatchLayout BL)
{
    kernel_entry();
    __shared__ VertexSmem sm[VT / 32];
    const uint2 *bi = at<uint2>(ws, BL.bin_items);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint32_t n = at<BatchCtrl>(ws, BL.bctrl)->nbin_items;
    const int warp = (int)(threadIdx.x >> 5);
    for (uint32_t w = blockIdx.x; w < n; w += gridDim.x) {
        const uint2 item = bi[w];
        const SetInfo &S = sets[item.x];
        const float2 *p = reinterpret_cast<const float2 *>(pts) + S.pt_begin;
        const int64_t m = S.n;
        const FanInfo &info = at<FanInfo>(ws, BL.fan)[item.x];
        if (info.tight) {   // the farthest samples themselves (a chord's rounded point would lie deeper)
            const unsigned long long *slot = bx_slots(ws, BL, S);
            float2 *raw = bx_raw(ws, BL, S, info.nb);
            for (int k = (int)item.y + (int)threadIdx.x; k < (int)item.y + kBxBinRun; k += VT) {
                const unsigned long long v = __ldcg(slot + k);
                const uint32_t i = ~(uint32_t)v;
                raw[k] = v != 0ull ? fan_space(__ldg(p + ((int64_t)i < m ? i : 0u)), octs[item.x].scale)
                                   : make_float2(__int_as_float(0x7fc00000), 0.0f);
            }
            continue;   // block-uniform
        }
        make_vertices(
            SetBins{info.nb}, sm[warp], bx_slots(ws, BL, S), (int)item.y + warp * VB,
            fan_centre(octs[item.x]),
            [&](uint32_t i) { return fan_space(__ldg(p + ((int64_t)i < m ? i : 0u)), octs[item.x].scale); },
            bx_raw(ws, BL, S, info.nb));
        __syncwarp();
    }
}

// A block per fan set: empty bins repeat the vertex before them; the proofs
// of fan_build_kernel; and whether the fan drops at least an eighth of a
// sample.
__global__ void __launch_bounds__(BT, 2) bx_fan_build_kernel(const float *__restrict__ pts, void *ws, BatchLayout BL)
{
    kernel_entry();
    __shared__ int s_w[BT / 32];
    __shared__ int s_last;
    __shared__ uint32_t s_inv, s_edges, s_gaps, s_in, s_seen;
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint32_t nfan = at<BatchCtrl>(ws, BL.bctrl)->nfan;
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    for (uint32_t k = blockIdx.x; k < nfan; k += gridDim.x) {
        const uint32_t set = at<uint32_t>(ws, BL.fan_set)[k];
        const SetInfo &S = sets[set];
        const Octagon &o = octs[set];
        FanInfo &info = at<FanInfo>(ws, BL.fan)[set];
        const float2 *raw = bx_raw(ws, BL, S, info.nb);
        float2 *V = reinterpret_cast<float2 *>(bx_slots(ws, BL, S));
        const SetBins nb{info.nb};
        const int NB = (int)nb.n;
        const float2 c = fan_centre(o);
        __syncthreads();   // the shared words of the previous set have been read
        if (tid == 0) {
            s_last = -1;
            s_inv = s_edges = s_gaps = s_in = s_seen = 0u;
        }
        __syncthreads();
        int last = -1;   // the last bin with a vertex (what the first empty bins repeat)
        for (int b = (int)tid; b < NB; b += BT)
            if (raw[b].x == raw[b].x) last = b;
        last = __reduce_max_sync(0xffffffffu, last);
        if (lane == 0) atomicMax(&s_last, last);
        __syncthreads();
        int carry = s_last;
        if (carry < 0) continue;   // block-uniform
        uint32_t inv = 0, edges = 0;
        bool gaps = false;
        for (int b0 = 0; b0 < NB; b0 += BT) {   // (NB is a multiple of kBxBinRun: the last chunk may be half full)
            const int b = b0 + (int)tid;
            const float2 mine = b < NB ? raw[b] : make_float2(__int_as_float(0x7fc00000), 0.0f);
            int src = mine.x == mine.x ? b : -1;
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, src, q);
                if (lane >= (uint32_t)q) src = max(src, u);
            }
            if (lane == 31) s_w[warp] = src;
            __syncthreads();
            static_assert(BT / 32 == 32, "a lane per warp");
            const int ends = s_w[lane];
            const int all = __reduce_max_sync(0xffffffffu, ends);
            src = max(src, __reduce_max_sync(0xffffffffu, lane < warp ? ends : -1));
            __syncthreads();   // s_w is written again by the next chunk
            if (src < 0) src = carry;
            if (all >= 0) carry = all;
            if (b < NB) {
                float2 v = src == b ? mine : raw[src];
                const float2 next = raw[b + 1 == NB ? 0 : b + 1];
                const float2 w = next.x == next.x ? next : v;
                if (v.x != w.x || v.y != w.y) {
                    const float r = disk_bound(c.x, c.y, v, w);
                    inv = max(inv, ~__float_as_uint(fmaxf(r, 0.0f)));
                    if (r < 0.0f) {
                        gaps = true;
                        v.x = __int_as_float(0x7fc00000);
                    } else {
                        ++edges;
                    }
                }
                V[b] = v;
            }
        }
        inv = __reduce_max_sync(0xffffffffu, inv);
        edges = __reduce_add_sync(0xffffffffu, edges);
        if (lane == 0) {
            atomicMax(&s_inv, inv);
            atomicAdd(&s_edges, edges);
        }
        if (gaps) s_gaps = 1u;
        __syncthreads();
        const float rho2 = __uint_as_float(~s_inv);
        const bool gap = s_gaps != 0u;
        if (!fan_holds(s_edges, gap, rho2, gap && centre_inside(o))) continue;   // block-uniform
        if (tid < (uint32_t)kBxSample) {   // (points of the first and last bins, whose neighbours wrap, are left out)
            const float2 p = fan_space(__ldg(reinterpret_cast<const float2 *>(pts) + S.pt_begin + S.n * tid / kBxSample), o.scale);
            const float2 d = sub2(p, c);
            const uint32_t b = fan_bin_biased(nb, d.x, d.y) - kBinBias;
            bool in = false;
            const bool seen = inner_bin(b, nb.n);
            if (seen) {
                const float2 Q = __ldcg(V + b);
                float e1, e2;
                const float side = det_bound(sub2(Q, c), d, e1);
                const float2 W = __ldcg(V + (side > 0.0f ? b + 1u : b - 1u));
                const float det = det_bound(sub2(W, Q), sub2(p, Q), e2);
                in = fabsf(side) > e1 && (side > 0.0f ? det : -det) > e2;
            }
            const uint32_t ni = __popc(__ballot_sync(0xffffffffu, in)), ns = __popc(__ballot_sync(0xffffffffu, seen));
            if (lane == 0) {
                atomicAdd(&s_in, ni);
                atomicAdd(&s_seen, ns);
            }
        }
        __syncthreads();
        if (tid == 0) {
            info.rho2 = gap ? 0.0f : rho2;
            info.ready = 8u * s_in >= s_seen ? 1u : 0u;
        }
    }
}

// The octagon, the sink and (fan) the vertices of set b into shared memory.
__device__ __forceinline__ void bx_load_set(FilterSmem &fs, float2 *sv, void *ws, const Layout &L, const BatchLayout &BL,
                                            uint32_t b)
{
    const SetInfo &S = at<SetInfo>(ws, BL.sets)[b];
    fill_octagon(fs.so, at<Octagon>(ws, BL.octs) + b);
    if (threadIdx.x == 0)
        fs.sink = Sink{at<uint32_t>(ws, BL.soct) + b, at<uint32_t>(ws, L.keys[0]) + S.pt_begin,
                       at<unsigned long long>(ws, L.pay[0]) + S.pt_begin};
    const FanInfo &info = at<FanInfo>(ws, BL.fan)[b];
    if (sv && info.ready) load_fan(sv, reinterpret_cast<const float2 *>(bx_slots(ws, BL, S)), (int)info.nb);
}

// Persistent blocks take the fan sets' work items by ticket; octagon and
// vertices are read again only when the set changes (a set's items follow one
// another).
__global__ void __launch_bounds__(CT, 1) bx_hull_filter_kernel(const float *__restrict__ pts, void *ws, Layout L,
                                                               BatchLayout BL, uint32_t chunk)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ FilterSmem fs;
    float2 *sv = reinterpret_cast<float2 *>(smem_raw + kQueueSmem) + 2;
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint2 *items = at<uint2>(ws, BL.fan_items);
    const uint32_t nitems = bc->nfan_items;
    uint32_t *queue = reinterpret_cast<uint32_t *>(smem_raw) + (threadIdx.x >> 5) * kQueue;
    uint32_t cur = 0xffffffffu, octs = 0;
    for (;;) {
        __syncthreads();   // the item and the set's data have been read
        if (threadIdx.x == 0) fs.item = atomicAdd(&bc->fan_ticket, 1u);
        __syncthreads();
        const uint32_t w = fs.item;
        if (w >= nitems) break;
        const uint2 item = items[w];
        if (item.x != cur) {
            cur = item.x;
            bx_load_set(fs, sv, ws, L, BL, cur);
            __syncthreads();
        }
        const SetInfo &S = sets[cur];
        const FanInfo &info = at<FanInfo>(ws, BL.fan)[cur];
        const bool fan = info.ready != 0u;
        const float scale = fs.so.scale, rho2t = fan ? disk_limit(info.rho2) : 0.0f;
        const float2 c = fan_centre(fs.so);
        const bool disk = info.tight == 0u && info.rho2 > 0.0f;
        const float *p = pts + 2 * S.pt_begin;
        const uint32_t first = item.y + threadIdx.x / kFiltThreads, end = min(item.y + chunk, S.ntiles);
        const FanView<SetBins, false> f{fan, SetBins{info.nb}, SharedFan(sv), c, rho2t, disk, 1.0f};
        if (fan && scale != 1.0f)
            filter_tiles<1>(fs, FanView<SetBins, true>{fan, SetBins{info.nb}, SharedFan(sv), c, rho2t, disk, scale}, queue,
                            p, (uint32_t)S.n, first, end, (uint32_t)CG, nullptr, octs);
        else if ((reinterpret_cast<uintptr_t>(p) & 15u) == 0)
            filter_tiles<2>(fs, f, queue, p, (uint32_t)S.n, first, end, (uint32_t)CG, nullptr, octs);
        else
            filter_tiles<1>(fs, f, queue, p, (uint32_t)S.n, first, end, (uint32_t)CG, nullptr, octs);
    }
}

// The same for the sets without a fan: many small blocks, no vertices.
__global__ void __launch_bounds__(kFiltThreads, 3) bx_plain_filter_kernel(const float *__restrict__ pts, void *ws, Layout L,
                                                                          BatchLayout BL)
{
    kernel_entry();
    __shared__ FilterSmem fs;
    __shared__ uint32_t s_queue[kFiltThreads / 32 * kQueue];
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint2 *items = at<uint2>(ws, BL.plain_items);
    const uint32_t nitems = bc->nplain_items;
    uint32_t cur = 0xffffffffu, octs = 0;
    for (;;) {
        __syncthreads();   // the item and the set's data have been read
        if (threadIdx.x == 0) fs.item = atomicAdd(&bc->plain_ticket, 1u);
        __syncthreads();
        const uint32_t w = fs.item;
        if (w >= nitems) break;
        const uint2 item = items[w];
        if (item.x != cur) {
            cur = item.x;
            bx_load_set(fs, nullptr, ws, L, BL, cur);
            __syncthreads();
        }
        if (fs.so.abort) continue;   // block-uniform
        const SetInfo &S = sets[cur];
        const FanView<SetBins, false> f{false, SetBins{4u}, SharedFan(nullptr), make_float2(0.0f, 0.0f), 0.0f, false, 1.0f};
        filter_tiles<1>(fs, f, s_queue + (threadIdx.x >> 5) * kQueue, pts + 2 * S.pt_begin, (uint32_t)S.n, item.y,
                        min(item.y + (uint32_t)kBxPlainChunk, S.ntiles), 1u, nullptr, octs);
    }
}

// One block: each set's survivors and the layout of the later stages: its
// super-chunks (4096 survivors, also the sort tiles) and merge-tree nodes.
__global__ void __launch_bounds__(1024) bx_layout_kernel(void *ws, BatchLayout BL)
{
    kernel_entry();
    __shared__ uint32_t s_w[3][32];
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    if (bc->abort) return;
    SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t *count = at<uint32_t>(ws, BL.soct);
    uint32_t *sc_set = at<uint32_t>(ws, BL.sc_set);
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const int64_t B = BL.num_sets;
    const int64_t per = ceil_div(B, (int64_t)blockDim.x);
    const int64_t b0 = min((int64_t)threadIdx.x * per, B), b1 = min(b0 + per, B);
    // super-chunks in two classes: the sort's, then those of the few-survivor
    // sets, which the chain kernel sorts itself
    uint32_t sc = 0, one = 0, nd = 0;
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t nsc = (uint32_t)ceil_div((int64_t)count[b], kChainC);
        if (count[b] - 1u < kBxLocalMax) ++one;
        else sc += nsc;
        nd += nsc > 0 ? (uint32_t)tree_nodes(nsc) + 1u : 0u;
    }
    uint32_t i0 = one, i1 = sc, i2 = nd;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u0 = __shfl_up_sync(0xffffffffu, i0, o), u1 = __shfl_up_sync(0xffffffffu, i1, o),
                       u2 = __shfl_up_sync(0xffffffffu, i2, o);
        if (lane >= (uint32_t)o) {
            i0 += u0;
            i1 += u1;
            i2 += u2;
        }
    }
    if (lane == 31) {
        s_w[0][warp] = i0;
        s_w[1][warp] = i1;
        s_w[2][warp] = i2;
    }
    __syncthreads();
    uint32_t rone = i0 - one, rsc = i1 - sc, rnd = i2 - nd, tsc = 0, tone = 0;
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) {
        if (w < warp) {
            rone += s_w[0][w];
            rsc += s_w[1][w];
            rnd += s_w[2][w];
        }
        tone += s_w[0][w];
        tsc += s_w[1][w];
    }
    rone += tsc;
    for (int64_t b = b0; b < b1; ++b) {
        const uint32_t s = count[b], nsc = (uint32_t)ceil_div((int64_t)s, kChainC);
        SetInfo &S = sets[b];
        S.surv_base = (uint64_t)S.pt_begin;
        S.s = s;
        S.nsc = nsc;
        uint32_t &at_sc = s - 1u < kBxLocalMax ? rone : rsc;
        S.sc_base = at_sc;
        S.node_base = rnd;
        for (uint32_t k = 0; k < nsc; ++k) sc_set[at_sc + k] = (uint32_t)b;
        at_sc += nsc;
        rnd += nsc > 0 ? (uint32_t)tree_nodes(nsc) + 1u : 0u;
    }
    if (threadIdx.x == 0) {
        bc->nsc = tsc + tone;
        bc->nsc_sort = tsc;
    }
}

}  // namespace

cudaError_t launch_bx_filter(const float *pts, void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st)
{
    const int sms = sm_count();
    static const bool attrs = [] {   // thread-safe one-time initialisation
        cudaFuncSetAttribute(bx_hull_filter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kQueueSmem + kFanTable);
        return true;
    }();
    (void)attrs;
    const uint32_t chunk = tune_value(CH_TUNE_BX_FAN_CHUNK) ? (uint32_t)tune_value(CH_TUNE_BX_FAN_CHUNK) : kBxFanChunk;
    const uint32_t stride = (uint32_t)tune_value(CH_TUNE_BX_FAN_STRIDE);
    const int tuned = tune_value(CH_TUNE_BX_FILTER);
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * 5, BL.tiles_max));
    probe_before(CH_K_KGON, st);
    launch_next(bx_fan_want_kernel, (unsigned)ceil_div(BL.num_sets, 8), 256, 0, st, pts, ws, BL);
    launch_next(bx_fan_select_kernel, 1, 1024, 0, st, ws, BL, chunk);
    launch_next(bx_fan_zero_kernel, g, 256, 0, st, ws, BL);
    launch_next(bx_fan_bins_kernel, g, kFiltThreads, 0, st, pts, ws, BL, chunk, stride);
    launch_next(bx_fan_vertex_kernel, g, VT, 0, st, pts, ws, BL);
    launch_next(bx_fan_build_kernel, (unsigned)std::min<int64_t>((int64_t)sms * 2, BL.num_sets), BT, 0, st, pts, ws, BL);
    note_kernels(CH_K_KGON, 6);
    probe_after(CH_K_KGON, st);
    probe_before(CH_K_FILTER, st);
    launch_next(bx_plain_filter_kernel,
                (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)sms * (tuned ? tuned : 3), BL.tiles_max)),
                kFiltThreads, 0, st, pts, ws, L, BL);
    launch_next(bx_hull_filter_kernel, (unsigned)std::min<int64_t>(sms, BL.tiles_max), CT, kQueueSmem + kFanTable, st, pts,
                ws, L, BL, chunk);
    launch_next(bx_layout_kernel, 1, 1024, 0, st, ws, BL);
    note_kernels(CH_K_FILTER, 3);
    probe_after(CH_K_FILTER, st);
    return cudaGetLastError();
}

}  // namespace ch
