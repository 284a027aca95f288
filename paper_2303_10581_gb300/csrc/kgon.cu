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
//    one FMA, which rounds by at most half an ulp of NB, or down to the bin.  A vertex is taken only where its value is at least a margin (1/32;
//    1/8) away from both ends of its bin, so as directions P comes strictly
//    before p and N strictly after it (or N == Q, whose sign is never proven);
//  - consecutive vertices v, w were proven strictly counter-clockwise around
//    c (v != w), less than half a turn apart, so p is in the wedge of (Q, N)
//    or of (P, Q), where strictly left of the edge is the triangle (c, Q, N)
//    or (c, P, Q).  The triangles wind around c once, so c and the
//    triangles' interiors are in the interior of a polygon of hull points;
//  - the quotient needs |dx| + |dy| within [2^-126, 2^126]: the set's box is
//    checked for the upper end, and a point closer to c than 2^-126 is
//    inside the disk around c that is proven inside the fan (the fan is off
//    unless its radius exceeds 2^-60).
// Nothing else is exact: a sign that is not proven keeps the point, and what
// is kept only costs the sort time.  (Sets so small that the products of the
// signs underflow, below 10^-15, or with a box above 2^62 keep all their
// points.)
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

#include "common.cuh"
#include "fan.cuh"
#include "launch.h"
#include "octtest.cuh"

namespace ch {
namespace {

constexpr int CT = 768;                  // threads per block of the filter pass: groups
constexpr int CG = CT / kFiltThreads;    // groups of kFiltThreads, each with its own tiles
constexpr uint32_t kKgonMinS = 1u << 16; // fewer octagon survivors: not worth a pass
constexpr int kFanTable = (kFanBins + 4) * 8;  // vertices, the last again before them and the first two after them (and padding)
constexpr int kQueue = 96;                     // points a warp of the filter pass queues
constexpr int kQueueSmem = CT / 32 * kQueue * 4;
constexpr float kFanMargin = 1.0f / 32.0f;     // of a vertex's pseudo-angle from its bin's ends
constexpr float kFan2Margin = 1.0f / 8.0f;     // second level
static_assert(kFiltItems == 16 && CT % kFiltThreads == 0, "16 items per filter thread");
static_assert(kFanTable + kQueueSmem <= 227 * 1024 - 1024, "table and queues fit a block's shared memory");

// det = (a - c) x (b - c) from the rounded differences, and a bound: a det
// beyond it in magnitude has the exact sign.  Shewchuk's orient2d error
// (orient_f32) is below 2^-22 (|l| + |r|) with l, r the products; |r| <= |l| +
// |det|, so |det| > 2^-20 |l| implies |det| > 2^-22 (|l| + |r|) (2^-140 for
// products that underflow; the fan's box rules out overflow).
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
    __device__ __forceinline__ const float2 *at(uint32_t biased) const { return V + (biased - kBinBias); }
    __device__ __forceinline__ float2 get(const float2 *a, int d) const { return __ldg(a + d); }
};

// Strictly inside the fan, proven (see the top of the file).  F: the
// vertices; before the first comes the last, after the last the first two
// again; d = fl(p - c).  Two vertices are read: in shared memory the reads of
// 32 random bins conflict (six wavefronts each), and a third would bound the
// pass.
template <int NB, class Fan>
__device__ __forceinline__ bool fan_inside(const Fan &F, float2 c, float2 d, float2 p)
{
    const auto a = F.at(fan_bin_biased<NB>(d.x, d.y));   // (a NaN: any vertex; such a point is next to c)
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
template <int NB>
__device__ __forceinline__ int vertex_bin(float dx, float dy, float margin)
{
    const float phi = fan_phi<NB>(dx, dy);
    const float f = __fadd_rd(phi, 0x1p23f);   // 2^23 + the bin
    const float mid = phi - (f - 0x1p23f) - 0.5f;
    return fabsf(mid) <= 0.5f - margin ? (int)(__float_as_uint(f) - kBinBias) : -1;
}

// Whether this call has a fan whose proofs hold (after fan_build_kernel).
__device__ __forceinline__ float fan_rho2(const KgonCtrl *kc) { return __uint_as_float(~kc->rho_inv); }
__device__ __forceinline__ bool fan_ready(const KgonCtrl *kc, const Kgon *g)
{
    return g->ok && !kc->bad && kc->edges >= 3u && fan_rho2(kc) > 0x1p-120f;
}

// ---------------------------------------------------------------------------
// first level: bins and vertices
// ---------------------------------------------------------------------------
// Every stride-th tile, in quarters (1024 points, four a thread) over a
// persistent grid: the bins' farthest points.  The first quarter's points
// take the octagon test as well: it tells how many points survive it (a point
// inside the octagon is an input point all the same, and rarely the
// farthest).  A point whose binary32 distance is clearly below its slot's
// needs no exact key.  Bound by the latency of the points' and then the
// slots' reads, so the next quarter's points are read while this one is
// binned, and few registers keep five blocks on an SM.
constexpr int BI = 4;   // points per thread and step

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
    const float cx = so.cx, cy = so.cy, r2ref = far_ref(so);
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
            live = load_part_ragged<G, BI>(pts, n, base, t, part, cx, cy, px, py);
        }
    };
    if (blockIdx.x < steps) fetch(blockIdx.x);
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
        if (bits_mode) {
            seen += __popc(mine);
            mine &= (uint32_t)at<uint16_t>(ws, L.keep_bits)[tile * kFiltThreads + t] >> (BI * part);
            kept += __popc(mine);
        } else if (part == 0u) {
            seen += __popc(mine);
            uint32_t out;
            oct_decide<BI>(so, qx, qy, out);   // (undecided points count)
            mine &= out;
            kept += __popc(mine);
        }
        if (!__any_sync(0xffffffffu, mine != 0u)) continue;
        uint32_t top[BI];   // the slots' keys (most points do not raise their bin's); ~0: no bin
        int b[BI];
#pragma unroll
        for (int k = 0; k < BI; ++k) {
            b[k] = vertex_bin<kFanBins>(__fsub_rn(qx[k], cx), __fsub_rn(qy[k], cy), kFanMargin);
            top[k] = 0u;
            if (!((mine >> k) & 1u)) b[k] = -1;
            if (b[k] >= 0) top[k] = __ldcg(reinterpret_cast<const uint32_t *>(kc->slot + b[k]) + 1);
        }
#pragma unroll
        for (int k = 0; k < BI; ++k) {
            const float dx = __fsub_rn(qx[k], cx), dy = __fsub_rn(qy[k], cy);
            const float r2 = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
            // (an empty slot's key is a NaN: not below)
            if (b[k] >= 0 && !(r2 - r2ref < __fmaf_rn(r2, -0x1p-20f, key_float(top[k])))) {
                const uint32_t key = far_key(qx[k], qy[k], cx, cy, r2ref);
                if (key >= top[k]) {
                    const uint32_t i = (uint32_t)item_point<G>(tile * kFiltTile, t, BI * part + k);
                    atomicMax(kc->slot + b[k], ((unsigned long long)key << 32) | (uint32_t)~i);
                }
            }
        }
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
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();   // s_w may still be read from an earlier call
    if (lane_id() == 0) s_w[threadIdx.x >> 5] = v;
    __syncthreads();
    int m = -1;
    for (int w = 0; w < BT / 32; ++w) m = max(m, s_w[w]);
    return m;
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
    for (int w = 0; w < (int)warp; ++w) incl = max(incl, s_scan[w]);
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

// In binary32 first (27648 binary64 quotients on 28 SMs would take 15 us),
// in binary64 where that proves nothing: a value in binary32, rounded down.
__device__ __forceinline__ float disk_bound(float cx, float cy, float2 v, float2 w)
{
    const float f = edge_bound<float>(cx, cy, v, w, 0x1p-24f);
    if (f >= 0x1p-100f && f <= 0x1p100f) return f;
    const double d = edge_bound<double>(cx, cy, v, w, 0x1p-53);
    return d < 0.0 ? -1.0f : (d <= 3.0e38 ? __double2float_rd(d) : 3.0e38f);
}

__device__ __forceinline__ bool fan_live(const KgonCtrl *kc, const Octagon *oct, int64_t n)
{
    // (an aborted call, the speculative sweep's candidates, a polygon without
    // edges: the bins pass left no sample)
    const uint32_t sample = kc->sample;
    const float box = __fadd_rn(__fsub_rn(oct->bxh, oct->bxl), __fsub_rn(oct->byh, oct->byl));
    return sample != 0u && (double)kc->inside / sample * (double)n >= (double)kKgonMinS && box < 0x1p62f;
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
// 1), unwrapped; from -+ NB when there is none.
template <int NB>
__device__ __forceinline__ int nearest_bin(const unsigned long long *slot, int from, int dir)
{
    const int lane = (int)lane_id();
    for (int k = 0; k < NB; k += 32) {
        const int j = dir > 0 ? from + k + lane : from - 1 - k - lane;
        const int w = j < 0 ? j + NB : (j >= NB ? j - NB : j);
        const uint32_t m = __ballot_sync(0xffffffffu, __ldcg(slot + w) != 0ull);
        if (m) return dir > 0 ? from + k + __ffs(m) - 1 : from - k - __ffs(m);
    }
    return dir > 0 ? from + NB : from - NB;
}

// Bins [b0, b0 + VB) of a fan with NB bins; point(i) reads input point i
// (clamped to the input); V receives the vertices, x = NaN for none.  False
// when there are no samples outside the range (no fan).
template <int NB, class Point>
__device__ __forceinline__ bool make_vertices(VertexSmem &sm, const unsigned long long *slot, int b0, float2 c, Point point,
                                              float2 *V)
{
    const int lane = (int)lane_id();
    const uint32_t lt = (1u << lane) - 1u;
    const int pb = nearest_bin<NB>(slot, b0, -1), nb = nearest_bin<NB>(slot, b0 + VB, 1);
    if (pb <= b0 + VB - 1 - NB || nb >= b0 + NB) return false;   // (only this range has samples)
    bool has[VB / 32];
    float2 own[VB / 32];
    int len = 1;
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
        const int j = lane ? nb : pb;
        const int w = j < 0 ? j + NB : (j >= NB ? j - NB : j);
        const int at = lane ? len : 0;
        sm.p[0][at] = point(~(uint32_t)__ldcg(slot + w));
        sm.bin[0][at] = j;
    }
    ++len;
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
        int lo = 0, hi = len - 1;   // last entry at or before bin b (entry 0 is before the range, the last after it)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (sm.bin[cur][mid] <= b) lo = mid;
            else hi = mid;
        }
        const float2 Lp = sm.p[cur][lo], Rp = sm.p[cur][lo + 1];
        float2 v = own[h];
        bool ok = has[h];
        if (sm.bin[cur][lo] != b) {
            const float lx = Lp.x - c.x, ly = Lp.y - c.y, ex = Rp.x - Lp.x, ey = Rp.y - Lp.y;
            const float num = lx * ey - ly * ex;
            const float own_den = (v.x - c.x) * ey - (v.y - c.y) * ex;
            if (!ok || num > own_den * (1.0f + 0x1p-18f)) {   // (own_den > 0: the sample is on the chord's side of c)
                const float2 d = fan_direction<NB>((float)b + 0.5f);
                const float s = num / (d.x * ey - d.y * ex) * (1.0f - 0x1p-20f);
                const float2 q = make_float2(__fmaf_rn(s, d.x, c.x), __fmaf_rn(s, d.y, c.y));
                if (fabsf(q.x) <= 3.0e38f && fabsf(q.y) <= 3.0e38f &&
                    vertex_bin<NB>(__fsub_rn(q.x, c.x), __fsub_rn(q.y, c.y), kFanMargin) == b &&
                    orient(Lp.x, Lp.y, Rp.x, Rp.y, q.x, q.y) > 0 && orient(Lp.x, Lp.y, Rp.x, Rp.y, c.x, c.y) > 0) {
                    v = q;
                    ok = true;
                }
            }
        }
        V[b] = ok ? v : make_float2(__int_as_float(0x7fc00000), 0.0f);
    }
    return true;
}

__global__ void __launch_bounds__(VT) fan_vertex_kernel(const float *__restrict__ pts, int64_t n, void *ws, Layout L)
{
    kernel_entry();
    __shared__ VertexSmem sm[VT / 32];
    const Octagon *oct = at<Octagon>(ws, L.oct);
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    if (!fan_live(kc, oct, n)) return;
    const int warp = (int)(threadIdx.x >> 5);
    const int b0 = (int)(blockIdx.x * (VT / 32) + warp) * VB;
    const bool ok = make_vertices<kFanBins>(
        sm[warp], kc->slot, b0, make_float2(oct->cx, oct->cy),
        [&](uint32_t i) { return input_point(pts, (int64_t)i < n ? i : 0u); }, at<Kgon>(ws, L.kgon)->raw);
    if (!ok && lane_id() == 0) kc->bad = 1u;
}

__global__ void __launch_bounds__(BT) fan_build_kernel(int64_t n, void *ws, Layout L)
{
    kernel_entry();
    __shared__ int s_w[BT / 32];
    __shared__ int s_scan[BT / 32];
    const Octagon *oct = at<Octagon>(ws, L.oct);
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    Kgon *g = at<Kgon>(ws, L.kgon);
    const uint32_t tid = threadIdx.x;
    const bool live = fan_live(kc, oct, n) && !(kc->bad & 1u);   // (bit 1 is set below)
    const int b = (int)(blockIdx.x * BT + tid);
    int src = -1;
    if (live) src = vertex_source([&](int j) { return g->raw[j].x == g->raw[j].x; }, s_w, s_scan);   // block-uniform
    if (src < 0) {
        if (blockIdx.x == 0 && tid == 0) g->ok = 0u;
        return;
    }
    const float cx = oct->cx, cy = oct->cy;
    const float2 v = g->raw[src], next = g->raw[next_bin(b)];
    g->v[b] = v;
    // the next bin's vertex: its own point, or this one's again
    const float2 w = next.x == next.x ? next : v;
    float r = __int_as_float(0x7f800000);
    const bool edge = v.x != w.x || v.y != w.y;
    bool bad = false;
    if (edge) {
        r = disk_bound(cx, cy, v, w);
        bad = r < 0.0f;
    }
    uint32_t inv = ~__float_as_uint(fmaxf(r, 0.0f));
    inv = __reduce_max_sync(0xffffffffu, inv);
    const uint32_t edges = __popc(__ballot_sync(0xffffffffu, edge));
    bad = __any_sync(0xffffffffu, bad);
    if (lane_id() == 0) {
        atomicMax(&kc->rho_inv, inv);
        if (edges) atomicAdd(&kc->edges, edges);
        if (bad) atomicOr(&kc->bad, 2u);
    }
    if (blockIdx.x == 0 && tid == 0) {
        g->cx = cx;
        g->cy = cy;
        g->ok = 1u;
    }
}

// ---------------------------------------------------------------------------
// the filter pass
// ---------------------------------------------------------------------------
// The warp's kept points (mask: this lane's items; get(q): the point and its
// index) to the end of the survivor list.
template <class Get>
__device__ __forceinline__ void append_survivors(uint32_t mask, void *ws, const Layout &L, Get get)
{
    const uint32_t lane = lane_id(), c = __popc(mask);
    if (!__any_sync(0xffffffffu, c != 0u)) return;
    uint32_t incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl += u;
    }
    uint32_t pos = 0;
    if (lane == 31) pos = atomicAdd(&at<Ctrl>(ws, L.ctrl)->surv_count, incl);
    pos = __shfl_sync(0xffffffffu, pos, 31) + incl - c;
#pragma unroll 1
    for (; mask; mask &= mask - 1u, ++pos) {
        uint32_t i;
        const float2 p = get(__ffs(mask) - 1, i);
        at<uint32_t>(ws, L.keys[0])[pos] = ord_key(p.x);
        at<unsigned long long>(ws, L.pay[0])[pos] = ((unsigned long long)ord_key(p.y) << 32) | i;
    }
}

// The speculative sweep's candidates (extremes.cu; every other point is
// proven inside the octagon): a warp per slice, the exact test.
__device__ __forceinline__ uint32_t filter_candidates(const OctSmem &so, void *ws, const Layout &L)
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
                keep = keep_point<false>(so, p.x, p.y);
            }
            mine += keep ? 1u : 0u;
            append_survivors(keep ? 1u : 0u, ws, L, [&](int, uint32_t &i) {
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

struct FanView {
    bool test;   // candidates
    SharedFan F;
    float2 c;
};

// An index with this bit (n < 2^30) is a point the octagon's forms may have
// left undecided: the exact test first, and then the fan test.
constexpr uint32_t kUnsettled = 0x80000000u;

// Whether point p (i: its index and kUnsettled) survives; octs counts the
// octagon survivors among the unsettled ones.
__device__ __forceinline__ bool settle(const OctSmem &so, const FanView &f, bool fan, uint32_t i, float2 p, uint32_t &octs)
{
    bool keep = true;
    if (i & kUnsettled) {
        keep = keep_point<false>(so, p.x, p.y);
        octs += keep ? 1u : 0u;
    }
    if (f.test || ((i & kUnsettled) && fan)) keep = keep && !fan_inside<kFanBins>(f.F, f.c, sub2(p, f.c), p);
    return keep;
}

// The last (up to) 32 points of the queue: the survivors to the list.
__device__ __forceinline__ void queue_drain(PointQueue &q, const OctSmem &so, const FanView &f, bool fan,
                                            const float *__restrict__ pts, void *ws, const Layout &L, uint32_t &octs)
{
    const uint32_t lane = lane_id(), m = min(q.n, 32u);
    q.n -= m;
    bool keep = lane < m;
    const uint32_t e = q.i[q.n + (keep ? lane : 0u)], i = e & ~kUnsettled;
    const float2 p = input_point(pts, i);
    __syncwarp();   // the slots may be filled again
    if (keep) keep = settle(so, f, fan, e, p, octs);
    const uint32_t b = __ballot_sync(0xffffffffu, keep);
    if (!b) return;
    uint32_t pos = 0;
    if (lane == 0) pos = atomicAdd(&at<Ctrl>(ws, L.ctrl)->surv_count, (uint32_t)__popc(b));
    pos = __shfl_sync(0xffffffffu, pos, 0) + __popc(b & ((1u << lane) - 1u));
    if (keep) {
        at<uint32_t>(ws, L.keys[0])[pos] = ord_key(p.x);
        at<unsigned long long>(ws, L.pay[0])[pos] = ((unsigned long long)ord_key(p.y) << 32) | i;
    }
}

// The tiles go in contiguous ranges to groups of kFiltThreads threads; a
// thread tests its 16 points of a tile eight at a time: the octagon's affine
// forms, then (fan) the fan test, branch-free -- or, in a warp where the disk
// holds most points, the disk test, the others going to the queue.
// bits_mode: a second polygon has refined the count pass's keep bits, which
// then stand for the octagon test.
// One block of 1024 threads per SM: the vertices and the queues take its
// shared memory.  Bound by issue and the vertices' bank conflicts on
// circle-like sets (about 18 instructions for the octagon, 27 for the fan and
// two vertex reads per point) and by HBM on others.  Testing and writing in
// one pass replaces a count pass, a fan pass and a scatter that each read the
// points again: 274 + 455 + 214 us on 10^8 points of the unit circle.
template <int G>
__global__ void __launch_bounds__(CT, 1) hull_filter_kernel(const float *__restrict__ pts, uint32_t n, void *ws, Layout L,
                                                            int has_fan, int use_bits, const int32_t *kdev)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ OctSmem so;
    __shared__ uint32_t s_oct;
    const Octagon *oct = at<Octagon>(ws, L.oct);
    if (oct->abort) return;
    KgonCtrl *kc = at<KgonCtrl>(ws, L.kgon_ctrl);
    fill_octagon(so, oct);
    if (threadIdx.x == 0) s_oct = 0u;
    const Kgon *g = at<Kgon>(ws, L.kgon);
    const bool fan = has_fan && !oct->spec && fan_ready(kc, g);
    float2 *sv = reinterpret_cast<float2 *>(smem_raw + kQueueSmem) + 1;
    if (fan) {
        for (int i = threadIdx.x; i < kFanBins; i += CT) sv[i] = __ldg(g->v + i);
        if (threadIdx.x == 0) {
            sv[-1] = __ldg(g->v + kFanBins - 1);
            sv[kFanBins] = __ldg(g->v);
            sv[kFanBins + 1] = __ldg(g->v + 1);
        }
    }
    __syncthreads();
    uint32_t octs = 0;   // octagon survivors of this thread
    if (oct->spec) {
        octs = filter_candidates(so, ws, L);
    } else {
        const bool bits_mode = use_bits && (!kdev || *kdev != 8);
        const float2 c = make_float2(so.cx, so.cy);
        const SharedFan F(sv);
        const uint32_t warp = threadIdx.x >> 5, lt = (1u << lane_id()) - 1u;
        PointQueue q{reinterpret_cast<uint32_t *>(smem_raw) + warp * kQueue, 0u};
        // r2 < rho2t proves |p - c|^2 < rho^2 (2^-20 covers the rounding of r2)
        const float rho2t = fan ? __fmul_rd(fan_rho2(kc), 1.0f - 0x1p-20f) : 0.0f;
        bool use_disk = fan;   // (then the queue holds candidates)
        const bool edges = !bits_mode && so.has_edges;
        const uint32_t ntiles = (n + kFiltTile - 1) / kFiltTile;   // (n < 2^30)
        const uint32_t t = threadIdx.x % kFiltThreads, gi = blockIdx.x * CG + threadIdx.x / kFiltThreads;
        const uint32_t per = (ntiles + gridDim.x * CG - 1) / (gridDim.x * CG);
        const uint32_t t1 = min(ntiles, (gi + 1) * per);
        for (uint32_t tile = gi * per; tile < t1; ++tile) {
            const uint32_t base = tile * kFiltTile;
            if (t == 0 && tile + 1 < t1) {   // the next tile streams into L2 meanwhile
                const float *next = pts + 2 * (size_t)(base + kFiltTile);
                if ((reinterpret_cast<uintptr_t>(next) & 15u) == 0)
                    bulk_prefetch_l2(next, (min((uint32_t)kFiltTile, n - base - kFiltTile) * 8u) & ~15u);
            }
            // kept: octagon survivors; drop: those of them inside the disk or
            // the fan; near: some may be undecided, and all of this lane's are
            // settled when they leave the queue (rare: next to the octagon)
            uint32_t kept = 0xffffu, drop = 0;
            bool near = false;
            if (bits_mode) kept = at<uint16_t>(ws, L.keep_bits)[tile * kFiltThreads + t];
#pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                float px[8], py[8];
                if (base + kFiltTile <= n) load_part<G, 8>(pts, base, t, half, px, py);
                else kept &= ~(0xffu << (8 * half)) |
                             load_part_ragged<G, 8>(pts, n, base, t, half, c.x, c.y, px, py) << (8 * half);
                if (edges) {
                    uint32_t out8;
                    near |= oct_decide<8>(so, px, py, out8);
                    kept &= ~(0xffu << (8 * half)) | out8 << (8 * half);
                }
                if (!fan) continue;
                uint32_t in = 0;
                if (use_disk) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        const float dx = __fsub_rn(px[k], c.x), dy = __fsub_rn(py[k], c.y);
                        if (__fmaf_rn(dx, dx, __fmul_rn(dy, dy)) < rho2t) in |= 1u << k;
                    }
                } else if (__any_sync(0xffffffffu, ((kept >> (8 * half)) & 0xffu) != 0u)) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        if (k % 4 == 0) asm volatile("" ::: "memory");   // four points at a time (more would spill)
                        const float2 p = make_float2(px[k], py[k]);
                        if (fan_inside<kFanBins>(F, c, sub2(p, c), p)) in |= 1u << k;
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
                    while (q.n) queue_drain(q, so, FanView{true, F, c}, fan, pts, ws, L, octs);
                    if (!near) octs -= __popc(kept);
                    use_disk = false;
                    --tile;   // once more, with the fan
                    continue;
                }
            }
            if (total == 0u) continue;
            const FanView f{use_disk, F, c};
            if (q.n + total <= (uint32_t)kQueue) {
                uint32_t at = q.n;
                q.n += total;
                // (a ballot per round: a lane has few points)
                while (at < q.n) {
                    const uint32_t m = __ballot_sync(0xffffffffu, live != 0u);
                    if (live)
                        q.i[at + __popc(m & lt)] = (uint32_t)item_point<G>(base, t, __ffs(live) - 1) | (near ? kUnsettled : 0u);
                    live &= live - 1u;
                    at += __popc(m);
                }
                __syncwarp();
                while (q.n >= 32u) queue_drain(q, so, f, fan, pts, ws, L, octs);
            } else {   // many at once: each lane its own, the points read again
                if (f.test || near) {
#pragma unroll 1
                    for (uint32_t m = live; m; m &= m - 1u) {
                        const uint32_t i = (uint32_t)item_point<G>(base, t, __ffs(m) - 1);
                        if (!settle(so, f, fan, i | (near ? kUnsettled : 0u), input_point(pts, i), octs))
                            live &= ~(m & (0u - m));
                    }
                }
                append_survivors(live, ws, L, [&](int k, uint32_t &i) {
                    const int64_t j = item_point<G>(base, t, k);
                    i = (uint32_t)j;
                    return input_point(pts, j);
                });
            }
        }
        while (q.n) queue_drain(q, so, FanView{use_disk, F, c}, fan, pts, ws, L, octs);
    }
    octs = __reduce_add_sync(0xffffffffu, octs);
    if (lane_id() == 0 && octs) atomicAdd(&s_oct, octs);
    __syncthreads();
    if (threadIdx.x == 0 && s_oct) atomicAdd(&kc->s_oct, s_oct);
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
//                       one for an empty sub-bin, cyclically); the proof
//                       that consecutive ones are counter-clockwise
//  fan2_test_kernel     the test of every survivor; the kept ones go to the
//                       sort's second buffers, which the sort then reads
// ---------------------------------------------------------------------------
constexpr int F2T = 256;
constexpr int F2I = 8;   // survivors per thread and step of the test
static_assert(kFan2Bins % BT == 0, "sub-bins split evenly over the build blocks");

__device__ __forceinline__ float2 surv_point(const uint32_t *keys, const unsigned long long *pay, uint32_t i)
{
    return make_float2(key_float(keys[i]), key_float((uint32_t)(pay[i] >> 32)));
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
    const float cx = g->cx, cy = g->cy, r2ref = far_ref(*oct);
    for (uint32_t i = blockIdx.x * F2T + threadIdx.x; i < m; i += gridDim.x * F2T) {
        const float2 p = surv_point(keys, pay, i);
        const int b = vertex_bin<kFan2Bins>(__fsub_rn(p.x, cx), __fsub_rn(p.y, cy), kFan2Margin);
        if (b < 0) continue;
        const unsigned long long v = ((unsigned long long)far_key(p.x, p.y, cx, cy, r2ref) << 32) | (uint32_t)~i;
        if (v > __ldcg(&slot[b])) atomicMax(&slot[b], v);   // the read only saves atomics
    }
}

// One thread per sub-bin, as fan_build_kernel; the table's ends are repeated
// at V[-1] and V[kFan2Bins], V[kFan2Bins + 1].
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
    float2 *V = at<float2>(ws, L.fan2_v) + 1;
    const int b = (int)(blockIdx.x * BT + threadIdx.x);
    const int src = vertex_source([&](int j) { return slot[j] != 0ull; }, s_w, s_scan);
    if (src < 0) {   // no survivor reached a slot: keep everything
        if (threadIdx.x == 0) f2->bad = 1u;
        return;
    }
    const float2 v = surv_point(keys, pay, ~(uint32_t)slot[src]);
    V[b] = v;
    if (b < 2) V[kFan2Bins + b] = v;
    if (b == kFan2Bins - 1) V[-1] = v;
    const unsigned long long nextp = slot[next_bin<kFan2Bins>(b)];
    const float2 w = nextp != 0ull ? surv_point(keys, pay, ~(uint32_t)nextp) : v;
    const bool edge = v.x != w.x || v.y != w.y;
    // c strictly left of v -> w, proven in binary32 or exactly
    const bool bad = edge && orient(v.x, v.y, w.x, w.y, g->cx, g->cy) <= 0;
    const uint32_t edges = __popc(__ballot_sync(0xffffffffu, edge));
    if (lane_id() == 0 && edges) atomicAdd(&f2->edges, edges);
    if (bad) f2->bad = 1u;
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
    const bool test = !f2->bad && f2->edges >= 3u;
    const Kgon *g = at<Kgon>(ws, L.kgon);
    const float2 c = make_float2(g->cx, g->cy);
    const GlobalFan F{at<float2>(ws, L.fan2_v) + 1};
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
                const float2 p = make_float2(key_float(kv[k]), key_float((uint32_t)(pv[k] >> 32)));
                if (fan_inside<kFan2Bins>(F, c, sub2(p, c), p)) in |= 1u << k;
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
        launch_next(fan_bins_kernel<G>, (unsigned)bb, kFiltThreads, 0, st, pts, (uint32_t)n, ws, L, (uint32_t)stride, use_bits, kdev);
        launch_next(fan_vertex_kernel, kFanBins / (VB * VT / 32), VT, 0, st, pts, n, ws, L);
        launch_next(fan_build_kernel, kFanBins / BT, BT, 0, st, n, ws, L);
        note_kernels(CH_K_KGON, 3);
        probe_after(CH_K_KGON, st);
    }
    probe_before(CH_K_FILTER, st);
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(ceil_div(ntiles, (int64_t)CG), sms));
    launch_next(hull_filter_kernel<G>, (unsigned)grid, CT, kQueueSmem + (has_fan ? kFanTable : 0), st, pts, (uint32_t)n, ws, L, has_fan, use_bits, kdev);
    note_kernels(CH_K_FILTER, 1);
    probe_after(CH_K_FILTER, st);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || L.fan2_bins == 0) return e;   // (a set too small for the second level)
    probe_before(CH_K_KGON, st);
    const int lg = tune_value(CH_TUNE_FAN2_MIN_LOG2);
    launch_next(fan2_max_kernel, sms * 8, F2T, 0, st, ws, L, lg ? (uint32_t)(1ull << lg) : kFan2MinS);
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
        int64_t bc = 0;
        cudaError_t e = launch_filter_count(pts, n, kg->kdev, ws, L, &bc, st);
        if (e == cudaSuccess) e = launch_kx_sv(pts, n, kg->dirs, kg->kdev, kg->K, kg->ext_out, ws, L, bc, st);
        if (e != cudaSuccess) return e;
    }
    const int32_t *kdev = bits ? kg->kdev : nullptr;
    return (reinterpret_cast<uintptr_t>(pts) & 15u) == 0
               ? launch_hull_filter_g<2>(pts, n, ws, L, bits ? 1 : 0, kdev, st)
               : launch_hull_filter_g<1>(pts, n, ws, L, bits ? 1 : 0, kdev, st);
}

namespace {

// ---------------------------------------------------------------------------
// many sets (ch_hull_batched): the same fan for every set with at least
// kKgonMinS octagon survivors, between the batched count pass and its scan
// ---------------------------------------------------------------------------
constexpr int kFanSmem = kFanBins * 8;
constexpr int FT = 512;                  // threads per block of the bins pass
constexpr int FITEMS = 8;                // points per thread per tile there
// The signs orient_f32 certifies, as two flags (det > bound, -det > bound;
// neither when undecided or when the terms may have overflowed): the same
// arithmetic on the rounded differences a - c and b - c, without turning
// the flags into an integer.
struct Sgn {
    bool pos, neg;
};
__device__ __forceinline__ Sgn sgn_ref(float acx, float acy, float bcx, float bcy)
{
    const float detleft = __fmul_rn(acx, bcy);
    const float detright = __fmul_rn(acy, bcx);
    const float det = __fsub_rn(detleft, detright);
    const float detsum = __fadd_rn(fabsf(detleft), fabsf(detright));
    const float eb = __fmaf_ru(detsum, 2.384185791015625e-07f /* 2^-22 */, 7.174648137343064e-43f /* 2^-140 */);
    const bool ok = detsum <= 3.0e38f;
    return {ok && det > eb, ok && -det > eb};
}

template <int NB = kFanBins>
__device__ __forceinline__ int fan_signs_f32(const float2 *V, float cx, float cy, float px, float py)
{
    const float dx = __fsub_rn(px, cx), dy = __fsub_rn(py, cy);
    const int b = (int)min(fan_bin<NB>(dx, dy), NB - 1u);
    const float2 v = V[b];
    const Sgn o = sgn_ref(__fsub_rn(v.x, cx), __fsub_rn(v.y, cy), dx, dy);                   // (v, p, c)
    const float2 w = V[o.pos ? next_bin<NB>(b) : prev_bin<NB>(b)];
    const Sgn e1 = sgn_ref(__fsub_rn(v.x, px), __fsub_rn(v.y, py), __fsub_rn(w.x, px), __fsub_rn(w.y, py));   // (v, w, p)
    const Sgn e2 = sgn_ref(dx, dy, __fsub_rn(w.x, cx), __fsub_rn(w.y, cy));                   // (p, w, c)
    // inside: the three signs certified equal (strictly inside the triangle
    // on o's side); outside: one of the edges certified opposite to o
    const bool in = (o.pos && e1.pos && e2.pos) || (o.neg && e1.neg && e2.neg);
    const bool out = (o.pos && (e1.neg || e2.neg)) || (o.neg && (e1.pos || e2.pos));
    return in ? 1 : (out ? 0 : 2);
}

template <int NB = kFanBins>
__device__ __noinline__ bool fan_inside_exact(const float2 *V, float cx, float cy, float px, float py)
{
    const int b = (int)min(fan_bin<NB>(px - cx, py - cy), NB - 1u);
    const float2 v = V[b];
    const int o = orient(cx, cy, v.x, v.y, px, py);
    if (o == 0) return false;
    const float2 w = V[o > 0 ? next_bin<NB>(b) : prev_bin<NB>(b)];
    return orient(v.x, v.y, w.x, w.y, px, py) == o && orient(w.x, w.y, cx, cy, px, py) == o;
}

constexpr int kBxBinStride = 2;   // built-in: the bins see every 2nd tile of a set (1 and 4 measured slower overall)

// One block: numbers the sets that get a fan and lays out the refine's
// work items (runs of up to kBxFanChunk tiles of one such set).
__global__ void __launch_bounds__(1024) bx_fan_select_kernel(void *ws, Layout L, BatchLayout BL, uint32_t chunk)
{
    kernel_entry();
    __shared__ uint32_t s_w[2][32];
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint32_t *soct = at<uint32_t>(ws, BL.soct);
    const uint32_t *nonfin = at<uint32_t>(ws, BL.nonfinite);
    int32_t *fan_id = at<int32_t>(ws, BL.fan_id);
    uint32_t *fan_set = at<uint32_t>(ws, BL.fan_set);
    uint2 *items = at<uint2>(ws, BL.fan_items);
    const int64_t B = BL.num_sets;
    const bool off = bc->abort != 0;
    const uint32_t lane = lane_id(), warp = threadIdx.x >> 5;
    const int64_t per = ceil_div(B, (int64_t)blockDim.x);
    const int64_t b0 = min((int64_t)threadIdx.x * per, B), b1 = min(b0 + per, B);
    auto wants = [&](int64_t b) {
        return !off && soct[b] >= kKgonMinS && !octs[b].abort && octs[b].has_edges && nonfin[b] == 0u;
    };
    uint32_t nf = 0, ni = 0;
    for (int64_t b = b0; b < b1; ++b)
        if (wants(b)) {
            ++nf;
            ni += (uint32_t)ceil_div((int64_t)sets[b].ntiles, (int64_t)chunk);
        }
    uint32_t inf = nf, ini = ni;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(0xffffffffu, inf, o), c = __shfl_up_sync(0xffffffffu, ini, o);
        if (lane >= (uint32_t)o) {
            inf += a;
            ini += c;
        }
    }
    if (lane == 31) {
        s_w[0][warp] = inf;
        s_w[1][warp] = ini;
    }
    __syncthreads();
    uint32_t bf = 0, bi = 0, tf = 0, ti = 0;
    for (uint32_t w = 0; w < blockDim.x / 32; ++w) {
        if (w < warp) {
            bf += s_w[0][w];
            bi += s_w[1][w];
        }
        tf += s_w[0][w];
        ti += s_w[1][w];
    }
    uint32_t f = bf + inf - nf, it = bi + ini - ni;
    for (int64_t b = b0; b < b1; ++b) {
        if (wants(b) && f < (uint32_t)BL.max_fan) {
            fan_id[b] = (int32_t)f;
            fan_set[f] = (uint32_t)b;
            for (uint32_t c = 0; c < sets[b].ntiles; c += chunk) items[it++] = make_uint2(f, sets[b].tile_base + c);
            ++f;
        } else {
            fan_id[b] = -1;
        }
    }
    if (threadIdx.x == 0) {
        bc->nfan = min(tf, (uint32_t)BL.max_fan);
        bc->nitems = min(ti, (uint32_t)BL.max_items);
    }
}

// Per work item, every kBxBinStride-th tile (counted from the set's first):
// each point's bin around the set's box centre, packed (far_key << 32 |
// ~index) into the fan's global slots by atomicMax (the read first saves
// most atomics).
__global__ void __launch_bounds__(FT) bx_fan_bins_kernel(const float *__restrict__ pts, void *ws, Layout L,
                                                         BatchLayout BL, uint32_t chunk, uint32_t stride)
{
    kernel_entry();
    const BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint32_t *fan_set = at<uint32_t>(ws, BL.fan_set);
    const uint2 *items = at<uint2>(ws, BL.fan_items);
    unsigned long long *slots = at<unsigned long long>(ws, BL.fan_slot);
    const uint32_t nitems = bc->nitems;
    for (uint32_t w = blockIdx.x; w < nitems; w += gridDim.x) {
        const uint2 item = items[w];
        const uint32_t b = fan_set[item.x];
        const SetInfo &S = sets[b];
        const float cx = octs[b].cx, cy = octs[b].cy, r2ref = far_ref(octs[b]);
        const float2 *p2 = reinterpret_cast<const float2 *>(pts) + S.pt_begin;
        unsigned long long *sl = slots + (size_t)item.x * kFanBins;
        const uint32_t tend = min(item.y + chunk, S.tile_base + S.ntiles);
        for (uint32_t t = item.y; t < tend; ++t) {
            if ((t - S.tile_base) % stride) continue;
            const int64_t lo = (int64_t)(t - S.tile_base) * kFiltTile, hi = min(lo + kFiltTile, S.n);
            float2 p[FITEMS];
#pragma unroll
            for (int r = 0; r < FITEMS; ++r) {
                const int64_t i = lo + r * FT + threadIdx.x;
                p[r] = i < hi ? __ldg(p2 + i) : make_float2(0.0f, 0.0f);
            }
#pragma unroll
            for (int r = 0; r < FITEMS; ++r) {
                const int64_t i = lo + r * FT + threadIdx.x;
                if (i < hi) {
                    const float dx = p[r].x - cx, dy = p[r].y - cy;
                    const int bin = (int)min(fan_bin(dx, dy), kFanBins - 1u);
                    const unsigned long long v =
                        ((unsigned long long)far_key(p[r].x, p[r].y, cx, cy, r2ref) << 32) | (uint32_t)~(uint32_t)i;
                    if (v > __ldcg(sl + bin)) atomicMax(sl + bin, v);
                }
            }
        }
    }
}

// One block per fan (grid-stride): the exact centre check against the
// set's octagon, then every bin's vertex (the sampled point of the last
// non-empty bin at or before it, cyclically), and the slots are left zero
// for the next call.  Thread t owns the kBinsPerThread consecutive bins
// from t * kBinsPerThread: a scan in registers, one block scan of the
// threads' last non-empty bins.
constexpr int kBinsPerThread = kFanBins / BT;
static_assert(kFanBins % BT == 0, "bins split evenly over the threads");

__global__ void __launch_bounds__(BT) bx_fan_build_kernel(const float *__restrict__ pts, void *ws, Layout L,
                                                          BatchLayout BL)
{
    kernel_entry();
    __shared__ int s_w[BT / 32];
    __shared__ int s_ok;
    const BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const Octagon *octs = at<Octagon>(ws, BL.octs);
    const uint32_t *fan_set = at<uint32_t>(ws, BL.fan_set);
    uint32_t *fan_ok = at<uint32_t>(ws, BL.fan_ok);
    float2 *fan_c = at<float2>(ws, BL.fan_c);
    unsigned long long *slots = at<unsigned long long>(ws, BL.fan_slot);
    float2 *verts = at<float2>(ws, BL.fan_v);
    const uint32_t tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
    const uint32_t nfan = bc->nfan;
    for (uint32_t k = blockIdx.x; k < nfan; k += gridDim.x) {
        const uint32_t b = fan_set[k];
        const Octagon &oct = octs[b];
        const float cx = oct.cx, cy = oct.cy;
        unsigned long long *sl = slots + (size_t)k * kFanBins + (size_t)tid * kBinsPerThread;
        float2 *V = verts + (size_t)k * kFanBins + (size_t)tid * kBinsPerThread;
        const float2 *p2 = reinterpret_cast<const float2 *>(pts) + sets[b].pt_begin;
        const int64_t nb = sets[b].n;
        __syncthreads();   // shared words of the previous fan have been read
        if (tid == 0) s_ok = 1;
        __syncthreads();
        if (tid < 8 && ((oct.valid >> tid) & 1u) && orient(oct.ax[tid], oct.ay[tid], oct.bx[tid], oct.by[tid], cx, cy) <= 0)
            s_ok = 0;
        // this thread's bins: the point index of each non-empty one, ~0u empty
        uint32_t idx[kBinsPerThread];
        int mylast = -1;
#pragma unroll
        for (int j = 0; j < kBinsPerThread; ++j) {
            const unsigned long long v = __ldcg(sl + j);
            idx[j] = v != 0ull ? ~(uint32_t)v : ~0u;
            if (v != 0ull) mylast = j;
        }
        // the last non-empty bin of the threads before this one (exclusive
        // max-scan over thread order), and the last overall (wrap-around)
        int incl = mylast >= 0 ? (int)(tid * kBinsPerThread) + mylast : -1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= (uint32_t)o) incl = max(incl, u);
        }
        int excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) excl = -1;
        if (lane == 31) s_w[warp] = incl;
        __syncthreads();
        int before = -1, last = -1;
        for (uint32_t w = 0; w < BT / 32; ++w) {
            if (w < warp) before = max(before, s_w[w]);
            last = max(last, s_w[w]);
        }
        before = max(before, excl);
        const bool live = s_ok && last >= 0;
        if (live) {
            // the vertex index of a bin with no sample: that of the last
            // non-empty bin before it (cyclically); it lies in another
            // thread's range, read from the slots (not zeroed yet)
            int cur = before >= 0 ? before : last;
            uint32_t ci = ~(uint32_t)__ldcg(slots + (size_t)k * kFanBins + cur);
#pragma unroll
            for (int j = 0; j < kBinsPerThread; ++j) {
                if (idx[j] != ~0u) ci = idx[j];
                V[j] = __ldg(p2 + ((int64_t)ci < nb ? ci : 0u));
            }
        }
        __syncthreads();   // every read of the slots is done
#pragma unroll
        for (int j = 0; j < kBinsPerThread; ++j) sl[j] = 0ull;
        if (tid == 0) {
            fan_ok[k] = live ? 1u : 0u;
            fan_c[k] = make_float2(cx, cy);
        }
    }
}

// Persistent blocks take work items by ticket; the 27648 vertices of the
// item's fan are loaded into shared memory when the fan changes (items of
// one fan are consecutive).  The four groups of kFiltThreads threads share
// the item's tiles; thread t holds the 16 keep bits of count-pass thread t
// (point lo + r * 256 + t for bit r).  Kept points strictly inside the fan
// lose their bit, and the tile's count drops by the number removed.
__global__ void __launch_bounds__(CT, 1) bx_fan_refine_kernel(const float *__restrict__ pts, void *ws, Layout L,
                                                              BatchLayout BL, uint32_t chunk)
{
    kernel_entry();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sv = reinterpret_cast<float2 *>(smem_raw);   // kFanBins vertices
    __shared__ uint32_t s_item;
    BatchCtrl *bc = at<BatchCtrl>(ws, BL.bctrl);
    const SetInfo *sets = at<SetInfo>(ws, BL.sets);
    const uint32_t *fan_set = at<uint32_t>(ws, BL.fan_set);
    const uint32_t *fan_ok = at<uint32_t>(ws, BL.fan_ok);
    const float2 *fan_c = at<float2>(ws, BL.fan_c);
    const float2 *verts = at<float2>(ws, BL.fan_v);
    const uint2 *items = at<uint2>(ws, BL.fan_items);
    uint16_t *bits = at<uint16_t>(ws, L.keep_bits);
    unsigned long long *status = at<unsigned long long>(ws, L.filt_status);
    const uint32_t nitems = bc->nitems;
    const uint32_t grp = threadIdx.x / kFiltThreads, t = threadIdx.x % kFiltThreads, lane = lane_id();
    int64_t cur = -1;
    for (;;) {
        __syncthreads();   // s_item of the previous item has been read
        if (threadIdx.x == 0) s_item = atomicAdd(&bc->fan_ticket, 1u);
        __syncthreads();
        const uint32_t w = s_item;
        if (w >= nitems) break;
        const uint2 item = items[w];
        if (!fan_ok[item.x]) continue;   // block-uniform
        if ((int64_t)item.x != cur) {
            const float4 *src = reinterpret_cast<const float4 *>(verts + (size_t)item.x * kFanBins);
            float4 *dst = reinterpret_cast<float4 *>(sv);
            for (int i = threadIdx.x; i < kFanBins / 2; i += CT) dst[i] = __ldg(src + i);
            __syncthreads();
            cur = item.x;
        }
        const SetInfo &S = sets[fan_set[item.x]];
        const float2 c = fan_c[item.x];
        const float2 *p2 = reinterpret_cast<const float2 *>(pts) + S.pt_begin;
        const uint32_t tend = min(item.y + chunk, S.tile_base + S.ntiles);
        for (uint32_t tile = item.y + grp; tile < tend; tile += CG) {
            const int64_t lo = (int64_t)(tile - S.tile_base) * kFiltTile;
            const uint32_t kb = bits[(size_t)tile * kFiltThreads + t];
            uint32_t in = 0;
            if (kb) {
                float2 p[kFiltItems];
#pragma unroll
                for (int r = 0; r < kFiltItems; ++r)
                    p[r] = ((kb >> r) & 1u) ? __ldcs(p2 + lo + r * kFiltThreads + t) : make_float2(0.0f, 0.0f);
                uint32_t und = 0;
#pragma unroll
                for (int r = 0; r < kFiltItems; ++r) {
                    const int f = fan_signs_f32(sv, c.x, c.y, p[r].x, p[r].y);
                    in |= (f == 1 ? 1u : 0u) << r;
                    und |= (f == 2 ? 1u : 0u) << r;
                }
                in &= kb;
                und &= kb;
                while (und) {
                    const int r = __ffs(und) - 1;
                    und &= und - 1u;
                    const float2 q = p2[lo + r * kFiltThreads + t];
                    if (fan_inside_exact(sv, c.x, c.y, q.x, q.y)) in |= 1u << r;
                }
                if (in) bits[(size_t)tile * kFiltThreads + t] = (uint16_t)(kb & ~in);
            }
            uint32_t removed = __popc(in);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) removed += __shfl_xor_sync(0xffffffffu, removed, o);
            if (lane == 0 && removed) atomicAdd(&status[tile], 0ull - (unsigned long long)removed);
        }
    }
}

}  // namespace

cudaError_t launch_bx_fan(const float *pts, void *ws, const Layout &L, const BatchLayout &BL, cudaStream_t st)
{
    const int sms = sm_count();
    static const bool attrs = [] {
        cudaFuncSetAttribute(bx_fan_refine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFanSmem);
        return true;
    }();
    (void)attrs;
    const uint32_t chunk = tune_value(CH_TUNE_BX_FAN_CHUNK) ? (uint32_t)tune_value(CH_TUNE_BX_FAN_CHUNK) : kBxFanChunk;
    const uint32_t stride = tune_value(CH_TUNE_BX_FAN_STRIDE) ? (uint32_t)tune_value(CH_TUNE_BX_FAN_STRIDE)
                                                              : kBxBinStride;
    probe_before(CH_K_KGON, st);
    launch_next(bx_fan_select_kernel, 1, 1024, 0, st, ws, L, BL, chunk);
    launch_next(bx_fan_bins_kernel, (unsigned)(sms * 4), FT, 0, st, pts, ws, L, BL, chunk, stride);
    launch_next(bx_fan_build_kernel, (unsigned)(sms * 2), BT, 0, st, pts, ws, L, BL);
    launch_next(bx_fan_refine_kernel, (unsigned)sms, CT, kFanSmem, st, pts, ws, L, BL, chunk);
    note_kernels(CH_K_KGON, 4);
    probe_after(CH_K_KGON, st);
    return cudaGetLastError();
}

}  // namespace ch
