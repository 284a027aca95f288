// octtest.cuh -- the point test of Sec. 3.2 (is a point strictly inside the
// eight-vertex polygon?), shared by the filter's passes (filter.cu) and the
// hull step's filter (kgon.cu).
//
// A point is discarded when it is strictly left of every valid edge.  With
// c the polygon's box centre, (u, v) = fl(p - c), edge k's value is
//   T_k = fma(tx_k, u, fma(ty_k, v, tz_k)),
// an affine form scaled so that its rounding error is below 1 for every
// point of the polygon's box (build_octagon_warp, which has the proof):
// min_k T_k > 1 proves the point strictly inside, min_k T_k < -1 proves it
// kept, anything else (a band of relative width 2^-20 around the boundary)
// is decided exactly by keep_point.  Two differences, 16 FMAs (8
// instructions: two points at once) and 4 three-operand minima decide nearly
// every point, whatever the polygon's shape.  Testing the edge
// of the point's octant first and the other seven in a second, queued step
// took 46 instructions for a circle's points and sent most points of a thin
// rotated ellipse to the second step: the hull of 10^8 such points took 2167
// us, 1387 with these forms; 4096 sets in a batch 13.6 ms, 12.7 with them.
#pragma once

#include "common.cuh"

namespace ch {

// Outside the closed bounding box of the polygon's vertices: never strictly
// inside the polygon.  Only tested when the vertices were supplied by the
// caller (BOX); the data's own extremes span a box holding every point.
template <bool BOX>
__device__ __forceinline__ bool outside_box(const Octagon &o, float x, float y)
{
    if constexpr (BOX) return x < o.bxl || x > o.bxh || y < o.byl || y > o.byh;
    return false;
}

// keep(p) <=> NOT (p strictly left of every valid edge): the forms first,
// all at once, then exact signs at the edges they leave undecided (the forms
// hold for points inside the vertices' bounding box; when they are off, all
// edges are undecided).
// Bound by latency: few points come here, unless the input lies on the
// polygon's edges (a rectangle's sides, a coarse grid), and then all.  One edge
// after the other, each by a static bound first, 300007 points on a square's
// sides took the filter 74 us and on a 16 x 16 grid 56; so 25 and 20.
template <bool BOX>
__device__ __noinline__ bool keep_point(const Octagon &o, float x, float y)
{
    if (!o.has_edges || outside_box<BOX>(o, x, y)) return true;
    const float u = __fsub_rn(x, o.cx), v = __fsub_rn(y, o.cy);
    uint32_t open = 0;
    bool out = false;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float t = __fmaf_rn(o.tx[k], u, __fmaf_rn(o.ty[k], v, o.tz[k]));
        out |= t < -1.0f;
        open |= t > 1.0f ? 0u : 1u << k;
    }
    if (out) return true;
#pragma unroll 1
    for (open &= o.valid; open; open &= open - 1u) {
        const int e = __ffs(open) - 1;
        if (orient_rest(o.ax[e], o.ay[e], o.bx[e], o.by[e], x, y) <= 0) return true;
    }
    return false;
}

// The polygon in shared memory, the edges' affine forms twice over for the
// packed arithmetic.
struct OctSmem : Octagon {
    float4 txy[8];   // tx, tx, ty, ty
    float2 tzz[8];   // tz, tz
};

// Copies the polygon `g` to shared memory; the caller synchronises before
// `so` is read.
__device__ __forceinline__ void fill_octagon(OctSmem &so, const Octagon *g)
{
    const uint32_t *src = reinterpret_cast<const uint32_t *>(g);
    uint32_t *dst = reinterpret_cast<uint32_t *>(static_cast<Octagon *>(&so));
    for (uint32_t w = threadIdx.x; w < sizeof(Octagon) / 4; w += blockDim.x) dst[w] = src[w];
    if (threadIdx.x < 8) {
        const float tx = g->tx[threadIdx.x], ty = g->ty[threadIdx.x], tz = g->tz[threadIdx.x];
        so.txy[threadIdx.x] = make_float4(tx, tx, ty, ty);
        so.tzz[threadIdx.x] = make_float2(tz, tz);
    }
}

// N points at once: bit q of `keep` unless point q is proven strictly inside
// the polygon; the result says whether any of them is undecided
// (keep_point settles it; the NaN-propagating minima leave a point undecided
// whose difference overflowed).  The edges are the outer loop, so
// their forms are read once for the N points, and two points share an FMA
// instruction.
template <int N>
__device__ __forceinline__ bool oct_decide(const OctSmem &o, const float (&px)[N], const float (&py)[N], uint32_t &keep)
{
    f32x2 u[N / 2], v[N / 2];
    float m[N];
    const float cx = o.cx, cy = o.cy;
#pragma unroll
    for (int q = 0; q < N / 2; ++q) {
        u[q] = pack2(__fsub_rn(px[2 * q], cx), __fsub_rn(px[2 * q + 1], cx));
        v[q] = pack2(__fsub_rn(py[2 * q], cy), __fsub_rn(py[2 * q + 1], cy));
    }
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
        asm volatile("" ::: "memory");   // (two edges' forms in registers at a time)
        const float4 ta = o.txy[k], tb = o.txy[k + 1];
        const float2 za = o.tzz[k], zb = o.tzz[k + 1];
        const f32x2 xa = pack2(ta.x, ta.y), ya = pack2(ta.z, ta.w), xb = pack2(tb.x, tb.y), yb = pack2(tb.z, tb.w);
        const f32x2 z0 = pack2(za.x, za.y), z1 = pack2(zb.x, zb.y);
#pragma unroll
        for (int q = 0; q < N / 2; ++q) {
            const float2 a = unpack2(fma2(xa, u[q], fma2(ya, v[q], z0)));
            const float2 b = unpack2(fma2(xb, u[q], fma2(yb, v[q], z1)));
            m[2 * q] = k == 0 ? min_nan(a.x, b.x) : min_nan(m[2 * q], a.x, b.x);
            m[2 * q + 1] = k == 0 ? min_nan(a.y, b.y) : min_nan(m[2 * q + 1], a.y, b.y);
        }
    }
    keep = 0u;
    float near = 2.0f;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        if (!(m[q] > 1.0f)) keep |= 1u << q;
        near = min_nan(near, fabsf(m[q]));
    }
    return !(near > 1.0f);
}

// Point of item q of the 16 that thread t (of kFiltThreads) has in the
// 4096-point tile at `base`: item q = r * G + h is point base + (r *
// kFiltThreads + t) * G + h (G = 2: pairs of points, read 16 bytes at once).
template <int G>
__device__ __forceinline__ int64_t item_point(int64_t base, uint32_t t, int q)
{
    return base + (int64_t)((q / G) * kFiltThreads + t) * G + q % G;
}

__device__ __forceinline__ float2 input_point(const float *pts, int64_t i)
{
    return __ldg(reinterpret_cast<const float2 *>(pts) + i);
}

// Items N part .. N part + N - 1 of a thread's 16 in the tile at `base`, all of
// them below n (G = 2: 16-byte loads).
template <int G, int N>
__device__ __forceinline__ void load_part(const float *__restrict__ pts, int64_t base, uint32_t t, int part,
                                          float (&px)[N], float (&py)[N])
{
    if constexpr (G == 2) {
        const float4 *p4 = reinterpret_cast<const float4 *>(pts) + base / 2 + part * (N / 2) * kFiltThreads + t;
        float4 v[N / 2];
#pragma unroll
        for (int r = 0; r < N / 2; ++r) v[r] = __ldg(p4 + r * kFiltThreads);
#pragma unroll
        for (int r = 0; r < N / 2; ++r) {
            px[2 * r] = v[r].x;
            py[2 * r] = v[r].y;
            px[2 * r + 1] = v[r].z;
            py[2 * r + 1] = v[r].w;
        }
    } else {
        const float2 *p2 = reinterpret_cast<const float2 *>(pts) + base + part * N * kFiltThreads + t;
#pragma unroll
        for (int r = 0; r < N; ++r) {
            const float2 v = __ldg(p2 + r * kFiltThreads);
            px[r] = v.x;
            py[r] = v.y;
        }
    }
}

// The same where the tile ends before them: the centre stands in for the
// missing points; returns the bits of those that exist.
template <int G, int N>
__device__ __forceinline__ uint32_t load_part_ragged(const float *__restrict__ pts, int64_t n, int64_t base, uint32_t t,
                                                     int part, float cx, float cy, float (&px)[N], float (&py)[N])
{
    uint32_t live = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
        const int64_t i = item_point<G>(base, t, N * part + k);
        const float2 v = i < n ? input_point(pts, i) : make_float2(cx, cy);
        px[k] = v.x;
        py[k] = v.y;
        live |= (i < n ? 1u : 0u) << k;
    }
    return live;
}

}  // namespace ch
