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
// is decided exactly by keep_point.  Two differences, 16 FMAs and 7 minima
// decide nearly every point, whatever the polygon's shape.  Testing the edge
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

// keep(p) <=> NOT (p strictly left of every valid edge); see
// build_octagon_warp for the error bound of the binary32 test, which holds
// for points inside the vertices' bounding box.
template <bool BOX>
__device__ __noinline__ bool keep_point(const Octagon &o, float x, float y)
{
    if (x >= o.xl && x <= o.xh && y >= o.yl && y <= o.yh) return false;
    if (!o.has_edges || outside_box<BOX>(o, x, y)) return true;
#pragma unroll 1
    for (int e = 0; e < 8; ++e) {
        if (!((o.valid >> e) & 1u)) continue;
        const float u = __fsub_rn(x, o.ax[e]);
        const float v = __fsub_rn(y, o.ay[e]);
        const float t = __fsub_rn(__fmul_rn(o.dx[e], v), __fmul_rn(o.dy[e], u));
        const float bnd = o.bound[e];
        if (t > bnd) continue;
        if (t < -bnd) return true;
        if (orient_d(o.ax[e], o.ay[e], o.bx[e], o.by[e], x, y) <= 0) return true;
    }
    return false;
}

// The polygon in shared memory, the edges' affine forms packed.
struct OctSmem : Octagon {
    float4 t4[8];   // (tx, ty, tz, -)
};

// Copies the polygon `g` to shared memory; the caller synchronises before
// `so` is read.
__device__ __forceinline__ void fill_octagon(OctSmem &so, const Octagon *g)
{
    const uint32_t *src = reinterpret_cast<const uint32_t *>(g);
    uint32_t *dst = reinterpret_cast<uint32_t *>(static_cast<Octagon *>(&so));
    for (uint32_t w = threadIdx.x; w < sizeof(Octagon) / 4; w += blockDim.x) dst[w] = src[w];
    if (threadIdx.x < 8)
        so.t4[threadIdx.x] = make_float4(g->tx[threadIdx.x], g->ty[threadIdx.x], g->tz[threadIdx.x], 0.0f);
}

// NaN-propagating minimum: an overflowed difference (or edge forms that are
// switched off) must leave a point undecided, not inside.
__device__ __forceinline__ float min_nan(float a, float b)
{
    float d;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
    return d;
}

// N points at once: bit q of `in` when point q is proven strictly inside,
// of `und` when it is undecided.  The edges are the outer loop, so their
// forms are read once for the N points.
template <int N>
__device__ __forceinline__ void oct_decide(const OctSmem &o, const float (&px)[N], const float (&py)[N], uint32_t &in,
                                           uint32_t &und)
{
    float u[N], v[N], m[N];
    const float cx = o.cx, cy = o.cy;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        u[q] = __fsub_rn(px[q], cx);
        v[q] = __fsub_rn(py[q], cy);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        const float4 t = o.t4[k];
#pragma unroll
        for (int q = 0; q < N; ++q) {
            const float T = __fmaf_rn(t.x, u[q], __fmaf_rn(t.y, v[q], t.z));
            m[q] = k == 0 ? T : min_nan(m[q], T);
        }
    }
    in = und = 0u;
#pragma unroll
    for (int q = 0; q < N; ++q) {
        const bool i = m[q] > 1.0f;
        in |= (i ? 1u : 0u) << q;
        und |= (!i && !(m[q] < -1.0f) ? 1u : 0u) << q;
    }
}

}  // namespace ch
