// fan.cuh -- the hull step's fan: angular bins around the centre and the
// order key of the farthest-point choice (kgon.cu).
#pragma once

#include "common.cuh"

namespace ch {

// The first level's sample: every fan_sample_stride(tiles)-th 4096-point
// tile (at least every tile; about kFanBinTiles tiles, at most every 16th).
// Of 10^8 circle points 7.5 M reach the second level with every 16th tile and
// 7.0 M with every 8th, whose bins take 40 us more.
constexpr int64_t kFanBinTiles = 1536;
__host__ __device__ inline int64_t fan_sample_stride(int64_t tiles)
{
    const int64_t s = tiles / kFanBinTiles;
    return s < 1 ? 1 : (s > 16 ? 16 : s);
}

// A fan's number of bins NB (a multiple of 4, below 2^22): known at compile
// time, or a set's own.
template <int NB>
struct FixedBins {
    static_assert(NB % 4 == 0 && NB < (1 << 22), "the shifted offsets are exact");
    __device__ static constexpr float quarter() { return NB / 4.0f; }
    __device__ static constexpr uint32_t count() { return NB; }
};
struct SetBins {
    uint32_t n;
    __device__ float quarter() const { return (float)(n / 4u); }
    __device__ uint32_t count() const { return n; }
};

// Scaled pseudo-angle of the direction (dx, dy): in [0, NB], growing with
// the angle counter-clockwise from -y; bin b holds [b, b + 1).  With t = dy /
// (|dx| + |dy|) it is (1 + t) NB / 4 on the right and (3 - t) NB / 4 on the
// left: one test and one FMA.  (dx = dy = 0 gives a NaN.)
__device__ __forceinline__ float fan_turn(float dx, float dy)   // t on the right, -t on the left
{
    float r;   // (at most 1 ulp off; a subnormal sum counts as zero)
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__fadd_rn(fabsf(dx), fabsf(dy))));
    return __uint_as_float(__float_as_uint(__fmul_rn(dy, r)) ^ (__float_as_uint(dx) & 0x80000000u));
}

template <class Bins>
__device__ __forceinline__ float fan_phi(Bins nb, float dx, float dy)
{
    const bool left = (int)__float_as_uint(dx) < 0;
    return __fmaf_rn(fan_turn(dx, dy), nb.quarter(), left ? 3.0f * nb.quarter() : nb.quarter());
}

// kBinBias + its bin, the bin in [-1, NB] (a NaN: kBinBias + NB): the same FMA
// shifted by 2^23 and rounded down leaves the bin in the low mantissa bits.
// (-1: straight below, a reciprocal one ulp too large makes t less than -1.  A
// table that is read at such an index has an entry, and one beside it, on
// either side; inner_bin tells where one is not wanted.)
constexpr uint32_t kBinBias = 0x4b000000u;
template <class Bins>
__device__ __forceinline__ uint32_t fan_bin_biased(Bins nb, float dx, float dy)
{
    const bool left = (int)__float_as_uint(dx) < 0;
    const float f = __fmaf_rd(fan_turn(dx, dy), nb.quarter(),
                              left ? 0x1p23f + 3.0f * nb.quarter() : 0x1p23f + nb.quarter());
    return min(__float_as_uint(f), kBinBias + nb.count());
}

// Whether bin b (less kBinBias, modulo 2^32) has neighbours on both sides: in
// [1, nb - 2].
__host__ __device__ inline bool inner_bin(uint32_t b, uint32_t nb) { return b - 1u < nb - 2u; }

// The direction of pseudo-angle a (|x| + |y| = 1).
template <class Bins>
__device__ __forceinline__ float2 fan_direction(Bins nb, float a)
{
    const float q = a / nb.quarter();
    const float t = q < 2.0f ? q - 1.0f : 3.0f - q;
    return make_float2(q < 2.0f ? 1.0f - fabsf(t) : fabsf(t) - 1.0f, t);
}

// Order key for the farthest-point choice of a bin: |p - c|^2 - r2ref,
// from the differences p - c and their squares as exact pairs (two-sum,
// two-product by FMA), rounded once at the end.  The binary32 square
// |p - c|^2 itself resolves only 2^-23 of its value, while on the unit
// circle the radii of binary32 points differ by about 10^-7 and the top
// points of a bin by far less: the vertex would be any of its top points
// and the chords sag below the others.  Any key would keep the test exact
// (a vertex only has to be an input point); this one finds the farthest.
// r2ref: a squared distance of the set's scale (Sterbenz: the last
// difference is exact when the sum is within a factor 2 of it).
__device__ __forceinline__ uint32_t far_key(float px, float py, float cx, float cy, float r2ref)
{
    float dxh, dxl, dyh, dyl;
    two_diff(px, cx, dxh, dxl);
    two_diff(py, cy, dyh, dyl);
    const float sxh = __fmul_rn(dxh, dxh), sxl = __fmaf_rn(dxh, dxh, -sxh);
    const float syh = __fmul_rn(dyh, dyh), syl = __fmaf_rn(dyh, dyh, -syh);
    float sh, sl;
    two_sum(sxh, syh, sh, sl);
    const float cross = __fmul_rn(2.0f, __fmaf_rn(dxh, dxl, __fmul_rn(dyh, dyl)));
    const float lo = __fadd_rn(__fadd_rn(sl, __fadd_rn(sxl, syl)), cross);
    return ord_key(__fadd_rn(__fsub_rn(sh, r2ref), lo));
}

// A point (the centre) as the fan's arithmetic sees it: times the set's power
// of two.  Squares and products of differences neither overflow nor vanish
// then, whatever the set's size; a coordinate that becomes subnormal moves by
// 2^-150 at most, of a box of size 1 to 4.
__device__ __forceinline__ float2 fan_space(float2 p, float scale)
{
    return make_float2(__fmul_rn(p.x, scale), __fmul_rn(p.y, scale));
}
__device__ __forceinline__ float2 fan_centre(const Octagon &o) { return fan_space(make_float2(o.cx, o.cy), o.scale); }

// r2ref of far_key for a polygon's set: the squared distance from its
// centre to its first vertex (binary32).
__device__ __forceinline__ float far_ref(const Octagon &o)
{
    const float ux = __fmul_rn(__fsub_rn(o.ax[0], o.cx), o.scale), uy = __fmul_rn(__fsub_rn(o.ay[0], o.cy), o.scale);
    return __fmaf_rn(ux, ux, __fmul_rn(uy, uy));
}

}  // namespace ch
