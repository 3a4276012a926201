// Boxes of the BVH's nodes: how the scene upload codes them and how a ray meets them.
//
// A box is a centre and a half extent along each axis, on the scene's grid: 65536 positions an axis, the
// centre a 16-bit position, the half extent a binary16 number of steps; or, in a wide scene, whose
// geometry the grid is too coarse for, two floats.  The code compiles with the host compiler too (see
// hpt_pair.cuh).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "hpt_pair.cuh"

namespace hpt {

struct Box {
    float lo[3], hi[3];
    void reset()
    {
        for (int k = 0; k < 3; ++k) { lo[k] = INFINITY; hi[k] = -INFINITY; }
    }
    void grow(const Box &b)
    {
        for (int k = 0; k < 3; ++k) { lo[k] = std::min(lo[k], b.lo[k]); hi[k] = std::max(hi[k], b.hi[k]); }
    }
    void grow(const float *p)
    {
        for (int k = 0; k < 3; ++k) { lo[k] = std::min(lo[k], p[k]); hi[k] = std::max(hi[k], p[k]); }
    }
};

struct BoxGrid {
    float lo[3], step[3];
};

// ---- the scene's side -----------------------------------------------------------------------
// what every box is padded by, a few float ulps of the scene's largest coordinate
inline float box_pad(float max_abs) { return 2e-6f * max_abs + 1e-12f; }

// The grid of the node boxes: 65536 positions along each axis across the scene's padded bounds, or,
// where a few triangles stretch those bounds beyond 16 times what holds the others (a far ground
// under millimetre objects), across the bounds of the others: the box of a node with such a
// triangle then reaches to infinity along that axis instead of every box being coarse (spheres of
// 1 mm over a 4 m ground, 960 x 540 frame: 23.9 ms with float boxes, 28.9 on a grid of all, 22.7 so).
inline BoxGrid box_grid(const std::vector<Box> &pb, const std::vector<int> &prims, float pad)
{
    Box all, core;
    all.reset();
    core.reset();
    for (int t : prims) all.grow(pb[t]);
    for (int t : prims)
        for (int k = 0; k < 3; ++k)
            if (pb[t].hi[k] - pb[t].lo[k] <= 0.25f * (all.hi[k] - all.lo[k])) {
                core.lo[k] = std::min(core.lo[k], pb[t].lo[k]);
                core.hi[k] = std::max(core.hi[k], pb[t].hi[k]);
            }
    BoxGrid g;
    for (int k = 0; k < 3; ++k) {
        const bool use_core = core.hi[k] >= core.lo[k] && 16.0f * (core.hi[k] - core.lo[k] + 2.0f * pad) < all.hi[k] - all.lo[k];
        const Box &b = use_core ? core : all;
        g.lo[k] = b.lo[k] - pad;
        g.step[k] = (float)(((double)b.hi[k] + pad - g.lo[k]) / 65534.0);
    }
    return g;
}

// The interval lo .. hi of axis k on the grid: the centre's nearest position, and the half extent in
// steps, rounded up, that reaches one step past both padded planes.
inline void box_code(const BoxGrid &g, float pad, float lo, float hi, int k, unsigned &c, unsigned &h)
{
    const double s = g.step[k], l = ((double)lo - pad - g.lo[k]) / s - 1.0, u = ((double)hi + pad - g.lo[k]) / s + 1.0;
    c = (unsigned)std::min(65535.0, std::max(0.0, std::floor(0.5 * (l + u) + 0.5)));
    const double e = std::max(u - (double)c, (double)c - l);
    __half v = __float2half_ru((float)e);
    if ((double)__half2float(v) < e) v = __ushort_as_half((unsigned short)(__half_as_ushort(v) + 1));
    h = __half_as_ushort(v);
}
constexpr unsigned NO_BOX = 0xFC00u;   // half extent -inf: a child that is never entered

// The same interval as two floats: its middle, and the half extent, rounded up, that reaches both padded planes.
// Wide scenes have the grid { 0, 0, 0 }, { 1, 1, 1 }.
inline void box_code_wide(float pad, float lo, float hi, float &c, float &h)
{
    const double l = (double)lo - pad, u = (double)hi + pad;
    c = (float)(0.5 * (l + u));
    const double e = std::max(u - (double)c, (double)c - l);
    h = (float)e;
    if ((double)h < e) h = std::nextafter(h, INFINITY);
}
constexpr BoxGrid WIDE_GRID = {{0.0f, 0.0f, 0.0f}, {1.0f, 1.0f, 1.0f}};

// The surface of a box coded on the grid with half extents h over its surface as padded floats; 0 if it reaches to
// infinity.
inline double box_growth(const BoxGrid &g, float pad, const Box &b, const unsigned h[3])
{
    double f[3], q[3];
    for (int k = 0; k < 3; ++k) {
        f[k] = (double)b.hi[k] - b.lo[k] + 2.0 * pad;
        q[k] = 2.0 * (double)__half2float(__ushort_as_half((unsigned short)h[k])) * g.step[k];
        if (!std::isfinite(q[k])) return 0.0;
    }
    return (q[0] * q[1] + q[1] * q[2] + q[2] * q[0]) / (f[0] * f[1] + f[1] * f[2] + f[2] * f[0]);
}

// Whether a scene is wide: the grid makes its boxes more than WIDE_GROWTH times as large, in the geometric mean
// over the tree's nodes.  Two groups of finely tessellated spheres (edges of 13 um) apart, 960 x 540 x 16 frame on
// the grid / with float boxes / with the two-plane float boxes of before, in ms, and the growth:
//   0.1 m 6.4 / 6.6 / 7.9 (1.50)   0.2 m 7.3 / 6.7 / 8.1 (2.01)   0.5 m 10.6 / 7.0 / 8.7 (3.7)   3 m 71.9 / 10.6 / 14.0 (19)
// and 5.9 / 5.9 / 6.9 (1.49) with edges of 26 um 0.2 m apart.  Ordinary scenes are at 1.00 to 1.03, where the
// grid wins by 13 to 21 %.
constexpr double WIDE_GROWTH = 1.5;
class BoxGrowth {
    double log_sum = 0.0, product = 1.0;
    long long n = 0;

  public:
    void add(double f)
    {
        if (!(f > 0.0)) return;
        product *= f;
        ++n;
        if (product > 1e100) {
            log_sum += std::log(product);
            product = 1.0;
        }
    }
    bool wide() const { return log_sum + std::log(product) > n * std::log(WIDE_GROWTH); }
};

// Whether rays from anywhere in 'o' reach the node boxes (see grid_ray), 'bound' being the largest coordinate of
// the padded geometry: pad is 2e-6 of it.
constexpr float BOX_ULPS = 9.0f, BOX_NEAR = 0.55f;
inline bool origins_near(const BoxGrid &g, bool wide, float bound, const Box &o)
{
    for (int k = 0; k < 3; ++k) {
        const float dist = std::max(std::fabs(o.lo[k] - g.lo[k]), std::fabs(o.hi[k] - g.lo[k]));
        const float past = 1.99e-6f * bound + (wide ? 0.0f : g.step[k]);
        if (!(BOX_ULPS * 0x1p-24f / past * dist + BOX_NEAR <= 1.0f)) return false;
    }
    return true;
}

// ---- the ray's side -------------------------------------------------------------------------
// A ray prepared for the boxes of a scene's grid: with q a box centre in grid steps and
// c' = 2^23 + q its float (the bits 0x4B000000 | q), the distance to the centre's plane is
// c' * st + k, st = step / d and k = (grid origin - o) / d - 2^23 st.
struct GridRay {
    float3 st, sa, k;   // sa = |st|
};

// With u = 2^-24 and X the point of a box that the ray meets, the slab of an axis is off by no more than
// 4u |X - o| (the reciprocal, within 2 ulp of itself), u |X - lo| (rounding st), 3u |lo - o| (the difference,
// its product and k), half a step (rounding k, which 2^23 st dominates) and 2u |X - o| (the two FMAs):
// together at most BOX_ULPS u (|lo - o| + |X - lo|) + step / 2.  A half extent reaches past the geometry by
// pad + step, pad being 33u max_abs.  Of that step / 2 and the part with |X - lo| take at most BOX_NEAR wherever the
// geometry lies (|X - lo| is at most 65536 steps on a grid of all triangles, and 2 max_abs beyond a core grid), so
// a box is not missed from an origin up to some two sizes of the scene away, nor from one on the
// geometry.  First rays that would start farther away (origins_near) start where far_start says.
// WIDE: the scene may be a wide one, of no 2^23 and no steps (half a step less is off, and the half extents reach
// past the geometry by pad alone, which is enough as well).
template <bool WIDE, class SCENE>
__device__ __forceinline__ GridRay grid_ray(const SCENE &sc, float3 o, float3 inv)
{
    GridRay r;
    r.st = make_float3(sc.grid.step[0] * inv.x, sc.grid.step[1] * inv.y, sc.grid.step[2] * inv.z);
    r.sa = make_float3(fabsf(r.st.x), fabsf(r.st.y), fabsf(r.st.z));
    const float off = WIDE && sc.wide ? 0.0f : -8388608.0f;
    r.k = make_float3(fmaf(off, r.st.x, (sc.grid.lo[0] - o.x) * inv.x), fmaf(off, r.st.y, (sc.grid.lo[1] - o.y) * inv.y),
                      fmaf(off, r.st.z, (sc.grid.lo[2] - o.z) * inv.z));
    return r;
}

// How far along it a ray from far away may start without passing by any of the geometry in 'b' (0 for one
// that does not meet b): where it enters b widened by a 32nd of its size and by what the float arithmetic here can
// be off, 2^-18 of the distance.  Started there, after the advance in the coherent arithmetic, the float ray is
// within the reach of the boxes, and its tests lose nothing to the distance.
__device__ __forceinline__ float far_start(const Box &b, float3 o, float3 d)
{
    const float oo[3] = {o.x, o.y, o.z}, dd[3] = {d.x, d.y, d.z};
    const float m = 0.03125f * fmaxf(fmaxf(b.hi[0] - b.lo[0], b.hi[1] - b.lo[1]), b.hi[2] - b.lo[2]) +
                    0x1p-18f * fmaxf(fmaxf(fabsf(o.x), fabsf(o.y)), fabsf(o.z));
    float in = 0.0f, out = 1e30f;
    for (int k = 0; k < 3; ++k) {
        const float inv = fabsf(dd[k]) > 1e-20f ? 1.0f / dd[k] : copysignf(1e20f, dd[k]);
        const float t0 = (b.lo[k] - m - oo[k]) * inv, t1 = (b.hi[k] + m - oo[k]) * inv;
        in = fmaxf(in, fminf(t0, t1));
        out = fminf(out, fmaxf(t0, t1));
    }
    return in <= out ? in : 0.0f;
}

// Entry and exit distances (clipped to [0, tl]) of a ray in the two child boxes of a node: q = the
// centres (on a grid 2^23 + the position), h = the half extents, of child 0 and child 1 on each axis.  With tc the
// distance to the centre an axis's slab is [tc - h sa, tc + h sa], which takes no minimum and maximum of its two
// planes, and the children go through as one packed pair.
__device__ __forceinline__ void box_pair(const float2 q[3], const float2 h[3], const GridRay &r, float tl, float &c0min,
                                         float &c0max, float &c1min, float &c1max)
{
    f2 t[3];
    const float st[3] = {r.st.x, r.st.y, r.st.z}, kk[3] = {r.k.x, r.k.y, r.k.z}, sa[3] = {r.sa.x, r.sa.y, r.sa.z};
    float n0[3], n1[3], x0[3], x1[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        t[a] = fma2(pk(q[a].x, q[a].y), pk(st[a], st[a]), pk(kk[a], kk[a]));
        upk(fma2(pk(h[a].x, h[a].y), pk(-sa[a], -sa[a]), t[a]), n0[a], n1[a]);
        upk(fma2(pk(h[a].x, h[a].y), pk(sa[a], sa[a]), t[a]), x0[a], x1[a]);
    }
    c0min = fmaxf(fmaxf(n0[0], n0[1]), fmaxf(n0[2], 0.0f));
    c0max = fminf(fminf(x0[0], x0[1]), fminf(x0[2], tl));
    c1min = fmaxf(fmaxf(n1[0], n1[1]), fmaxf(n1[2], 0.0f));
    c1max = fminf(fminf(x1[0], x1[1]), fminf(x1[2], tl));
}
// a word of a node: the 16-bit centres of both children on an axis (child 0 in the low half), or their binary16 half
// extents
__device__ __forceinline__ float2 centres(unsigned w)
{
    return make_float2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7410)), __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7432)));
}
__device__ __forceinline__ float2 extents(unsigned w) { return __half22float2(*reinterpret_cast<const __half2 *>(&w)); }

}  // namespace hpt
