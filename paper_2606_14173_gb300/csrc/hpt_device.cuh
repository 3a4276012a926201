#pragma once
// Device building blocks of the wave path tracer: small vector math, the Philox4x32-10
// counter-based generator, float BVH traversal with near-edge tracking, the double-precision
// re-decision of a coherent hit, surface attributes, textures, the ambient cache and BSDFs.
#include <cstdint>
#include <cfloat>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "hpt_internal.h"
#include "hpt_real.cuh"

namespace hpt {

#define INC_OFFSET 1e-7f        // incoherent origin offset along the geometric normal (m)
#define COH_TMIN 1e-9           // coherent continuation minimum distance (m)
#define SHADOW_SHRINK 1e-5f
#define NEAR_MARGIN 1e-4f       // barycentric band treated as "near an edge" on coherent rays
#define TIE_REL 2e-6f           // relative distance band treated as a tie on coherent rays
#define WATERTIGHT_EPS 2e-5f    // most barycentric slack of float tests on incoherent rays (per
                                // triangle: a band of 1e-6 x the scene's largest coordinate)
#define PI_F 3.14159265358979f
#define INV_PI_F 0.318309886183791f

// ------------------------------------------------------------------------------ small math
__device__ __forceinline__ float3 f3(float x, float y, float z) { return make_float3(x, y, z); }
__device__ __forceinline__ float3 operator+(float3 a, float3 b) { return f3(a.x + b.x, a.y + b.y, a.z + b.z); }
__device__ __forceinline__ float3 operator-(float3 a, float3 b) { return f3(a.x - b.x, a.y - b.y, a.z - b.z); }
__device__ __forceinline__ float3 operator*(float3 a, float s) { return f3(a.x * s, a.y * s, a.z * s); }
__device__ __forceinline__ float3 operator-(float3 a) { return f3(-a.x, -a.y, -a.z); }
__device__ __forceinline__ float dot3(float3 a, float3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ float3 cross3(float3 a, float3 b)
{
    return f3(a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x);
}
__device__ __forceinline__ float3 normalize3(float3 a) { return a * rsqrtf(dot3(a, a)); }
// the same products with every rounding spelled out (fixed FMA contraction), so that a result does
// not depend on how the compiler contracts the surrounding code of a given build
__device__ __forceinline__ float dot3_rn(float3 a, float3 b) { return fmaf(a.x, b.x, fmaf(a.y, b.y, __fmul_rn(a.z, b.z))); }
__device__ __forceinline__ float3 cross3_rn(float3 a, float3 b)
{
    return f3(fmaf(a.y, b.z, -__fmul_rn(a.z, b.y)), fmaf(a.z, b.x, -__fmul_rn(a.x, b.z)), fmaf(a.x, b.y, -__fmul_rn(a.y, b.x)));
}
// the same for the microfacet code: a b + c d and a b - c d with the first product inside the FMA, and
// the two orders of a dot product that it uses
__device__ __forceinline__ float sum2_rn(float a, float b, float c, float d) { return fmaf(a, b, __fmul_rn(c, d)); }
__device__ __forceinline__ float diff2_rn(float a, float b, float c, float d) { return fmaf(a, b, -__fmul_rn(c, d)); }
__device__ __forceinline__ float dot3_zxy(float3 a, float3 b) { return fmaf(a.z, b.z, fmaf(a.x, b.x, __fmul_rn(a.y, b.y))); }
__device__ __forceinline__ float dot3_zyx(float3 a, float3 b) { return fmaf(a.z, b.z, fmaf(a.y, b.y, __fmul_rn(a.x, b.x))); }
__device__ __forceinline__ float3 xyz(float4 a) { return f3(a.x, a.y, a.z); }

template <class R> struct R3 {
    R x, y, z;
};
template <class R> __device__ __forceinline__ R3<R> neg(R3<R> a) { R3<R> v; v.x = -a.x; v.y = -a.y; v.z = -a.z; return v; }
template <class R> __device__ __forceinline__ R3<R> r3(R x, R y, R z) { R3<R> v; v.x = x; v.y = y; v.z = z; return v; }
template <class R> __device__ __forceinline__ R3<R> operator+(R3<R> a, R3<R> b) { return r3<R>(a.x + b.x, a.y + b.y, a.z + b.z); }
template <class R> __device__ __forceinline__ R3<R> operator-(R3<R> a, R3<R> b) { return r3<R>(a.x - b.x, a.y - b.y, a.z - b.z); }
template <class R> __device__ __forceinline__ R3<R> scale(R3<R> a, R s) { return r3<R>(a.x * s, a.y * s, a.z * s); }
template <class R> __device__ __forceinline__ R rdot(R3<R> a, R3<R> b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
// In double, the products of the delta vertices with every rounding spelled out (the same reason as
// below: a result must not depend on how the compiler contracts the code around it); double-float
// operations fix their roundings themselves.
__device__ __forceinline__ double sum2_rn(double a, double b, double c, double d) { return __fma_rn(a, b, __dmul_rn(c, d)); }
__device__ __forceinline__ double rdot_zxy(R3<double> a, R3<double> b) { return __fma_rn(a.z, b.z, sum2_rn(a.x, b.x, a.y, b.y)); }
__device__ __forceinline__ double rdot_zyx(R3<double> a, R3<double> b) { return __fma_rn(a.z, b.z, sum2_rn(a.y, b.y, a.x, b.x)); }
__device__ __forceinline__ double mix3(double a, float x, double b, float y, double c, float z)
{
    return __fma_rn(c, (double)z, sum2_rn(a, (double)x, b, (double)y));
}
__device__ __forceinline__ double diff2(double a, double b, double c, double d) { return __fma_rn(-c, d, __dmul_rn(a, b)); }
__device__ __forceinline__ df rdot_zxy(R3<df> a, R3<df> b) { return rdot(a, b); }
__device__ __forceinline__ df rdot_zyx(R3<df> a, R3<df> b) { return rdot(a, b); }
__device__ __forceinline__ df mix3(df a, float x, df b, float y, df c, float z) { return mul_f(a, x) + mul_f(b, y) + mul_f(c, z); }
__device__ __forceinline__ df diff2(df a, df b, df c, df d) { return a * b - c * d; }
template <class R> __device__ __forceinline__ float3 tof3(R3<R> a)
{
    return f3(RealOps<R>::to_f(a.x), RealOps<R>::to_f(a.y), RealOps<R>::to_f(a.z));
}
template <class R> __device__ __forceinline__ R3<R> fromf3(float3 a)
{
    return r3<R>(RealOps<R>::f(a.x), RealOps<R>::f(a.y), RealOps<R>::f(a.z));
}

// ------------------------------------------------------------------- Philox4x32-10 (SC'11)
__device__ __forceinline__ uint4 philox(uint4 c, unsigned k0, unsigned k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
        unsigned hi0 = __umulhi(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
        unsigned hi1 = __umulhi(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    }
    return c;
}
__device__ __forceinline__ float u24(unsigned x) { return (float)(x >> 8) * (1.0f / 16777216.0f); }

// path draws: counter (pixel, sample, vertex<<8 | group, lambda<<16 | 0xFFFF)
__device__ __forceinline__ float4 path_draw(const DevJob &J, unsigned pix, unsigned s, unsigned v, unsigned g, unsigned lam)
{
    uint4 o = philox(make_uint4(pix, s, (v << 8) | g, (lam << 16) | 0xFFFFu), J.seed_lo, J.seed_hi);
    return make_float4(u24(o.x), u24(o.y), u24(o.z), u24(o.w));
}

// ------------------------------------------------------------------------------- traversal
struct HitF {
    float t, u, v;
    int tri;
};

// Triangles whose float test was within its error band (near an edge, or tied in distance):
// the closest hit among them is re-decided in the coherent arithmetic.
constexpr int NCAND = 4;

struct Counters {
    unsigned rays, boxes, tris, refines, fallbacks, shadows, bounces, samples;
};


// 32 bytes through the read-only path in one instruction (p 32-byte aligned): a node of the BVH.  Rays
// of a warp that are at different nodes take an L1 data wavefront each per load instruction, and the
// trace kernels are bound by those: a node in one load instead of two is what its 16-bit form is for.
__device__ __forceinline__ void ldg256(const uint4 *p, uint4 &a, uint4 &b)
{
    asm("ld.global.nc.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
        : "l"(p));
}

__device__ __forceinline__ void ldg256(const float4 *p, float4 &a, float4 &b)
{
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(a.x), "=f"(a.y), "=f"(a.z), "=f"(a.w), "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
        : "l"(p));
}

// Closest (or any) hit of a float ray against the BVH.  TRACK: collect the triangles met within
// NEAR_MARGIN of an edge, or tied in distance within TIE_REL, no farther than the float winner,
// so that the caller can re-decide the hit in the coherent arithmetic.  The traversal stack has
// slimit entries (stride SSTRIDE), one of them the sentinel: a near-first traversal holds at most one
// far child per inner level of its path, and slimit is at least the tree's depth (its inner levels,
// at most TSTACK - 1 by construction) plus one, so only the checked build looks.
//
// What bounds it (30-sphere scene, the pixels' first rays): issue (64-66 % of the slots) with a warp's
// lanes at different nodes (18 of 32 active).  With 64-byte nodes and corner boxes L1's data
// wavefronts came first (73 % busy: one per lane and load); 32-byte nodes take half of them (42 %).
// Together with the sentinel and without the bounds check of a push: 1080p frame 235 -> 223 ms,
// 185k-triangle frame 68.1 -> 62.1 ms, 64^3 bake 4.63 -> 4.37 ms, the fields the same bits.
#ifndef HPT_VOTE_F
#define HPT_VOTE_F 10
#endif
// The traversal is a state that is stepped, so that a warp can give a lane whose ray has ended another
// one while the others go on.  WIDE: the ray's scene may be a wide one.
template <bool STATS, bool TRACK, int SSTRIDE, bool WIDE>
struct Traversal {
    static constexpr int SENT = 0x7FFFFFFF;    // stack exhausted: the entry under all others
    float3 o, d;
    GridRay gr;
    HitF h;
    int n_cand;                                // TRACK: candidates met, > NCAND: some were dropped
    const uint4 *nodes;
    const float4 *tris;
    int node, leaf;                            // next node; pending leaf (< 0; 0 = none: the root is never one)
    int sp, skip;
    bool any;                                  // any hit before the ray's end, else the closest
    bool wide;                                 // nodes of 64 bytes

    __device__ __forceinline__ void start(const DevScene &sc, float3 o_, float3 d_, float tmax, int skip_, bool any_,
                                          bool primary, int *stk)
    {
        o = o_;
        d = d_;
        // approximate reciprocals (within 2 ulp): they only steer the boxes, whose slack counts with that
        const float3 inv = f3(fabsf(d.x) > 1e-20f ? __fdividef(1.0f, d.x) : copysignf(1e20f, d.x),
                              fabsf(d.y) > 1e-20f ? __fdividef(1.0f, d.y) : copysignf(1e20f, d.y),
                              fabsf(d.z) > 1e-20f ? __fdividef(1.0f, d.z) : copysignf(1e20f, d.z));
        gr = grid_ray<WIDE>(sc, o, inv);
        wide = WIDE && sc.wide;
        h.t = tmax;
        h.tri = -1;
        h.u = h.v = 0.0f;
        n_cand = 0;
        // the pixels' first rays walk the tree built for their direction; the closest hit and the
        // candidates do not depend on the tree
        nodes = primary ? sc.nodes_p : sc.nodes;
        tris = primary ? sc.tri4_p : sc.tri4;
        skip = skip_;
        any = any_;
        node = 0;
        leaf = 0;
        stk[0] = SENT;
        sp = 1;
    }
    __device__ __forceinline__ bool done() const { return node == SENT && leaf == 0; }

    // remember a candidate (once), in the thread's entries above the stack
    __device__ __forceinline__ void add_cand(int *cands, int id)
    {
        for (int k = 0; k < min(n_cand, NCAND); ++k)
            if (cands[k * SSTRIDE] == id) return;
        if (n_cand < NCAND) cands[n_cand * SSTRIDE] = id;
        ++n_cand;
    }

    // Descend, then test a leaf.  Speculative descent (Aila and Laine 2009): a leaf met while none is
    // pending is postponed and the descent continues until all but a few of the warp's rays hold a leaf
    // (HPT_VOTE_F / 32 of those that came in); then each tests one leaf and descends again, so that no
    // lane waits long for another's second leaf or last nodes.  Culling uses the closest hit known so
    // far, so only the order of the visits changes: the closest hit (ties to the lower id) is the same,
    // and the candidates of a coherent ray, re-decided exactly, lead to the same decision.
    // 1080p frame: all rays hold a leaf and every leaf is tested 198.8 ms, all but 8/32 and one leaf 192.4,
    // 12/32 193.0, 16/32 195.7; one triangle instead of one leaf 202.8.
    __device__ __forceinline__ void step(const DevScene &sc, bool primary, int *stk, int slimit, int &status, Counters &cnt)
    {
        const float cull = TRACK ? (1.0f + 4.0f * TIE_REL) : 1.0f;
        const int few = (__popc(__activemask()) * HPT_VOTE_F) >> 5;
        while ((unsigned)node < (unsigned)SENT) {
            if (!HPT_IN(node, primary ? sc.n_nodes_p : sc.n_nodes)) {
                status |= ST_BOUNDS;
                node = SENT;
                break;
            }
            uint4 na, nb;
            float2 c[3], hh[3];
            int l0, l1;
            if (WIDE && wide) {
                float4 fa, fb;
                ldg256(reinterpret_cast<const float4 *>(nodes + 4 * node), fa, fb);
                ldg256(nodes + 4 * node + 2, na, nb);
                c[0] = make_float2(fa.x, fa.y);
                c[1] = make_float2(fa.z, fa.w);
                c[2] = make_float2(fb.x, fb.y);
                hh[0] = make_float2(fb.z, fb.w);
                hh[1] = make_float2(__uint_as_float(na.x), __uint_as_float(na.y));
                hh[2] = make_float2(__uint_as_float(na.z), __uint_as_float(na.w));
                l0 = (int)nb.x;
                l1 = (int)nb.y;
            } else {
                ldg256(nodes + 2 * node, na, nb);
                c[0] = centres(na.x);
                c[1] = centres(na.y);
                c[2] = centres(na.z);
                hh[0] = extents(na.w);
                hh[1] = extents(nb.x);
                hh[2] = extents(nb.y);
                l0 = (int)nb.z;
                l1 = (int)nb.w;
            }
            float c0min, c0max, c1min, c1max;
            box_pair(c, hh, gr, h.t * cull, c0min, c0max, c1min, c1max);
            if (STATS) cnt.boxes += 2;
            const bool h0 = c0min <= c0max, h1 = c1min <= c1max;
            if (!h0 && !h1) {
                node = stk[(--sp) * SSTRIDE];
            } else {
                node = h0 ? l0 : l1;
                if (h0 && h1) {
                    int other = l1;
                    if (c1min < c0min) { node = l1; other = l0; }
                    if (HPT_IN(sp, slimit)) stk[(sp++) * SSTRIDE] = other;
                    else status |= ST_STACK_OVERFLOW;
                }
            }
            if (node < 0 && leaf == 0) {
                leaf = node;
                node = stk[(--sp) * SSTRIDE];
            }
            if (__popc(__ballot_sync(__activemask(), leaf == 0)) <= few) break;
        }
        if (leaf < 0) {
            // leaf: ~(start << 8 | count)
            const int code = ~leaf, start = code >> 8;
            int count = code & 255;
            if (count > 0 && !HPT_IN(start + count - 1, primary ? sc.n_tri4_p : sc.n_tri4)) {
                status |= ST_BOUNDS;
                count = 0;
            }
            for (int i = start; i < start + count; ++i) {
                const float4 *tp = tris + 3 * i;
                const float4 A = __ldg(tp), E1 = __ldg(tp + 1), E2 = __ldg(tp + 2);
                const int id = __float_as_int(A.w);
                if (STATS) cnt.tris++;
                if (id == skip) continue;
                if (!HPT_IN(id, sc.n_tris)) {
                    status |= ST_BOUNDS;
                    continue;
                }
                const float3 e1 = xyz(E1), e2 = xyz(E2);
                const float3 pv = cross3_rn(d, e2);
                const float det = dot3_rn(e1, pv);
                const float idet = __fdividef(1.0f, det);
                const float3 tv = o - xyz(A);
                const float u = __fmul_rn(dot3_rn(tv, pv), idet);
                const float3 qv = cross3_rn(tv, e1);
                const float v = __fmul_rn(dot3_rn(d, qv), idet);
                const float t = __fmul_rn(dot3_rn(e2, qv), idet);
                if (TRACK) {
                    const float m = fminf(fminf(u, v), 1.0f - u - v);
                    if (fabsf(m) < NEAR_MARGIN && t > 0.0f && t <= h.t * (1.0f + 10.0f * TIE_REL))
                        add_cand(stk + slimit * SSTRIDE, id);
                }
                // the slack of the float test of incoherent rays closes cracks between neighbours; per
                // triangle it is a band of fixed width in space (E1.w), so that large triangles do not
                // grow far past their outer edges
                const float ew = TRACK ? 0.0f : E1.w;
                const bool inside = (u >= -ew) && (v >= -ew) && (u + v <= 1.0f + ew) && (t > 0.0f);
                if (!inside) continue;
                if (!TRACK && any) {
                    if (t < h.t) {             // the ray's end
                        h.t = t;
                        h.tri = id;
                        node = SENT;
                        break;
                    }
                    continue;
                }
                if (TRACK && h.tri >= 0 && fabsf(t - h.t) <= TIE_REL * h.t) {
                    add_cand(stk + slimit * SSTRIDE, h.tri);
                    add_cand(stk + slimit * SSTRIDE, id);
                }
                if (t < h.t || (t == h.t && id < h.tri)) {
                    h.t = t; h.u = u; h.v = v; h.tri = id;
                }
            }
            leaf = 0;
            if (node < 0) {
                leaf = node;
                node = stk[(--sp) * SSTRIDE];
            }
        }
    }
};

// Double-precision closest hit used when the float traversal of a coherent ray was not
// conclusive.  Exact triangle edges (from the float32 vertices), Moller-Trumbore in double,
// ties to the lower triangle id -- the decision rule of the definition.
//
// The box tests need not be exact, only conservative: every box the double ray meets at some t
// in [0, best] must be visited, and which boxes are visited changes the work, never the winner.
// They run in float against the boxes widened by w = 2^-17 (|o|_inf + M), M the largest
// coordinate magnitude of the scene's bounds.  For a point X = o + t d inside the bounds, the
// float ray (o and d rounded to float) passes within 2^-24 (|o|_inf + |X - o|_inf) <=
// 2^-24 (2 |o|_inf + M) of X, and the slab arithmetic (the rounded reciprocal, the rounded
// origin products, one FMA) errs by a few units of 2^-24 (|o|_inf + M) in space; w covers both
// with a margin of about 8.  Culling uses the double best rounded up to float with a margin of
// 2^-16.  (GB300 runs float at 64 times the double rate; the boxes are most of the work.)
template <int SSTRIDE, bool WIDE>
__device__ __noinline__ int traverse_fp64(const DevScene &sc, double ox, double oy, double oz, double dx, double dy,
                                          double dz, double tmin, int skip, double *t_out, int *stk, int slimit,
                                          int &status)
{
    const float3 of = f3((float)ox, (float)oy, (float)oz);
    const float3 dfl = f3((float)dx, (float)dy, (float)dz);
    const float M = sc.bound;
    const float w = (fmaxf(fmaxf(fabsf(of.x), fabsf(of.y)), fabsf(of.z)) + M) * 0x1p-17f;
    const float3 inv = f3(fabsf(dfl.x) > 1e-20f ? 1.0f / dfl.x : copysignf(1e20f, dfl.x),
                          fabsf(dfl.y) > 1e-20f ? 1.0f / dfl.y : copysignf(1e20f, dfl.y),
                          fabsf(dfl.z) > 1e-20f ? 1.0f / dfl.z : copysignf(1e20f, dfl.z));
    const GridRay gr = grid_ray<WIDE>(sc, of, inv);
    const float ws[3] = {w / sc.grid.step[0], w / sc.grid.step[1], w / sc.grid.step[2]};   // w in grid steps
    double best = 1e300;
    int best_id = -1;
    float tl = 1e30f;
    int sp = 0, node = 0;
    for (;;) {
        while (node >= 0) {
            if (!HPT_IN(node, sc.n_nodes)) {
                status |= ST_BOUNDS;
                *t_out = best;
                return best_id;
            }
            // 16-byte loads: ptxas of CUDA 13.0 fails on the 32-byte form in this non-inlined function
            float2 c[3], hh[3];
            int l0, l1;
            if (WIDE && sc.wide) {
                const uint4 n0 = __ldg(sc.nodes + 4 * node), n1 = __ldg(sc.nodes + 4 * node + 1), n2 = __ldg(sc.nodes + 4 * node + 2),
                            n3 = __ldg(sc.nodes + 4 * node + 3);
                c[0] = make_float2(__uint_as_float(n0.x), __uint_as_float(n0.y));
                c[1] = make_float2(__uint_as_float(n0.z), __uint_as_float(n0.w));
                c[2] = make_float2(__uint_as_float(n1.x), __uint_as_float(n1.y));
                hh[0] = make_float2(__uint_as_float(n1.z), __uint_as_float(n1.w));
                hh[1] = make_float2(__uint_as_float(n2.x), __uint_as_float(n2.y));
                hh[2] = make_float2(__uint_as_float(n2.z), __uint_as_float(n2.w));
                l0 = (int)n3.x;
                l1 = (int)n3.y;
            } else {
                const uint4 na = __ldg(sc.nodes + 2 * node), nb = __ldg(sc.nodes + 2 * node + 1);
                c[0] = centres(na.x);
                c[1] = centres(na.y);
                c[2] = centres(na.z);
                hh[0] = extents(na.w);
                hh[1] = extents(nb.x);
                hh[2] = extents(nb.y);
                l0 = (int)nb.z;
                l1 = (int)nb.w;
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) hh[k] = make_float2(hh[k].x + ws[k], hh[k].y + ws[k]);
            float t0a, t0b, t1a, t1b;
            box_pair(c, hh, gr, tl, t0a, t0b, t1a, t1b);
            const bool h0 = t0a <= t0b, h1 = t1a <= t1b;
            if (!h0 && !h1) {
                if (sp == 0) { *t_out = best; return best_id; }
                node = stk[(--sp) * SSTRIDE];
            } else {
                node = h0 ? l0 : l1;
                if (h0 && h1) {
                    int other = l1;
                    if (t1a < t0a) { node = l1; other = l0; }
                    if (sp < slimit) stk[(sp++) * SSTRIDE] = other;
                    else status |= ST_FALLBACK_STACK;
                }
            }
        }
        int code = ~node;
        int start = code >> 8, count = code & 255;
        if (count > 0 && !HPT_IN(start + count - 1, sc.n_tri4)) {
            status |= ST_BOUNDS;
            count = 0;
        }
        for (int i = start; i < start + count; ++i) {
            int id = __float_as_int(__ldg(sc.tri4 + 3 * i).w);
            if (id == skip) continue;
            if (!HPT_IN(id, sc.n_tris)) {
                status |= ST_BOUNDS;
                continue;
            }
            // Most triangles of a leaf are missed by far, and a double test takes some thousand cycles: a
            // float test rejects those whose barycentrics are outside by more than it can err (edges and
            // directions within 2^-24 of themselves, positions within 2^-23 of |o| + |v0|; the bounds
            // are some 16 times what these and the roundings of the products come to).
            {
                const float4 A = __ldg(sc.tri4 + 3 * i), E1 = __ldg(sc.tri4 + 3 * i + 1), E2 = __ldg(sc.tri4 + 3 * i + 2);
                const float3 e1 = xyz(E1), e2 = xyz(E2), pv = cross3(dfl, e2), tv = of - xyz(A), qv = cross3(tv, e1);
                const float det = dot3(e1, pv), sg = det > 0.0f ? 1.0f : -1.0f;
                const float un = sg * dot3(tv, pv), vn = sg * dot3(dfl, qv);
                const float m1 = fmaxf(fmaxf(fabsf(e1.x), fabsf(e1.y)), fabsf(e1.z)), m2 = fmaxf(fmaxf(fabsf(e2.x), fabsf(e2.y)), fabsf(e2.z));
                const float mo = fmaxf(fmaxf(fabsf(of.x), fabsf(of.y)), fabsf(of.z)) + fmaxf(fmaxf(fabsf(A.x), fabsf(A.y)), fabsf(A.z));
                const float eu = 0x1p-16f * mo * m2, ev = 0x1p-16f * mo * m1, ed = 0x1p-16f * m1 * m2;
                if (fabsf(det) > ed && (un < -eu || vn < -ev || un + vn > fabsf(det) + eu + ev + ed)) continue;
            }
            uint4 ix4 = __ldg(sc.tri_attr + id);
            const float4 p0 = __ldg(sc.vrec + 2 * ix4.x), p1 = __ldg(sc.vrec + 2 * ix4.y), p2 = __ldg(sc.vrec + 2 * ix4.z);
            double v0x = p0.x, v0y = p0.y, v0z = p0.z;
            double e1x = (double)p1.x - v0x, e1y = (double)p1.y - v0y, e1z = (double)p1.z - v0z;
            double e2x = (double)p2.x - v0x, e2y = (double)p2.y - v0y, e2z = (double)p2.z - v0z;
            double px = dy * e2z - dz * e2y, py = dz * e2x - dx * e2z, pz = dx * e2y - dy * e2x;
            double det = e1x * px + e1y * py + e1z * pz;
            if (det == 0.0) continue;
            double id_ = 1.0 / det;
            double tx = ox - v0x, ty = oy - v0y, tz = oz - v0z;
            double u = (tx * px + ty * py + tz * pz) * id_;
            double qx = ty * e1z - tz * e1y, qy = tz * e1x - tx * e1z, qz = tx * e1y - ty * e1x;
            double v = (dx * qx + dy * qy + dz * qz) * id_;
            double t = (e2x * qx + e2y * qy + e2z * qz) * id_;
            if (u < 0.0 || v < 0.0 || u + v > 1.0 || !(t > tmin)) continue;
            if (t < best || (t == best && id < best_id)) {
                best = t;
                best_id = id;
                tl = __double2float_ru(best) * (1.0f + 0x1p-16f);
            }
        }
        if (sp == 0) break;
        node = stk[(--sp) * SSTRIDE];
    }
    *t_out = best;
    return best_id;
}

// ------------------------------------------------------------------------ surface and BSDFs
struct Surf {
    float3 p, ng, ns;   // point, unit geometric normal (winding), unit shading normal
    float u, v;         // texture coordinates
    int tri, mat;
};

// a vertex record: position, shading normal, texture coordinates, in one 32-byte load
struct Vert {
    float3 p, n;
    float u, v;
};
__device__ __forceinline__ Vert vertex_of(const DevScene &sc, unsigned i)
{
    float4 a, b;
    ldg256(sc.vrec + 2 * (size_t)i, a, b);
    Vert r;
    r.p = f3(a.x, a.y, a.z);
    r.n = f3(a.w, b.x, b.y);
    r.u = b.z;
    r.v = b.w;
    return r;
}

// the surface at barycentrics b1, b2 of a triangle with vertices V0, V1, V2
__device__ __forceinline__ Surf make_surf(const DevScene &sc, int tri, int mat, const Vert &V0, const Vert &V1, const Vert &V2,
                                          float3 p, float b1, float b2)
{
    Surf S;
    S.p = p;
    S.tri = tri;
    S.mat = mat;
    S.ng = xyz(__ldg(sc.tri_ng + tri));
    float b0 = 1.0f - b1 - b2;
    float3 n = f3(b0 * V0.n.x + b1 * V1.n.x + b2 * V2.n.x, b0 * V0.n.y + b1 * V1.n.y + b2 * V2.n.y,
                  b0 * V0.n.z + b1 * V1.n.z + b2 * V2.n.z);
    S.ns = normalize3(n);
    S.u = b0 * V0.u + b1 * V1.u + b2 * V2.u;
    S.v = b0 * V0.v + b1 * V1.v + b2 * V2.v;
    return S;
}
__device__ __forceinline__ Surf make_surf(const DevScene &sc, int tri, float3 p, float b1, float b2)
{
    const uint4 ix = __ldg(sc.tri_attr + tri);
    return make_surf(sc, tri, (int)ix.w, vertex_of(sc, ix.x), vertex_of(sc, ix.y), vertex_of(sc, ix.z), p, b1, b2);
}

__device__ __forceinline__ float tex_lookup(const DevScene &sc, int tex, float u, float v, int ch)
{
    int off = __ldg(sc.tex_info + 3 * tex), w = __ldg(sc.tex_info + 3 * tex + 1), hgt = __ldg(sc.tex_info + 3 * tex + 2);
    float x = u * (float)w - 0.5f, y = v * (float)hgt - 0.5f;
    float fx0 = floorf(x), fy0 = floorf(y);
    float fx = x - fx0, fy = y - fy0;
    int x0 = (int)fx0, y0 = (int)fy0, x1 = x0 + 1, y1 = y0 + 1;
    x0 = min(max(x0, 0), w - 1); x1 = min(max(x1, 0), w - 1);
    y0 = min(max(y0, 0), hgt - 1); y1 = min(max(y1, 0), hgt - 1);
    const float *d = sc.tex + off;
    float a = __ldg(d + (y0 * w + x0) * 3 + ch), b = __ldg(d + (y0 * w + x1) * 3 + ch);
    float c = __ldg(d + (y1 * w + x0) * 3 + ch), e = __ldg(d + (y1 * w + x1) * 3 + ch);
    return (a * (1.0f - fx) + b * fx) * (1.0f - fy) + (c * (1.0f - fx) + e * fx) * fy;
}

__device__ __forceinline__ float albedo_of(const DevScene &sc, const MatDev &M, const Surf &S, int ch)
{
    float a = M.albedo[ch];
    return M.tex >= 0 ? a * tex_lookup(sc, M.tex, S.u, S.v, ch) : a;
}

__device__ __forceinline__ float emitted(const DevScene &sc, const MatDev &M, const Surf &S, float3 wo, int ch)
{
    float Le = M.Le[ch];
    if (Le == 0.0f || dot3(wo, S.ng) <= 0.0f) return 0.0f;
    if (M.emit_tex && M.tex >= 0) Le *= tex_lookup(sc, M.tex, S.u, S.v, ch);
    return Le;
}

__device__ __forceinline__ float cache_lookup(const DevScene &sc, float3 p, int ch)
{
    int R = sc.cache_res;
    float g[3] = {p.x, p.y, p.z}, f[3];
    int i0[3], i1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float lo = sc.cache_bmin[k], hi = sc.cache_bmax[k];
        float gg = (g[k] - lo) / (hi - lo) * (float)R - 0.5f;
        float fl = floorf(gg);
        f[k] = gg - fl;
        int a = (int)fl, b = a + 1;
        i0[k] = min(max(a, 0), R - 1);
        i1[k] = min(max(b, 0), R - 1);
    }
    float acc = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        int ix = (c & 1) ? i1[0] : i0[0], iy = (c & 2) ? i1[1] : i0[1], iz = (c & 4) ? i1[2] : i0[2];
        float w = ((c & 1) ? f[0] : 1.0f - f[0]) * ((c & 2) ? f[1] : 1.0f - f[1]) * ((c & 4) ? f[2] : 1.0f - f[2]);
        unsigned short hb = __ldg(sc.cache + (((size_t)iz * R + iy) * R + ix) * 3 + ch);
        acc += w * __half2float(__ushort_as_half(hb));
    }
    return acc;
}

// orthonormal basis around a unit normal (Duff et al., JCGT 2017)
__device__ __forceinline__ void make_frame(float3 n, float3 &t, float3 &b)
{
    float sg = n.z >= 0.0f ? 1.0f : -1.0f;
    float a = -1.0f / (sg + n.z);
    float c = n.x * n.y * a;
    t = f3(1.0f + sg * n.x * n.x * a, sg * c, -sg * n.x);
    b = f3(c, sg + n.y * n.y * a, -n.y);
}

__device__ __forceinline__ float fresnel_dielectric(float ci, float n_i, float n_t)
{
    float eta = n_i / n_t;
    float s2 = eta * eta * (1.0f - ci * ci);
    if (s2 >= 1.0f) return 1.0f;
    float ct = sqrtf(1.0f - s2);
    float rs = (n_i * ci - n_t * ct) / (n_i * ci + n_t * ct);
    float rp = (n_t * ci - n_i * ct) / (n_t * ci + n_i * ct);
    return 0.5f * (rs * rs + rp * rp);
}

__device__ __forceinline__ float ggx_D(float a, float3 h)
{
    if (h.z <= 0.0f) return 0.0f;
    float a2 = a * a;
    float q = sum2_rn(h.x, h.x, h.y, h.y) / a2 + h.z * h.z;
    return 1.0f / (PI_F * a2 * q * q);
}
__device__ __forceinline__ float ggx_G1(float a, float3 w)
{
    if (w.z <= 0.0f) return 0.0f;
    float t2 = sum2_rn(w.x, w.x, w.y, w.y) / (w.z * w.z);
    float lam = 0.5f * (-1.0f + sqrtf(1.0f + a * a * t2));
    return 1.0f / (1.0f + lam);
}
__device__ __forceinline__ float schlick(float F0, float c)
{
    float m = 1.0f - c;
    float m2 = m * m;
    return F0 + (1.0f - F0) * m2 * m2 * m;
}

// BSDF value and sampling pdf of a non-delta material (world-frame directions); a = albedo
__device__ __forceinline__ void bsdf_eval(const MatDev &M, float a, float3 ns, float3 wo, float3 wi, float &f,
                                          float &pdf)
{
    f = 0.0f;
    pdf = 0.0f;
    if (M.kind == 0) {
        float c = dot3(wi, ns);
        if (c <= 0.0f) return;
        f = a * INV_PI_F;
        pdf = c * INV_PI_F;
    } else if (M.kind == 1) {
        float3 t, b;
        make_frame(ns, t, b);
        float3 lo = f3(dot3_zyx(wo, t), dot3_zyx(wo, b), dot3_zxy(wo, ns));
        float3 li = f3(dot3_zxy(wi, t), dot3_zxy(wi, b), dot3_zxy(wi, ns));
        if (lo.z <= 0.0f || li.z <= 0.0f) return;
        float al = M.rough * M.rough;
        float3 h = lo + li;
        h = h * rsqrtf(dot3_zxy(h, h));
        float D = ggx_D(al, h);
        float G1o = ggx_G1(al, lo), G1i = ggx_G1(al, li);
        float F = schlick(a, dot3_zxy(li, h));
        f = F * D * G1o * G1i / (4.0f * lo.z * li.z);
        pdf = G1o * D / (4.0f * lo.z);
    }
}

}  // namespace hpt
