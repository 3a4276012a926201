// Wavefront kernels of the wave path tracer (templated on the coherent arithmetic R).
//
// A wave holds the paths of consecutive (wavelength, pixel) work items with all of their N
// samples; path p of a segment is sample s = p / n_items of item p % n_items, so adjacent paths
// belong to adjacent pixels.  Per wave:
//   k_gen                 s1, s2: pixel centre and a direction in the SLM cone, to world space
//   (k_trace, k_shade) x (max_depth + 1)
//     k_trace             s3: closest hit of coherent and incoherent rays, any hit of shadow rays
//                         (float BVH; when the float test of a coherent ray was within its error
//                         band of an edge or a tie, the hit is re-decided among the candidates in
//                         the coherent arithmetic)
//     k_shade             s3-s5: coherent refinement and delta lobes (R arithmetic), the real
//                         image point P, incoherent vertices with NEE and BSDF sampling (Eq. 1)
//   k_accum               s6-s9: per pixel and wavelength, the K facet phases and the
//                         Kahan-compensated Path-Reuse sums (Eq. 5) in sample order
// Queues are compacted with one atomic per warp.  Each path owns its state slots, so the order
// in which queues are filled does not change any result.
//
// Frame times in the comments compare within one comment: they were taken on different scenes and poses, and
// with the kernels around as they were then.
#pragma once
#include <type_traits>

#include "hpt_device.cuh"

namespace hpt {

// an 8-byte coherent slot: a double, or a double-float as its two floats' bits
template <class R> struct RS;
template <> struct RS<double> {
    static __device__ __forceinline__ double from(unsigned a, unsigned b) { return __hiloint2double((int)b, (int)a); }
    static __device__ __forceinline__ void to(double v, unsigned &a, unsigned &b)
    {
        a = (unsigned)__double2loint(v);
        b = (unsigned)__double2hiint(v);
    }
};
template <> struct RS<df> {
    static __device__ __forceinline__ df from(unsigned a, unsigned b) { return mkdf(__uint_as_float(a), __uint_as_float(b)); }
    static __device__ __forceinline__ void to(df v, unsigned &a, unsigned &b)
    {
        a = __float_as_uint(v.hi);
        b = __float_as_uint(v.lo);
    }
};

// the coherent state of path p: origin, direction and optical path length
template <class R>
__device__ __forceinline__ void coh_load(const PathBufs &pb, int p, R3<R> &o, R3<R> &d, R &opl)
{
    const uint4 a = pb.cs0[p], b = pb.cs1[p], c = pb.cs2[p];
    const uint2 e = pb.cs3[p];
    o = r3<R>(RS<R>::from(a.x, a.y), RS<R>::from(a.z, a.w), RS<R>::from(b.x, b.y));
    d = r3<R>(RS<R>::from(b.z, b.w), RS<R>::from(c.x, c.y), RS<R>::from(c.z, c.w));
    opl = RS<R>::from(e.x, e.y);
}

template <class R>
__device__ __forceinline__ void coh_store(const PathBufs &pb, int p, const R3<R> &o, const R3<R> &d, R opl)
{
    uint4 a, b, c;
    uint2 e;
    RS<R>::to(o.x, a.x, a.y);
    RS<R>::to(o.y, a.z, a.w);
    RS<R>::to(o.z, b.x, b.y);
    RS<R>::to(d.x, b.z, b.w);
    RS<R>::to(d.y, c.x, c.y);
    RS<R>::to(d.z, c.z, c.w);
    RS<R>::to(opl, e.x, e.y);
    pb.cs0[p] = a;
    pb.cs1[p] = b;
    pb.cs2[p] = c;
    pb.cs3[p] = e;
}

enum : int { VF_V = 0xFF, VF_PREV_DELTA = 1 << 8, VF_INC_FIRST = 1 << 9, VF_HASP = 1 << 10, VF_BAKE = 1 << 11 };
constexpr int Q_FINALIZE = (int)0x80000000;   // no ray: a path that only waits for its shadow ray, or none
constexpr int Q_FIRST = 0x40000000;           // an image point handed over by the coherent shading
constexpr int Q_PATH = 0x3FFFFFFF;
// what a shading entry appends: a coherent or an incoherent entry, a finalising one, a shadow ray
enum : int { PUSH_NONE = 0, PUSH_A = 1, PUSH_A_FINAL = 2, PUSH_B = 4 };

struct PathId {
    const DevJob *J;
    int lam, ch, px, py, s;
    unsigned pix;
    bool valid;
};

__device__ __forceinline__ int seg_of_path(const WaveDesc &wd, int p)
{
    int k = 0;
    while (k + 1 < wd.n_seg && wd.seg[k + 1].path_offset <= p) ++k;
    return k;
}

__device__ __forceinline__ int fast_div(int n, const FastDiv &f)
{
    return f.shift < 0 ? n : (int)(__umulhi((unsigned)n, f.mul) >> (f.shift - 1));
}

__device__ __forceinline__ void decode_item(const DevJob *J, long long item, PathId &id)
{
    const long long per_lam = (long long)J->n_tiles * 32;
    const int lam = item < per_lam ? 0 : (item < 2 * per_lam ? 1 : 2);   // at most three wavelengths
    const int rem = (int)(item - (long long)lam * per_lam);
    const int tile = rem >> 5, l = rem & 31;
    const int ty = fast_div(tile, J->div_tiles_x), tx = tile - ty * J->n_tiles_x;
    id.J = J;
    id.lam = lam;
    id.px = tx * TILE_W + (l & (TILE_W - 1));
    id.py = ty * TILE_H + l / TILE_W;
    id.valid = id.px < J->W && id.py < J->H && lam < J->n_lambda;
    id.ch = J->channel[lam];
    id.pix = (unsigned)(id.py * J->W + id.px);
}

__device__ __forceinline__ PathId path_id(const JobTable *jt, const WaveDesc &wd, int p)
{
    const WaveSeg &g = wd.seg[seg_of_path(wd, p)];
    const int loc = p - g.path_offset;
    const int s = fast_div(loc, g.div_items), il = loc - s * g.item_count;
    PathId id;
    decode_item(jt->jobs + g.job, g.item_begin + il, id);
    id.s = s;
    return id;
}

// append to two queues at once, by a whole converged warp: lanes with a (b) add va (vb) to qa (qb).  One
// atomic instruction serves both counters (lane 0 adds to one, lane 1 to the other), so a warp waits
// for one round trip per pass of the shading loop, where an atomic per queue and per group of lanes
// that happened to be converged took up to three.
__device__ __forceinline__ void enqueue2(bool a, int va, int *qa, int *ca, bool b, int vb, int *qb, int *cb)
{
    const unsigned ma = __ballot_sync(0xFFFFFFFFu, a), mb = __ballot_sync(0xFFFFFFFFu, b);
    const int lane = threadIdx.x & 31;
    int base = 0;
    if (lane < 2) {
        const int n = __popc(lane ? mb : ma);
        if (n) base = atomicAdd(lane ? cb : ca, n);
    }
    const int ba = __shfl_sync(0xFFFFFFFFu, base, 0), bb = __shfl_sync(0xFFFFFFFFu, base, 1);
    const unsigned below = (1u << lane) - 1u;
    if (a) qa[ba + __popc(ma & below)] = va;
    if (b) qb[bb + __popc(mb & below)] = vb;
}

__device__ __forceinline__ void flush_counters(const Counters &cnt, SlotScratch *scr)
{
    const unsigned v[8] = {cnt.samples, cnt.rays, cnt.boxes, cnt.tris, cnt.refines, cnt.fallbacks, cnt.shadows, cnt.bounces};
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        unsigned long long x = v[k];
        for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, off);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(&scr->counters[k], x);
    }
}

// ------------------------------------------------------------------------------- s1 + s2
template <class R>
__global__ void __launch_bounds__(GEN_BLOCK) k_gen(const JobTable *__restrict__ jt, const WaveDesc wd, PathBufs pb,
                                                   SlotScratch *__restrict__ scr)
{
    using RO = RealOps<R>;
    const int p = blockIdx.x * GEN_BLOCK + threadIdx.x;
    if (p >= wd.n_paths) return;
    const PathId id = path_id(jt, wd, p);
    pb.amp[p] = 0.0f;
    if (id.J->kind == 1) {
        // cache bake (a wave of bake jobs only): every path starts as an incoherent ray from its
        // cell centre in a direction uniform on the sphere, drawn at vertex 0
        if (p == 0) scr->qcount[0][1] = wd.n_paths;
        pb.q[1][0][p] = id.valid ? p : (p | Q_FINALIZE);
        pb.inc[p] = make_float4(0.0f, 1.0f, 0.0f, 0.0f);
        pb.inc2[p] = make_float2(0.0f, __int_as_float(0));
        if (!id.valid) return;
        const DevJob &J = *id.J;
        const float4 u = path_draw(J, id.pix, (unsigned)id.s, 0u, 0u, (unsigned)id.lam);
        const float ct = 1.0f - 2.0f * u.x, st = 2.0f * sqrtf(u.x * (1.0f - u.x));
        float sp, cp;
        sincospif(2.0f * u.y, &sp, &cp);
        const int iy = id.py % J.W, iz = id.py / J.W;
        const float3 x = f3(J.bake_lo[0] + ((float)id.px + 0.5f) * J.bake_h[0], J.bake_lo[1] + ((float)iy + 0.5f) * J.bake_h[1],
                            J.bake_lo[2] + ((float)iz + 0.5f) * J.bake_h[2]);
        pb.ray_o[p] = make_float4(x.x, x.y, x.z, 1e30f);
        pb.ray_d[p] = make_float4(st * cp, st * sp, ct, __int_as_float(-1));
        pb.inc2[p] = make_float2(0.0f, __int_as_float(VF_PREV_DELTA | VF_BAKE));
        return;
    }
    // the first coherent queue is the identity; paths of pixels outside a ragged SLM are marked
    if (p == 0) scr->qcount[0][0] = wd.n_paths;
    pb.q[0][0][p] = id.valid ? p : (p | Q_FINALIZE);
    if (!id.valid) return;
    const DevJob &J = *id.J;
    const float4 u = path_draw(J, id.pix, (unsigned)id.s, 0u, 0u, (unsigned)id.lam);
    const R x = RO::mulf(RO::rc(J.pitch), (float)id.px + 0.5f - 0.5f * (float)J.W);
    const R y = RO::mulf(RO::rc(J.pitch), (float)id.py + 0.5f - 0.5f * (float)J.H);
    const R s1 = RO::mulf(RO::rc(J.h_cone[id.lam]), u.x);    // 1 - cos(theta)
    const R ct = RO::f(1.0f) - s1;
    const R sn = RO::sqrt_(s1 * (RO::f(2.0f) - s1));
    R sp, cp;
    RO::sincos2pi(u.y, J.sincos_tab, sp, cp);
    const R3<R> dh = r3<R>(sn * cp, sn * sp, ct);
    R3<R> co, cd;
    if (J.t_identity) {
        co = r3<R>(x, y, RO::f(0.0f));
        cd = dh;
    } else {
        // T = [Rm | t]: world origin Rm^T (x - t), world direction Rm^T d (Eq. 3, rigid T)
        const R3<R> q = r3<R>(x - RO::rc(J.t[0]), y - RO::rc(J.t[1]), -RO::rc(J.t[2]));
        const R3<R> c0 = r3<R>(RO::rc(J.R[0]), RO::rc(J.R[3]), RO::rc(J.R[6]));
        const R3<R> c1 = r3<R>(RO::rc(J.R[1]), RO::rc(J.R[4]), RO::rc(J.R[7]));
        const R3<R> c2 = r3<R>(RO::rc(J.R[2]), RO::rc(J.R[5]), RO::rc(J.R[8]));
        co = r3<R>(rdot(c0, q), rdot(c1, q), rdot(c2, q));
        cd = r3<R>(rdot(c0, dh), rdot(c1, dh), rdot(c2, dh));
    }
    coh_store<R>(pb, p, co, cd, RO::f(0.0f));
    pb.coh4[p] = make_float4(1.0f, 1.0f, RO::to_f(ct), __int_as_float(0));
    pb.inc2[p] = make_float2(0.0f, __int_as_float(0));
    const float3 of = tof3(co), df_ = tof3(cd);
    pb.ray_o[p] = make_float4(of.x, of.y, of.z, 1e30f);
    pb.ray_d[p] = make_float4(df_.x, df_.y, df_.z, __int_as_float(-1));
}

// After k_gen, in waves with a job whose first rays begin far from the scene (J.far): their float rays are moved
// along the paths' own rays towards the geometry; the second time takes back what float error the first
// left.  Nothing depends on a first ray's distance but the hit that it finds: the coherent shading works out
// the distance from the path's own origin, and the bake's first vertex weighs no light by it.  (In k_gen this
// took its 32 registers to 48, or spilled.)
template <class R>
__global__ void __launch_bounds__(GEN_BLOCK) k_start_near(const JobTable *__restrict__ jt, const WaveDesc wd, PathBufs pb)
{
    const int p = blockIdx.x * GEN_BLOCK + threadIdx.x;
    if (p >= wd.n_paths) return;
    const PathId id = path_id(jt, wd, p);
    if (!id.valid || !id.J->far) return;
    const float4 r = pb.ray_o[p];
    const float3 df_ = xyz(pb.ray_d[p]);
    float3 of = xyz(r);
    R3<R> o = fromf3<R>(of), d = fromf3<R>(df_);
    R opl;
    if (id.J->kind != 1) coh_load<R>(pb, p, o, d, opl);
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
        o = o + scale(d, RealOps<R>::f(far_start(id.J->bounds, of, df_)));
        of = tof3(o);
    }
    pb.ray_o[p] = make_float4(of.x, of.y, of.z, r.w);
}

// ------------------------------------------------------------------------------------ s3
template <class R> __device__ __forceinline__ bool r_less(R a, R b);
template <> __device__ __forceinline__ bool r_less<double>(double a, double b) { return a < b; }
template <> __device__ __forceinline__ bool r_less<df>(df a, df b) { return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo); }
template <class R> __device__ __forceinline__ bool r_nonneg(R a);
template <> __device__ __forceinline__ bool r_nonneg<double>(double a) { return a >= 0.0; }
template <> __device__ __forceinline__ bool r_nonneg<df>(df a) { return a.hi > 0.0f || (a.hi == 0.0f && a.lo >= 0.0f); }

// a triangle's refinement record
template <class R> __device__ __forceinline__ void load_ref(const DevScene &sc, int tri, R q[REF_N])
{
#pragma unroll
    for (int i = 0; i < REF_N; i += 2) RealOps<R>::load2(sc.ref64, sc.refdf, tri * REF_N + i, q[i], q[i + 1]);
}

// Plane intersection and barycentric inside test of one triangle in the coherent arithmetic
// (the decision rule of the definition: closed triangle, distance beyond tmin).
template <class R>
__device__ __forceinline__ bool exact_hit(const DevScene &sc, int tri, const R3<R> &co, const R3<R> &cd, R tmin, R &t)
{
    using RO = RealOps<R>;
    R q[REF_N];
    load_ref<R>(sc, tri, q);
    const R3<R> n = r3<R>(q[0], q[1], q[2]);
    const R den = rdot(n, cd);
    if (RO::to_f(den) == 0.0f) return false;
    t = (q[3] - rdot(n, co)) / den;
    if (!r_less<R>(tmin, t)) return false;
    const uint4 ix = __ldg(sc.tri_attr + tri);
    const R3<R> dP = (co + scale(cd, t)) - fromf3<R>(xyz(__ldg(sc.vrec + 2 * ix.x)));
    const R b1 = rdot(r3<R>(q[4], q[5], q[6]), dP);
    const R b2 = rdot(r3<R>(q[7], q[8], q[9]), dP);
    return r_nonneg<R>(b1) && r_nonneg<R>(b2) && r_nonneg<R>(RO::f(1.0f) - b1 - b2);
}

// The hit of a coherent ray whose float test was within its error band: decided among the candidates
// and the float winner in the coherent arithmetic; by a full double traversal only when the list
// overflowed or no candidate holds.  Rare (0.06 % of the rays), so a function of its own.
struct Decision {
    int tri;
    unsigned status;
    bool fallback;
};
template <class R, bool WIDE>
__device__ __noinline__ Decision redecide(const DevScene *scp, const R3<R> co, const R3<R> cd, bool cont, int tri, int n_cand,
                                          float4 ids, int skip)
{
    using RO = RealOps<R>;
    const DevScene &sc = *scp;
    const R tmin = cont ? RO::fromd(COH_TMIN) : RO::f(0.0f);   // cont: a continuation after a delta vertex
    Decision r = {-1, 0u, false};
    R bt = RO::f(0.0f);
    if (n_cand <= NCAND) {
        for (int k = -1; k < n_cand; ++k) {
            const int id = k < 0 ? tri : __float_as_int(k == 0 ? ids.x : (k == 1 ? ids.y : (k == 2 ? ids.z : ids.w)));
            if (id < 0 || id == skip) continue;
            if (!HPT_IN(id, sc.n_tris)) {
                r.status |= ST_BOUNDS;
                continue;
            }
            R tk;
            if (exact_hit<R>(sc, id, co, cd, tmin, tk) &&
                (r.tri < 0 || r_less<R>(tk, bt) || (!r_less<R>(bt, tk) && id < r.tri))) {
                r.tri = id;
                bt = tk;
            }
        }
    }
    if (r.tri < 0) {
        r.fallback = true;
        int stk[TSTACK], status = 0;
        double tt;
        r.tri = traverse_fp64<1, WIDE>(sc, RO::to_d(co.x), RO::to_d(co.y), RO::to_d(co.z), RO::to_d(cd.x), RO::to_d(cd.y),
                                 RO::to_d(cd.z), cont ? COH_TMIN : 0.0, skip, &tt, stk, TSTACK, status);
        r.status |= (unsigned)status;
    }
    return r;
}

// resident blocks per SM the trace and shading kernels are compiled for (bounds their registers)
#ifndef HPT_SHADE_MINB
#define HPT_SHADE_MINB 6            // 80 registers, for the state loads that are in flight together (1080p frame, both
                                    // kernels at 9 / 8 / 7 / 6 / 5 blocks: 221.5 / 219.1 / 216.5 / 214.3 / 216.2 ms)
#endif
#ifndef HPT_SHADE_INC_MINB
#define HPT_SHADE_INC_MINB HPT_SHADE_MINB   // the incoherent shading kernel
#endif
// The two trace kernels keep the same shared memory a block and blocks an SM: with different ones an SM
// has to drain one kernel before it can take the other's carveout (5 % of the frame).  56 registers:
// 1080p frame at 8 / 9 / 10 / 12 blocks 203.6 / 198.3 / 207.8 / 256.1 ms.
#ifndef HPT_TRACE_MINB
#define HPT_TRACE_MINB 9
#endif
#ifndef HPT_TRACE_INC_MINB
#define HPT_TRACE_INC_MINB 9        // the incoherent / shadow-ray trace kernel
#endif
#ifndef HPT_TRACE_WIDE_MINB
#define HPT_TRACE_WIDE_MINB 8       // of wide scenes: twelve floats a node (3 m clusters at 9 / 8 blocks 12.2 / 10.5 ms)
#endif
#ifndef HPT_REFILL
#define HPT_REFILL (COH ? 16 : 12)
#endif
#ifndef HPT_ACCUM_MINB
#define HPT_ACCUM_MINB 5            // 96 registers, for the samples loaded ahead (1080p frame at 8 / 7 / 5 blocks
                                    // 188.2 / 187.0 / 185.7 ms; one sample at a time 190.5)
#endif

// COH = true: the coherent queue of the iteration (closest hit, uncertain ones decided in the coherent
// arithmetic); false: the incoherent and shadow queues (float closest / any hit only).  WIDE: for waves with a
// wide scene.
template <class R, bool STATS, bool COH, bool WIDE>
__global__ void __launch_bounds__(TRACE_BLOCK, WIDE ? HPT_TRACE_WIDE_MINB : COH ? HPT_TRACE_MINB : HPT_TRACE_INC_MINB)
    k_trace(const JobTable *__restrict__ jt, const WaveDesc wd, PathBufs pb, SlotScratch *__restrict__ scr, int it)
{
    using RO = RealOps<R>;
    extern __shared__ int s_stack[];          // wd.stack_n traversal stack entries per thread
    int *stk = s_stack + threadIdx.x;
    const int slimit = wd.stack_n;
    const int ni = scr->qcount[it][COH ? 0 : 1], total = ni + (COH ? 0 : scr->qcount[it][2]);
    const int par = it & 1;
    int status = 0;
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
    // A warp takes every nwarps-th chunk of 32 queue entries; its lanes take the entries of its chunks in
    // turn, a lane that has finished its ray another one as soon as HPT_REFILL lanes have (rays of
    // neighbouring pixels need from a few to over a hundred steps, and a warp that kept its 32 rays ran
    // for the longest with 13 lanes active).  It pays since nodes are one L1 wavefront a lane: then rays
    // at unlike depths cost L1 little.  1080p frame with a refill at 32 / 20 / 16 / 12 / 8 idle lanes: 221.5
    // / 206.7 / 206.6 / 204.8 / 206.3 ms.
    const int lane = threadIdx.x & 31, nwarps = gridDim.x * (TRACE_BLOCK / 32);
    const int warp = blockIdx.x * (TRACE_BLOCK / 32) + (threadIdx.x >> 5);
    auto entry_of = [&](int v) { return ((v >> 5) * nwarps + warp) * 32 + (v & 31); };   // the warp's v-th entry
    int taken = 0;                       // entries of the warp's chunks handed out
    int p = -1;                          // the lane's path, -1: none
    int n_uncertain = 0;
    Traversal<STATS, COH, TRACE_BLOCK, WIDE> tr;
    tr.node = Traversal<STATS, COH, TRACE_BLOCK, WIDE>::SENT;
    tr.leaf = 0;
    for (;;) {
        const bool busy = p >= 0 && !tr.done();
        if (__popc(__ballot_sync(0xFFFFFFFFu, busy)) <= 32 - HPT_REFILL) {
            bool uncertain = false;
            int q = -1;
            if (p >= 0 && !busy) {
                // the ray's result
                if (!COH && tr.any) {
                    pb.occl[p] = tr.h.tri >= 0 ? 1 : 0;
                } else if (!COH) {
                    pb.hit[p] = make_float4(tr.h.t, tr.h.u, tr.h.v, __int_as_float(tr.h.tri));
                } else {
                    // where the float test was within its error band the hit is decided below: the number
                    // of candidates goes with the hit, their ids to the path's shadow slot
                    uncertain = tr.n_cand > 0;
                    if (uncertain) {
                        const int *c = stk + slimit * TRACE_BLOCK;
                        float4 ids = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        ids.x = __int_as_float(c[0]);
                        if (tr.n_cand > 1) ids.y = __int_as_float(c[TRACE_BLOCK]);
                        if (tr.n_cand > 2) ids.z = __int_as_float(c[2 * TRACE_BLOCK]);
                        if (tr.n_cand > 3) ids.w = __int_as_float(c[3 * TRACE_BLOCK]);
                        pb.sh_d[p] = ids;
                    }
                    pb.hit[p] = make_float4(tr.h.t, __int_as_float(tr.n_cand), 0.0f, __int_as_float(tr.h.tri));
                }
                q = p;
                p = -1;
            }
            if (COH) {
                // the warp's uncertain hits, listed in its own part of the next coherent queue, which is
                // filled only by the shading after this kernel
                const unsigned m = __ballot_sync(0xFFFFFFFFu, uncertain);
                if (uncertain) pb.q[0][par ^ 1][entry_of(n_uncertain + __popc(m & ((1u << lane) - 1u)))] = q;
                n_uncertain += __popc(m);
            }
            __syncwarp();
            // new rays for the idle lanes; an entry may have none (Q_FINALIZE)
            for (;;) {
                const unsigned idle = __ballot_sync(0xFFFFFFFFu, p < 0);
                if (__popc(idle) < HPT_REFILL || entry_of(taken) >= total) break;
                if (p < 0) {
                    const int idx = entry_of(taken + __popc(idle & ((1u << lane) - 1u)));
                    const int kind = COH ? 0 : (idx < ni ? 1 : 2), qi = kind == 2 ? idx - ni : idx;
                    int e = Q_FINALIZE;
                    if (idx < total) {
                        if (HPT_IN(qi, pb.capacity)) e = pb.q[kind][par][qi];
                        else status |= ST_BOUNDS;
                    }
                    if (!(e & Q_FINALIZE)) {
                        if (!HPT_IN(e, wd.n_paths)) {
                            status |= ST_BOUNDS;
                        } else {
                            const DevScene &sc = jt->jobs[wd.seg[seg_of_path(wd, e)].job].sc;
                            const float4 o4 = pb.ray_o[e], d4 = pb.ray_d[e];
                            if (STATS) cnt.rays++;
                            if (kind == 2) {
                                const float4 s4 = pb.sh_d[e];
                                if (STATS) cnt.shadows++;
                                tr.start(sc, xyz(o4), xyz(s4), s4.w, __float_as_int(d4.w), true, false, stk);
                            } else {
                                if (STATS && kind == 1) cnt.bounces++;
                                tr.start(sc, xyz(o4), xyz(d4), 1e30f, __float_as_int(d4.w), false, COH && it == 0, stk);
                            }
                            p = e;
                        }
                    }
                }
                taken += __popc(idle);
            }
            if (!__any_sync(0xFFFFFFFFu, p >= 0)) break;
        }
        if (p >= 0 && !tr.done()) {
            const DevScene &sc = HPT_CHECKED ? jt->jobs[wd.seg[seg_of_path(wd, p)].job].sc : jt->jobs[0].sc;   // sizes to check against
            tr.step(sc, COH && it == 0, stk, slimit, status, cnt);
        }
        __syncwarp();
    }
    if (COH) {
        // Decide the uncertain hits in the coherent arithmetic.  Rare (0.06 % of the rays) and costly
        // (double precision), so after the warp's rays and in a function of its own: in the loop above its
        // registers would be spilled around it, and in the shading it took that kernel's registers and
        // instruction cache.
        __syncwarp();
        for (int v = lane; v < n_uncertain; v += 32) {
            const int u = pb.q[0][par ^ 1][entry_of(v)];
            R3<R> co, cd;
            R opl_unused;
            coh_load<R>(pb, u, co, cd, opl_unused);
            const float4 h = pb.hit[u];
            const Decision r = redecide<R, WIDE>(&jt->jobs[wd.seg[seg_of_path(wd, u)].job].sc, co, cd, __float_as_int(pb.coh4[u].w) > 0,
                                           __float_as_int(h.w), __float_as_int(h.y), pb.sh_d[u], __float_as_int(pb.ray_d[u].w));
            pb.hit[u] = make_float4(h.x, 0.0f, 0.0f, __int_as_float(r.tri));
            status |= (int)r.status;
            if (STATS) {
                cnt.refines++;
                cnt.fallbacks += r.fallback;
            }
        }
        __syncwarp();
    }
    if (STATS) flush_counters(cnt, scr);
    if (status) atomicOr(&scr->status, (unsigned)status);
}

// ------------------------------------------------------------------------------- s3 - s5
struct IncState {
    float L, beta, ppdf, tprev, nee;
    int vfl;
};

// One vertex of the incoherent path (Eq. 1): MIS-weighted emission, then a delta continuation,
// or the ambient cache, or NEE to a rectangular light plus a BSDF-sampled continuation.  Rays
// are written to the path's state; returns the entries to append (A: the incoherent queue, B: the shadow
// queue), PUSH_NONE when the path ends here.
__device__ __forceinline__ int vertex(const PathId &id, IncState &st, const Surf &S, float3 wo, const PathBufs &pb, int p)
{
    const DevJob &J = *id.J;
    const DevScene &sc = J.sc;
    const MatDev M = sc.mats[S.mat];
    const int ch = id.ch;
    const int v = st.vfl & VF_V;
    const bool prev_delta = st.vfl & VF_PREV_DELTA;
    const float Le = emitted(sc, M, S, wo, ch);
    if (Le > 0.0f) {
        float w = 1.0f;
        if (!prev_delta && M.kind == 4 && M.light >= 0 && sc.n_lights > 0) {
            const LightDev &Lt = sc.lights[M.light];
            const float cl = dot3(wo, f3(Lt.n[0], Lt.n[1], Lt.n[2]));
            const float pl = st.tprev * st.tprev / (cl * Lt.area) / (float)sc.n_lights;
            w = st.ppdf * st.ppdf / (st.ppdf * st.ppdf + pl * pl);
        }
        st.L += st.beta * Le * w;
    }
    if (M.kind == 4) return PUSH_NONE;
    float3 ng = S.ng, ns = S.ns;
    const bool front = dot3(wo, ng) > 0.0f;
    const float4 u = path_draw(J, id.pix, (unsigned)id.s, (unsigned)v, 0u, (unsigned)id.lam);
    if (M.kind == 2 || M.kind == 3) {
        if (v >= J.max_depth) return PUSH_NONE;
        float3 wi;
        if (M.kind == 2) {
            if (!front) { ng = -ng; ns = -ns; }
            const float c = dot3(wo, ns);
            if (c <= 0.0f) return PUSH_NONE;
            wi = ns * (2.0f * c) - wo;
            if (dot3(wi, ng) <= 0.0f) return PUSH_NONE;
            st.beta *= albedo_of(sc, M, S, ch);
        } else {
            const float n_i = front ? 1.0f : M.ior, n_t = front ? M.ior : 1.0f;
            const float3 n = front ? ns : -ns, g = front ? ng : -ng;
            const float ci = dot3(wo, n);
            if (ci <= 0.0f) return PUSH_NONE;
            const float F = fresnel_dielectric(ci, n_i, n_t);
            if (u.x < F) {
                wi = n * (2.0f * ci) - wo;
                if (dot3(wi, g) <= 0.0f) return PUSH_NONE;
            } else {
                const float eta = n_i / n_t;
                const float ct = sqrtf(fmaxf(0.0f, 1.0f - eta * eta * (1.0f - ci * ci)));
                wi = wo * (-eta) + n * (eta * ci - ct);
                if (dot3(wi, g) >= 0.0f) return PUSH_NONE;
                st.beta *= eta * eta;
            }
        }
        st.vfl = (st.vfl | VF_PREV_DELTA) & ~VF_INC_FIRST;
        st.nee = 0.0f;
        const float3 o = S.p + (dot3(wi, S.ng) > 0.0f ? S.ng : -S.ng) * INC_OFFSET;
        pb.ray_o[p] = make_float4(o.x, o.y, o.z, 1e30f);
        pb.ray_d[p] = make_float4(wi.x, wi.y, wi.z, __int_as_float(S.tri));
        return PUSH_A;
    }
    // non-delta (Lambert, GGX)
    if (!front) { ng = -ng; ns = -ns; }
    if (dot3(wo, ns) <= 0.0f) return PUSH_NONE;
    if (J.use_cache && sc.cache_res > 0 && !(st.vfl & VF_INC_FIRST)) {
        st.L += st.beta * albedo_of(sc, M, S, ch) * INV_PI_F * cache_lookup(sc, S.p, ch);
        return PUSH_NONE;
    }
    const float3 org = S.p + ng * INC_OFFSET;
    const float alb = albedo_of(sc, M, S, ch);
    bool shadow = false;
    st.nee = 0.0f;
    if (sc.n_lights > 0) {
        int li = 0;
        if (sc.n_lights > 1) {
            const float4 u2 = path_draw(J, id.pix, (unsigned)id.s, (unsigned)v, 1u, (unsigned)id.lam);
            li = min((int)(u2.x * (float)sc.n_lights), sc.n_lights - 1);
        }
        const LightDev &Lt = sc.lights[li];
        const float3 y = f3(Lt.corner[0], Lt.corner[1], Lt.corner[2]) + f3(Lt.eu[0], Lt.eu[1], Lt.eu[2]) * u.x +
                         f3(Lt.ev[0], Lt.ev[1], Lt.ev[2]) * u.y;
        const float3 dv = y - org;
        const float dist = sqrtf(dot3(dv, dv));
        const float3 wl = dv * (1.0f / dist);
        const float cl = -dot3(wl, f3(Lt.n[0], Lt.n[1], Lt.n[2]));
        const float Ll = Lt.Le[ch];
        if (cl > 0.0f && dot3(wl, ng) > 0.0f && dot3(wl, ns) > 0.0f && Ll > 0.0f) {
            float f, pbs;
            bsdf_eval(M, alb, ns, wo, wl, f, pbs);
            const float pl = dist * dist / (cl * Lt.area) / (float)sc.n_lights;
            if (f > 0.0f) {
                const float wm = v < J.max_depth ? pl * pl / (pl * pl + pbs * pbs) : 1.0f;
                st.nee = st.beta * f * dot3(wl, ns) * Ll * wm / pl;
                shadow = true;
                pb.sh_d[p] = make_float4(wl.x, wl.y, wl.z, dist * (1.0f - SHADOW_SHRINK));
            }
        }
    }
    bool bounce = false;
    float3 wi = f3(0.0f, 0.0f, 1.0f);
    if (v < J.max_depth) {
        float3 t, b;
        make_frame(ns, t, b);
        float weight = 0.0f, pbs = 0.0f;
        if (M.kind == 0) {
            const float rr = sqrtf(u.z);
            float s_, c_;
            sincospif(2.0f * u.w, &s_, &c_);
            const float z = sqrtf(1.0f - u.z);
            wi = t * (rr * c_) + b * (rr * s_) + ns * z;
            bounce = dot3(wi, ng) > 0.0f;
            weight = alb;
            pbs = z * INV_PI_F;
        } else {
            const float al = M.rough * M.rough;
            const float3 lo = f3(dot3_zyx(wo, t), dot3_zyx(wo, b), dot3_zxy(wo, ns));
            if (lo.z > 0.0f) {
                float3 vh = f3(al * lo.x, al * lo.y, lo.z);
                vh = vh * rsqrtf(dot3_zxy(vh, vh));
                const float l2 = sum2_rn(vh.x, vh.x, vh.y, vh.y);
                const float3 T1 = l2 > 0.0f ? f3(-vh.y, vh.x, 0.0f) * rsqrtf(l2) : f3(1.0f, 0.0f, 0.0f);
                const float3 T2 = f3(diff2_rn(vh.y, T1.z, vh.z, T1.y), diff2_rn(vh.z, T1.x, vh.x, T1.z),
                                     diff2_rn(vh.x, T1.y, vh.y, T1.x));
                const float rr = sqrtf(u.z);
                float s_, c_;
                sincospif(2.0f * u.w, &s_, &c_);
                const float t1 = rr * c_;
                float t2 = rr * s_;
                const float sm = 0.5f * (1.0f + vh.z);
                t2 = sum2_rn(1.0f - sm, sqrtf(fmaxf(0.0f, 1.0f - t1 * t1)), sm, t2);
                const float tz = sqrtf(fmaxf(0.0f, 1.0f - t1 * t1 - t2 * t2));
                const float3 nh = f3(fmaf(vh.x, tz, sum2_rn(T1.x, t1, T2.x, t2)), fmaf(vh.y, tz, sum2_rn(T1.y, t1, T2.y, t2)),
                                     fmaf(vh.z, tz, sum2_rn(T1.z, t1, T2.z, t2)));
                float3 ne = f3(al * nh.x, al * nh.y, fmaxf(0.0f, nh.z));
                ne = ne * rsqrtf(dot3_zxy(ne, ne));
                const float c = dot3_zxy(lo, ne);
                const float3 li = ne * (2.0f * c) - lo;
                if (li.z > 0.0f) {
                    weight = schlick(alb, dot3_zxy(li, ne)) * ggx_G1(al, li);
                    pbs = ggx_G1(al, lo) * ggx_D(al, ne) / (4.0f * lo.z);
                    wi = f3(fmaf(ns.x, li.z, sum2_rn(t.x, li.x, b.x, li.y)), fmaf(ns.y, li.z, sum2_rn(t.y, li.x, b.y, li.y)),
                            fmaf(ns.z, li.z, sum2_rn(t.z, li.x, b.z, li.y)));
                    bounce = dot3(wi, ng) > 0.0f;
                }
            }
        }
        if (bounce) {
            st.beta *= weight;
            st.ppdf = pbs;
        }
    }
    st.vfl &= ~(VF_INC_FIRST | VF_PREV_DELTA);
    if (!shadow && !bounce) return PUSH_NONE;
    // both rays leave from the same side of a reflecting surface: one origin serves both
    pb.ray_o[p] = make_float4(org.x, org.y, org.z, 1e30f);
    pb.ray_d[p] = make_float4(wi.x, wi.y, wi.z, __int_as_float(S.tri));
    return (bounce ? PUSH_A : PUSH_A_FINAL) | (shadow ? PUSH_B : PUSH_NONE);
}

// COH = true: the coherent entries of the iteration; false: the incoherent ones (two kernels,
// so that each carries only its half of the shading code).
// Bound by the latency of a chain of loads (queue entry, state, hit's triangle, its vertices and
// material, texels) and of the queue counters' atomics: so the next queue entry is loaded a pass ahead,
// the path's whole state before any of it is looked at, a vertex as one 32-byte record and a
// refinement record as 16-byte pieces, and both counters are bumped by one atomic instruction a warp.
// 1080p frame 223 -> 215 ms, two-quad 256^2 frame 181 -> 155 us, 64^3 bake 4.06 -> 3.83 ms.
template <class R, bool STATS, bool COH>
__global__ void __launch_bounds__(SHADE_BLOCK, COH ? HPT_SHADE_MINB : HPT_SHADE_INC_MINB) k_shade(const JobTable *__restrict__ jt, const WaveDesc wd, PathBufs pb,
                                                       SlotScratch *__restrict__ scr, int it)
{
    using RO = RealOps<R>;
    const int total = scr->qcount[it][COH ? 0 : 1];
    const int par = it & 1, nx = par ^ 1;
    int *qcn = scr->qcount[it + 1];
    const int *queue = pb.q[COH ? 0 : 1][par];
    // A: the next iteration's coherent / incoherent queue; B: this iteration's incoherent queue (image
    // points) / the next one's shadow queue
    int *const qa = COH ? pb.q[0][nx] : pb.q[1][nx], *const qb = COH ? pb.q[1][par] : pb.q[2][nx];
    int *const ca = COH ? &qcn[0] : &qcn[1], *const cb = COH ? &scr->qcount[it][1] : &qcn[2];
    Counters cnt = {0, 0, 0, 0, 0, 0, 0, 0};
    unsigned status = 0;
    // one entry of path p: what it appends (a bitwise or of PUSH_*)
    auto entry = [&](int e, int p) -> int {
        if (!HPT_IN(p, wd.n_paths)) {
            status |= ST_BOUNDS;
            return PUSH_NONE;
        }
        if constexpr (COH) {
            // the path's state does not depend on the hit: all of its loads start together
            const int tri = __float_as_int(pb.hit[p].w);
            R3<R> co, cd;
            R opl;
            coh_load<R>(pb, p, co, cd, opl);
            const float4 c4 = pb.coh4[p];
            if (tri < 0) return PUSH_NONE;
            const PathId id = path_id(jt, wd, p);
            const DevJob &J = *id.J;
            const DevScene &sc = J.sc;
            if (!HPT_IN(tri, sc.n_tris)) {
                status |= ST_BOUNDS;
                return PUSH_NONE;
            }
            const float ncur = c4.x;
            // distance to the triangle's plane n . x = d0 in the coherent arithmetic
            R q[REF_N];
            load_ref<R>(sc, tri, q);
            const uint4 ix = __ldg(sc.tri_attr + tri);
            const R3<R> n = r3<R>(q[0], q[1], q[2]);
            const R t = (q[3] - rdot_zxy(n, co)) / rdot_zxy(n, cd);
            const R3<R> P = co + scale(cd, t);
            opl = opl + RO::mulf(t, ncur);        // OPL = sum n_i L_i (Sec. 4.2)
            const int cv = __float_as_int(c4.w) + 1;
            const int kind = sc.mats[ix.w].kind;
            float3 ng = xyz(__ldg(sc.tri_ng + tri));
            const R3<R> dP = P - fromf3<R>(xyz(__ldg(sc.vrec + 2 * ix.x)));
            const float3 dPf = tof3(dP);
            const float3 m1f = f3(RO::to_f(q[4]), RO::to_f(q[5]), RO::to_f(q[6]));
            const float3 m2f = f3(RO::to_f(q[7]), RO::to_f(q[8]), RO::to_f(q[9]));
            const float3 Pf = tof3(P);
            const float bb1 = dot3(m1f, dPf), bb2 = dot3(m2f, dPf);
            if (kind != 2 && kind != 3) {
                // P, the real image point.  For a rigid T the virtual image point
                // Q = T (O + d_OPL v) lies at distance r = d_OPL from the pixel along the
                // sampled hologram-space direction, whose z component is cos(theta).
                const float3 dl = tof3(cd);
                const float cosP = fabsf(dot3(dl, ng));
                const R ih = RO::rc(J.inv_facet);
                pb.fturn[p] = RO::frac_f(opl * RO::rc(J.inv_lambda[id.lam]));
                if (J.phase_mode == 2) {
                    // Eq. 4: the GRF sample under Q = x + d_OPL dh on the hologram plane
                    // (rigid T), dh the sampled hologram-space direction, redrawn here
                    const float4 u0 = path_draw(J, id.pix, (unsigned)id.s, 0u, 0u, (unsigned)id.lam);
                    const R s1 = RO::mulf(RO::rc(J.h_cone[id.lam]), u0.x);
                    const R sn = RO::sqrt_(s1 * (RO::f(2.0f) - s1));
                    R sp, cp;
                    RO::sincos2pi(u0.y, J.sincos_tab, sp, cp);
                    const R xq = RO::mulf(RO::rc(J.pitch), (float)id.px + 0.5f - 0.5f * (float)J.W) + opl * (sn * cp);
                    const R yq = RO::mulf(RO::rc(J.pitch), (float)id.py + 0.5f - 0.5f * (float)J.H) + opl * (sn * sp);
                    int jx = RO::floor_i(RO::addf(xq * RO::rc(J.inv_pitch), 0.5f * (float)J.grf_nx)) % J.grf_nx;
                    int jy = RO::floor_i(RO::addf(yq * RO::rc(J.inv_pitch), 0.5f * (float)J.grf_ny)) % J.grf_ny;
                    pb.cx[p] = jx < 0 ? jx + J.grf_nx : jx;
                    pb.cy[p] = jy < 0 ? jy + J.grf_ny : jy;
                    pb.cz[p] = 0;
                } else {
                    pb.cx[p] = RO::floor_i(P.x * ih);
                    pb.cy[p] = RO::floor_i(P.y * ih);
                    pb.cz[p] = RO::floor_i(P.z * ih);
                }
                // Eq. 2 with the obliquity factor cos(theta) (unless omitted)
                const float basep = (J.obliquity ? c4.z : 1.0f) * RO::to_f(opl) / (J.pdf_w[id.lam] * cosP * J.lambda_f[id.lam]);
                pb.cs3[p] = make_uint2(__float_as_uint(basep), __float_as_uint(c4.y));
                // the incoherent part starts at P: handed to this iteration's incoherent
                // shading as a hit at distance 0 from P (vertex count cv after its increment;
                // Q_FIRST stands for the radiance, throughput and distances of a new path),
                // so that the coherent kernel carries no BSDF / NEE code
                pb.inc2[p] = make_float2(0.0f, __int_as_float((cv - 1) | VF_PREV_DELTA | VF_INC_FIRST | VF_HASP));
                pb.ray_o[p] = make_float4(Pf.x, Pf.y, Pf.z, 1e30f);
                pb.ray_d[p] = make_float4(dl.x, dl.y, dl.z, __int_as_float(tri));
                pb.hit[p] = make_float4(0.0f, bb1, bb2, __int_as_float(tri));
                return PUSH_B;
            }
            if (cv >= J.max_depth) return PUSH_NONE;
            // delta vertex: shading normal and the new direction in the coherent arithmetic
            const MatDev M = sc.mats[ix.w];
            const Vert V0 = vertex_of(sc, ix.x), V1 = vertex_of(sc, ix.y), V2 = vertex_of(sc, ix.z);
            const R b1 = rdot_zxy(r3<R>(q[4], q[5], q[6]), dP);
            const R b2 = rdot_zxy(r3<R>(q[7], q[8], q[9]), dP);
            const R b0 = RO::f(1.0f) - b1 - b2;
            R3<R> ns = r3<R>(mix3(b0, V0.n.x, b1, V1.n.x, b2, V2.n.x), mix3(b0, V0.n.y, b1, V1.n.y, b2, V2.n.y),
                             mix3(b0, V0.n.z, b1, V1.n.z, b2, V2.n.z));
            ns = scale(ns, RO::f(1.0f) / RO::sqrt_(rdot_zxy(ns, ns)));
            const R3<R> wo_r = neg(cd);
            const bool front = dot3(tof3(wo_r), ng) > 0.0f;
            R3<R> wi = cd;
            bool ok = true;
            float betac = c4.y, nnew = ncur;
            if (kind == 2) {
                if (!front) { ns = neg(ns); ng = -ng; }
                const R c = rdot_zyx(wo_r, ns);
                if (!(RO::to_f(c) > 0.0f)) ok = false;
                else {
                    wi = scale(ns, RO::mulf(c, 2.0f)) - wo_r;
                    ok = dot3(tof3(wi), ng) > 0.0f;
                    const Surf S = make_surf(sc, tri, (int)ix.w, V0, V1, V2, Pf, bb1, bb2);
                    betac *= albedo_of(sc, M, S, id.ch);
                }
            } else {
                const float n_i = front ? 1.0f : M.ior, n_t = front ? M.ior : 1.0f;
                const R3<R> nn = front ? ns : neg(ns);
                const float3 g = front ? ng : -ng;
                const R ci = rdot_zyx(wo_r, nn);
                const float cif = RO::to_f(ci);
                if (!(cif > 0.0f)) ok = false;
                else {
                    const float F = fresnel_dielectric(cif, n_i, n_t);
                    const float4 u = path_draw(J, id.pix, (unsigned)id.s, (unsigned)cv, 0u, (unsigned)id.lam);
                    if (u.x < F) {
                        wi = scale(nn, RO::mulf(ci, 2.0f)) - wo_r;
                        ok = dot3(tof3(wi), g) > 0.0f;
                    } else {
                        const R eta = RO::f(n_i) / RO::f(n_t);
                        const R ct = RO::sqrt_(RO::f(1.0f) - eta * eta * (RO::f(1.0f) - ci * ci));
                        const R k = eta * ci - ct;
                        wi = r3<R>(diff2(nn.x, k, wo_r.x, eta), diff2(nn.y, k, wo_r.y, eta), diff2(nn.z, k, wo_r.z, eta));
                        ok = dot3(tof3(wi), g) < 0.0f;
                        betac *= RO::to_f(eta * eta);
                        nnew = n_t;
                    }
                }
            }
            if (!ok) return PUSH_NONE;
            coh_store<R>(pb, p, P, wi, opl);
            pb.coh4[p] = make_float4(nnew, betac, c4.z, __int_as_float(cv));
            const float3 pf = tof3(P), wf = tof3(wi);
            pb.ray_o[p] = make_float4(pf.x, pf.y, pf.z, 1e30f);
            pb.ray_d[p] = make_float4(wf.x, wf.y, wf.z, __int_as_float(tri));
            return PUSH_A;
        } else {
            // all of the path's state is loaded together, before anything depends on a part of it
            const bool first = e & Q_FIRST, ray = !(e & Q_FINALIZE);
            float4 s4 = make_float4(0.0f, 1.0f, 0.0f, 0.0f), h = make_float4(0.0f, 0.0f, 0.0f, __int_as_float(-1));
            float4 o4 = h, d4 = h;
            int occl = 0;
            const float2 s2 = pb.inc2[p];
            if (!first) {
                s4 = pb.inc[p];
                occl = pb.occl[p];
            }
            if (ray) {
                h = pb.hit[p];
                o4 = pb.ray_o[p];
                d4 = pb.ray_d[p];
            }
            const uint2 wgt = pb.cs3[p];
            IncState st;
            st.L = s4.x;
            st.beta = s4.y;
            st.ppdf = s4.z;
            st.tprev = s4.w;
            st.nee = s2.x;
            st.vfl = __float_as_int(s2.y);
            // the NEE of the previous vertex lands first, as in the sequential estimator
            if (st.nee > 0.0f && !occl) st.L += st.nee;
            st.nee = 0.0f;
            const int tri = __float_as_int(h.w);
            int push = PUSH_NONE;
            if (tri >= 0) {
                const PathId id = path_id(jt, wd, p);
                const DevScene &sc = id.J->sc;
                if (!HPT_IN(tri, sc.n_tris)) {
                    status |= ST_BOUNDS;
                    return PUSH_NONE;
                }
                st.vfl = (st.vfl & ~VF_V) | ((st.vfl & VF_V) + 1);
                st.tprev = h.x;
                const Surf S = make_surf(sc, tri, xyz(o4) + xyz(d4) * h.x, h.y, h.z);
                push = vertex(id, st, S, -xyz(d4), pb, p);
            }
            if (push == PUSH_NONE) {
                if (STATS) cnt.samples++;
                pb.amp[p] = (st.vfl & VF_BAKE) ? st.L
                            : (st.vfl & VF_HASP) ? __uint_as_float(wgt.x) * sqrtf(__uint_as_float(wgt.y) * st.L) : 0.0f;
            } else {
                pb.inc[p] = make_float4(st.L, st.beta, st.ppdf, st.tprev);
                pb.inc2[p] = make_float2(st.nee, __int_as_float(st.vfl));
            }
            return push;
        }
    };
    // whole warps take 32 consecutive entries at a time, the next ones' queue entries loaded ahead
    const int stride = gridDim.x * SHADE_BLOCK, lane = threadIdx.x & 31;
    int base = blockIdx.x * SHADE_BLOCK + (threadIdx.x & ~31);
    const int limit = HPT_CHECKED ? min(total, pb.capacity) : total;
    if (limit < total) status |= ST_BOUNDS;
    int next = base + lane < limit ? queue[base + lane] : Q_FINALIZE;
    if constexpr (COH && std::is_same<R, double>::value) {
        // In double precision the kernel is bound by the FP64 pipe (84 % busy with 20 of 32 lanes: misses,
        // image points and delta vertices side by side), so a warp gathers its entries by what they hit and
        // shades 32 of a kind: 1920 x 270 band 22.9 -> 20.7 ms and 18.9 -> 16.0 ms (two poses).  In
        // double-float it is bound by the state's loads, and the second look at the hit costs more than the
        // lanes give (1080p frame +0.7 %, 185k triangles +2 to +3 %).
        __shared__ int s_sorted[SHADE_BLOCK / 32][2][64];       // image points, delta vertices
        int (*const sorted)[64] = s_sorted[threadIdx.x >> 5];
        int held0 = 0, held1 = 0;
        for (;;) {
            while (base < limit && held0 < 32 && held1 < 32) {
                const int e = next, ni = base + stride + lane;
                next = ni < limit ? queue[ni] : Q_FINALIZE;
                int kind = -1;
                if (base + lane < limit && !(e & Q_FINALIZE)) {
                    if (!HPT_IN(e, wd.n_paths)) {
                        status |= ST_BOUNDS;
                    } else {
                        const int tri = __float_as_int(pb.hit[e].w);
                        if (tri >= 0) {
                            const DevScene &sc = jt->jobs[wd.seg[seg_of_path(wd, e)].job].sc;
                            if (!HPT_IN(tri, sc.n_tris)) {
                                status |= ST_BOUNDS;
                            } else {
                                const int m = sc.mats[__ldg(sc.tri_attr + tri).w].kind;
                                kind = m == 2 || m == 3;
                            }
                        }
                    }
                }
                const unsigned below = (1u << lane) - 1u;
                const unsigned m0 = __ballot_sync(0xFFFFFFFFu, kind == 0), m1 = __ballot_sync(0xFFFFFFFFu, kind == 1);
                if (kind >= 0) sorted[kind][kind ? held1 + __popc(m1 & below) : held0 + __popc(m0 & below)] = e;
                held0 += __popc(m0);
                held1 += __popc(m1);
                base += stride;
            }
            __syncwarp();
            const int k = held1 >= 32 || held0 == 0, held = k ? held1 : held0, n = min(held, 32);
            if (n == 0) break;
            const int v = sorted[k][lane], rest = sorted[k][32 + lane];
            __syncwarp();
            sorted[k][lane] = rest;
            (k ? held1 : held0) = held - n;
            const int push = lane < n ? entry(v, v) : PUSH_NONE;
            __syncwarp();
            enqueue2(push & PUSH_A, v, qa, ca, push & PUSH_B, v | Q_FIRST, qb, cb);
        }
    } else
    for (; base < limit; base += stride) {
        const int e = next, p = e & Q_PATH;
        const int ni = base + stride + lane;
        next = ni < limit ? queue[ni] : Q_FINALIZE;
        int push = PUSH_NONE;
        if (base + lane < limit && !(COH && (e & Q_FINALIZE))) push = entry(e, p);
        __syncwarp();
        enqueue2(push & (PUSH_A | PUSH_A_FINAL), push & PUSH_A_FINAL ? p | Q_FINALIZE : p, qa, ca, push & PUSH_B,
                 COH ? p | Q_FIRST : p, qb, cb);
    }
    if (STATS) flush_counters(cnt, scr);
    if (HPT_CHECKED && status) atomicOr(&scr->status, status);
}

// ------------------------------------------------------------------------------- s6 - s9
template <class R, bool WIDE>
__device__ __noinline__ float2 point_field(const DevJob *Jp, int lam, int px, int py, int *stk, int &status)
{
    using RO = RealOps<R>;
    const DevJob &J = *Jp;
    const DevScene &sc = J.sc;
    float2 acc = make_float2(0.0f, 0.0f);
    const R x = RO::mulf(RO::rc(J.pitch), (float)px + 0.5f - 0.5f * (float)J.W);
    const R y = RO::mulf(RO::rc(J.pitch), (float)py + 0.5f - 0.5f * (float)J.H);
    for (int e = 0; e < sc.n_points; ++e) {
        const double *pe = sc.points + 4 * e;
        const R3<R> pw = r3<R>(RO::fromd(pe[0]), RO::fromd(pe[1]), RO::fromd(pe[2]));
        R3<R> q, O;
        if (J.t_identity) {
            q = r3<R>(pw.x - x, pw.y - y, pw.z);
            O = r3<R>(x, y, RO::f(0.0f));
        } else {
            const R3<R> rw0 = r3<R>(RO::rc(J.R[0]), RO::rc(J.R[1]), RO::rc(J.R[2]));
            const R3<R> rw1 = r3<R>(RO::rc(J.R[3]), RO::rc(J.R[4]), RO::rc(J.R[5]));
            const R3<R> rw2 = r3<R>(RO::rc(J.R[6]), RO::rc(J.R[7]), RO::rc(J.R[8]));
            q = r3<R>(rdot(rw0, pw) + RO::rc(J.t[0]) - x, rdot(rw1, pw) + RO::rc(J.t[1]) - y,
                      rdot(rw2, pw) + RO::rc(J.t[2]));
            const R3<R> qq = r3<R>(x - RO::rc(J.t[0]), y - RO::rc(J.t[1]), -RO::rc(J.t[2]));
            const R3<R> c0 = r3<R>(RO::rc(J.R[0]), RO::rc(J.R[3]), RO::rc(J.R[6]));
            const R3<R> c1 = r3<R>(RO::rc(J.R[1]), RO::rc(J.R[4]), RO::rc(J.R[7]));
            const R3<R> c2 = r3<R>(RO::rc(J.R[2]), RO::rc(J.R[5]), RO::rc(J.R[8]));
            O = r3<R>(rdot(c0, qq), rdot(c1, qq), rdot(c2, qq));
        }
        const R r = RO::sqrt_(rdot(q, q));
        const float rf = RO::to_f(r);
        const float ct = RO::to_f(q.z) / rf;
        if (ct < J.cos_max[lam]) continue;
        const float3 Of = tof3(O);
        const float3 dw = tof3(pw - O);
        const float dist = sqrtf(dot3(dw, dw));
        Counters dummy;
        Traversal<false, false, ACCUM_BLOCK, WIDE> tr;
        // the segment from the pixel to just before the point, walked from its end that is nearer the scene
        float3 start = Of, dir = dw * (1.0f / dist);
        const float3 pf = tof3(pw);
        if (J.far && fmaxf(fmaxf(fabsf(pf.x), fabsf(pf.y)), fabsf(pf.z)) < fmaxf(fmaxf(fabsf(Of.x), fabsf(Of.y)), fabsf(Of.z))) {
            start = pf - dir * (SHADOW_SHRINK * dist);
            dir = -dir;
        }
        tr.start(sc, start, dir, dist * (1.0f - SHADOW_SHRINK), -1, true, false, stk);
        while (!tr.done()) tr.step(sc, false, stk, TSTACK, status, dummy);
        if (tr.h.tri >= 0)
            continue;
        const float turns = RO::frac_f(r * RO::rc(J.inv_lambda[lam]));
        float sn, cs;
        sincospif(2.0f * turns, &sn, &cs);
        const float a = (float)pe[3] * (J.obliquity ? ct : 1.0f) / rf;
        acc.x += a * cs;
        acc.y += a * sn;
    }
    return acc;
}

template <class R, bool WIDE>
__global__ void __launch_bounds__(ACCUM_BLOCK, HPT_ACCUM_MINB) k_accum(const JobTable *__restrict__ jt, const WaveDesc wd, PathBufs pb,
                                                       SlotScratch *__restrict__ scr)
{
    __shared__ int s_stack[TSTACK * ACCUM_BLOCK];
    const int i = blockIdx.x * ACCUM_BLOCK + threadIdx.x;
    if (i >= wd.n_items) return;
    int k = 0, first = 0;
    while (k + 1 < wd.n_seg && first + wd.seg[k].item_count <= i) {
        first += wd.seg[k].item_count;
        ++k;
    }
    const WaveSeg &g = wd.seg[k];
    const int il = i - first;
    PathId id;
    decode_item(jt->jobs + g.job, g.item_begin + il, id);
    if (!id.valid) return;
    const DevJob &J = *id.J;
    if (J.kind == 1) {
        // cache bake: E = pi / N sum of the arriving radiance, Kahan-compensated in sample order
        float a = 0.0f, c = 0.0f;
        for (int s = 0; s < g.spp; ++s) {
            const float y = pb.amp[g.path_offset + s * g.item_count + il] - c, t = a + y;
            c = (t - a) - y;
            a = t;
        }
        J.bake_out[(size_t)id.pix * 3 + id.lam] = 3.14159265f * (a - c) / (float)g.spp;
        return;
    }
    const int K = J.K, off = J.hologram_offset, spp = g.spp;
    float ar[KMAX], ai[KMAX], cr[KMAX], ci[KMAX];
#pragma unroll
    for (int j = 0; j < KMAX; ++j) ar[j] = ai[j] = cr[j] = ci[j] = 0.0f;
    // the records of two samples are loaded together, while the two before them are added: a thread otherwise
    // waits for memory once a sample
    struct Sample {
        float amp, ft;
        unsigned c0, c1, c2;
    };
    auto load = [&](int s) {
        Sample v = {0.0f, 0.0f, 0u, 0u, 0u};
        const int p = g.path_offset + s * g.item_count + il;
        if (s >= spp) return v;
        if (!HPT_IN(p, wd.n_paths)) {
            atomicOr(&scr->status, ST_BOUNDS);
            return v;
        }
        v.amp = pb.amp[p];
        v.ft = pb.fturn[p];
        v.c0 = (unsigned)pb.cx[p];
        v.c1 = (unsigned)pb.cy[p];
        v.c2 = (unsigned)pb.cz[p];
        return v;
    };
    auto add = [&](const Sample &v) {
        if (v.amp == 0.0f) return;
        const float amp = v.amp, ft = v.ft;
        const unsigned c0 = v.c0, c1 = v.c1, c2 = v.c2;
        uint4 ph = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int j = 0; j < KMAX; ++j) {
            if (j < K) {
                const int m = off + j;
                float u = 0.0f;
                if (J.phase_mode == 0) {
                    // s8: facet phase of hologram m, one Philox draw per four holograms
                    if (j == 0 || (m & 3) == 0)
                        ph = philox(make_uint4(c0, c1, c2, ((unsigned)id.lam << 16) | ((unsigned)m >> 2)), J.pseed_lo,
                                    J.pseed_hi);
                    const unsigned w = (m & 3) == 0 ? ph.x : ((m & 3) == 1 ? ph.y : ((m & 3) == 2 ? ph.z : ph.w));
                    u = u24(w);
                } else if (J.phase_mode == 2) {
                    // Eq. 4: phi_m sampled from the hologram's GRF map at the cell of Q
                    u = __ldg(J.grf + ((size_t)j * J.grf_ny + c1) * J.grf_nx + c0) * 0.159154943f;
                }
                float sn, cs;
                sincospif(2.0f * (ft + u), &sn, &cs);
                // s9: (1/(i lambda)) is folded into the amplitude: multiply the phasor by -i
                const float xr = amp * sn, xi = -amp * cs;
                const float yr = xr - cr[j], tr = ar[j] + yr;
                cr[j] = (tr - ar[j]) - yr;
                ar[j] = tr;
                const float yi = xi - ci[j], ti = ai[j] + yi;
                ci[j] = (ti - ai[j]) - yi;
                ai[j] = ti;
            }
        }
    };
    Sample v0 = load(0), v1 = load(1);
    for (int s = 2; s < spp + 2; s += 2) {
        const Sample n0 = load(s), n1 = load(s + 1);
        add(v0);
        add(v1);
        v0 = n0;
        v1 = n1;
    }
    float2 pf = make_float2(0.0f, 0.0f);
    if (J.sc.n_points > 0) {
        int status = 0;
        pf = point_field<R, WIDE>(id.J, id.lam, id.px, id.py, s_stack + threadIdx.x, status);
        if (status) atomicOr(&scr->status, (unsigned)status);
    }
    const float inv_n = 1.0f / (float)spp;
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
        if (j < K) {
            const size_t o = ((size_t)(id.lam * K + j) * J.H + id.py) * J.W + id.px;
            J.out[o] = make_float2((ar[j] - cr[j]) * inv_n + pf.x, (ai[j] - ci[j]) * inv_n + pf.y);
        }
    }
}

}  // namespace hpt
