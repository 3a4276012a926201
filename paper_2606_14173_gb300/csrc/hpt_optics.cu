// Wave optics around the tracer: the angular spectrum method of the two-stage scheme
// (hpt_asm_propagate) and the phase-only encoding (hpt_phase_encode).
//
// Both rest on a 2-D FFT convolution of power-of-two sizes made of packed half-length transforms
// (hpt_fft2.cuh): a row pass, a column pass and a row pass back.  The zero padding is never stored
// nor transformed; the transfer function is multiplied between the column pass's two transforms in
// registers; the encoding's phasors, residual, dot products and gradient step happen in the row
// passes' loads and stores.  The data are complex64; the twiddle factors are rounded from double-precision values.
// The transfer function's phase 2 pi z sqrt(1/lambda^2 - f^2), ~1e5 turns, is formed in
// double-float arithmetic before its fraction is taken.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <type_traits>
#include <vector>

#include <cuda_runtime.h>

#include "hpt.h"
#include "hpt_device.cuh"
#include "hpt_fft2.cuh"
#include "hpt_once.h"
#include "hpt_scratch.h"

namespace hpt {
int internal_ctx_device(const hpt_ctx *);
hpt_status internal_fail(hpt_status st, const char *msg);
hpt_status internal_check(hpt_ctx *ctx);
void internal_optics(const hpt_ctx *ctx, const float2 **tab, cudaMemPool_t *pool);
}  // namespace hpt

using namespace hpt;

namespace {

constexpr int FFT_MAX_LOG = FFT2_MAX_LM + 1;   // 8192 points
// Fields whose spectra go through the passes together: as many as keep the spectra within
// this many bytes.  Larger groups make longer launches, of which the last wave of blocks is a smaller
// part, and that is worth more than finding a pass's results in L2: 24 1080p fields (35 MB a
// spectrum) took 3.30 / 3.14 / 2.56 / 2.40 / 2.42 ms in groups of 40 / 96 / 150 / 300 / 600 MB.
constexpr size_t GROUP_BYTES = (size_t)300 << 20;

// ---- launch shapes --------------------------------------------------------------------------
// A block holds C transforms of T threads, 256 threads in all (512 in the row passes of the longest; 512-point halves and shorter fill
// warps with several transforms).  128 registers a thread: 64 of data, the rest twiddles and
// addresses in flight.
#ifndef HPT_OPT_REGS
#define HPT_OPT_REGS 128
#endif
__host__ __device__ constexpr int blk_c(int lm) { return fft2_threads(lm) >= 256 ? 1 : 256 / fft2_threads(lm); }
__host__ __device__ constexpr int blk_threads(int lm) { return blk_c(lm) * fft2_threads(lm); }
__host__ __device__ constexpr int blk_smem(int lm) { return blk_c(lm) * fft2_smem_elems(lm) * 16; }
#define OPT_BOUNDS(L) __launch_bounds__(blk_threads(L), 65536 / (HPT_OPT_REGS * blk_threads(L)))
// The row passes take two rows a block also where a row has 256 threads of its own: a 32-byte sector of
// the transposed spectrum holds two rows, and with one row a block each sector was written and read
// in halves by different SMs (three 3840 x 2160 fields: 1.70 ms with one row, 1.55 ms with two).  Four
// rows of 128 threads are slower than two (24 1080p fields: 2.54 against 2.25 ms): the barriers of a
// block of 512 threads then wait for more.
__host__ __device__ constexpr int row_c(int lm) { return fft2_threads(lm) == 256 ? 2 : blk_c(lm); }
__host__ __device__ constexpr int row_threads(int lm) { return row_c(lm) * fft2_threads(lm); }
__host__ __device__ constexpr int row_smem(int lm) { return row_c(lm) * fft2_smem_elems(lm) * 16; }
#define ROW_BOUNDS(L) __launch_bounds__(row_threads(L), 65536 / (HPT_OPT_REGS * row_threads(L)))

// The transform (c) and the thread within it (t) of this thread.  FAST: neighbouring threads belong
// to different transforms (rows next to each other share 32-byte sectors of the transposed
// spectrum); only where a transform spans whole warps, else a transform's threads are neighbours.
template <int LM, bool FAST>
struct Place {
    static constexpr int T = fft2_threads(LM), C = FAST ? row_c(LM) : blk_c(LM);
    static constexpr bool CF = FAST && T >= 32 && C > 1;
    static __device__ __forceinline__ int c() { return CF ? threadIdx.x % C : threadIdx.x / T; }
    static __device__ __forceinline__ int t() { return CF ? threadIdx.x / C : threadIdx.x % T; }
    // a barrier of the transform's threads (at least)
    static __device__ __forceinline__ void bar()
    {
        if constexpr (T < 32) __syncwarp();
        else if constexpr (CF || C == 1) __syncthreads();
        else asm volatile("bar.sync %0, %1;" ::"r"(threadIdx.x / T + 1), "n"(T) : "memory");
    }
};

// exp(-2 pi i n / 2M), n < M, from the table's place of the length.  A thread of a 16-point split has
// n = t + e M / 16: one root loaded, the others its products with exp(-2 pi i e / 32).  The passes are
// bound by L1, not by issue: 24 1080p fields 2.38 -> 2.25 ms against 16 loads, the results' error against
// 64 bits 2.45e-7 (2.2e-7 with loads, 2.9e-7 with the scalar transforms of before).
template <int LM> struct RootOf {
    float2 b;
    const float2 *w;
    __device__ __forceinline__ RootOf(const float2 *tab, int place, int t) : w(tab + place)
    {
        if (LM >= 4) b = __ldg(w + t);
    }
    __device__ __forceinline__ float2 at(int n, int e) const
    {
        if (LM >= 4) {
            constexpr float C[16] = {1.0f, 0.980785251f, 0.923879504f, 0.831469595f, 0.707106769f, 0.555570245f,
                                     0.382683426f, 0.195090324f, 0.0f, -0.195090324f, -0.382683426f, -0.555570245f,
                                     -0.707106769f, -0.831469595f, -0.923879504f, -0.980785251f};
            constexpr float S[16] = {0.0f, 0.195090324f, 0.382683426f, 0.555570245f, 0.707106769f, 0.831469595f,
                                     0.923879504f, 0.980785251f, 1.0f, 0.980785251f, 0.923879504f, 0.831469595f,
                                     0.707106769f, 0.555570245f, 0.382683426f, 0.195090324f};
            if (e == 0) return b;
            const float c = C[e], s = S[e];
            return make_float2(b.x * c + b.y * s, b.y * c - b.x * s);
        }
        return __ldg(w + n);
    }
};

// Programmatic dependent launch: the kernels of a chain let the next one's blocks become resident while
// their own last blocks still run.  Each waits for the end of the one before it, so that its own end
// implies the ends of all before it; until then it touches nothing that the chain writes (what the
// chain writes is read by plain loads, not as read-only data).  An encoding at 1920 x 1080, 7 launches
// an iteration: 2.80 -> 2.62 ms; three small fields 40.2 -> 38.8 us, three 3840 x 2160 fields 1.50 -> 1.48 ms.
// k_transfer, the first of every chain, is launched as usual and lets nothing in early: with the first
// row pass beside it, which only stores after it, the small fields take 43 us.
__device__ __forceinline__ void chain_next() { asm volatile("griddepcontrol.launch_dependents;"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// sums of N values over a block of up to 512 threads, in a fixed order, returned to the first warp
template <int N>
__device__ __forceinline__ void block_sum(double *v)
{
    __shared__ double sh[N][16];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < N; ++k) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int k = 0; k < N; ++k) sh[k][threadIdx.x >> 5] = v[k];
    __syncthreads();
    if (threadIdx.x < 32)
#pragma unroll
        for (int k = 0; k < N; ++k) {
            v[k] = (threadIdx.x & 15) < (blockDim.x >> 5) ? sh[k][threadIdx.x & 15] : 0.0;
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xFFFFFFFFu, v[k], o);
        }
}

// ---- the padded propagation -----------------------------------------------------------------
// What the forward row pass loads and what the backward one stores: the user's fields, or the
// encoding's steps (A the propagated field, T the target, s = <A, T> / <A, A>).
enum : int { ROW_FIELD = 0, ROW_PHASE = 1, ROW_RESIDUAL = 2, ROW_DOTS = 1, ROW_STEP = 2 };
struct RowIn {
    int mode;
    const float2 *field;     // ROW_FIELD: the field; ROW_RESIDUAL: A
    const float2 *target;    // ROW_RESIDUAL: T
    const float *phi;        // ROW_PHASE: the phase of a unit-amplitude field
    const double *sc;        // ROW_RESIDUAL: s
    double *part;            // ROW_RESIDUAL: a sum of |s A - T|^2 per block
};
struct RowOut {
    int mode;
    float2 *field;           // ROW_FIELD, ROW_DOTS: where the field goes
    const float2 *target;    // ROW_DOTS: T
    float *phi;              // ROW_STEP: the phase to step
    float lr;
    double *part;            // ROW_DOTS: sums of <A, T> (re, im) and <A, A> per block
};

// Pass 1: forward FFT along x of 'rows' rows of W points (H rows to a field), zero-extended to
// 2 M = 2^(LM+1): even frequencies in lane 0, odd in lane 1, stored as column pairs
// S[field][k][y] = (X[2k], X[2k+1]) with Hs (H rounded up to even) rows to a pair, so that the column
// pass reads each pair as one contiguous run.
// Bound by L1 (63 % busy): a store of 32 threads goes to 16 lines (a 32-byte sector each for two rows).
// 15.5 us a 1920 x 1080 field (13 us before, with row-major spectra, which the column pass then read 16 bytes
// at a time).
template <int LM>
__global__ void ROW_BOUNDS(LM) k_rows_in(const RowIn in, float4 *__restrict__ S, int rows, int W, int H, int Hs,
                                         const float2 *__restrict__ tab)
{
    using F = Fft2<LM, false>;
    using P = Place<LM, true>;
    extern __shared__ ulonglong2 sm[];
    const int c = P::c(), t = P::t();
    ulonglong2 *buf = sm + c * F::SMEM;
    const int row = blockIdx.x * P::C + c;
    const bool ok = row < rows;
    const int f = ok ? row / H : 0, y = ok ? row - f * H : 0;
    chain_next();
    chain_wait();
    const size_t base = (size_t)(ok ? row : 0) * W;
    c2 v[F::N];
    const Roots K = Roots::make();
    float2 x[F::N];
#pragma unroll
    for (int e = 0; e < F::N; ++e) x[e] = make_float2(0.0f, 0.0f);
    if (in.mode == ROW_FIELD) {
#pragma unroll
        for (int e = 0; e < F::N; ++e) {
            const int n = F::template in_index<0>(t, e);
            if (ok && n < W) x[e] = __ldg(in.field + base + n);
        }
    } else if (in.mode == ROW_PHASE) {
#pragma unroll
        for (int e = 0; e < F::N; ++e) {
            const int n = F::template in_index<0>(t, e);
            if (ok && n < W) sincosf(in.phi[base + n], &x[e].y, &x[e].x);
        }
    } else {
        // V = conj(s) (s A - T), with the loss |s A - T|^2 (at most 16 terms a thread in float, the
        // block's threads in double)
        const float sr = (float)in.sc[0], si = (float)in.sc[1];
        float l = 0.0f;
#pragma unroll
        for (int e = 0; e < F::N; ++e) {
            const int n = F::template in_index<0>(t, e);
            if (ok && n < W) {
                const float2 a = in.field[base + n], g = __ldg(in.target + base + n);
                const float rr = sr * a.x - si * a.y - g.x, ri = sr * a.y + si * a.x - g.y;
                l += rr * rr + ri * ri;
                x[e] = make_float2(sr * rr + si * ri, sr * ri - si * rr);
            }
        }
        double s = (double)l;
        block_sum<1>(&s);
        if (threadIdx.x == 0) in.part[blockIdx.x] = s;
    }
    const RootOf<LM> w(tab, F::ROOTS, t);
#pragma unroll
    for (int e = 0; e < F::N; ++e) {
        const int n = F::template in_index<0>(t, e);
        float2 o = make_float2(0.0f, 0.0f);
        if (n < W) {
            const float2 r = w.at(n, e);
            o = make_float2(x[e].x * r.x - x[e].y * r.y, x[e].x * r.y + x[e].y * r.x);
        }
        v[e] = {pk(x[e].x, o.x), pk(x[e].y, o.y)};
    }
    F::template run<0, true>(v, t, buf, tab, K, P::bar);
    if (!ok) return;
    float4 *d = S + (size_t)f * F::M * Hs + y;
#pragma unroll
    for (int e = 0; e < F::N; ++e) {
        const int k = F::template out_index<F::NP - 1>(t, e);
        float4 q;
        upk(v[e].re, q.x, q.z);
        upk(v[e].im, q.y, q.w);
        d[(size_t)k * Hs] = q;
    }
}

// Pass 2, in place on the column pairs: each column's H values, zero-extended to 2 M = 2^(LM+1),
// transformed, multiplied by the transfer function (CONJ: its conjugate, the propagation over -z of
// its propagating part) and transformed back, of which the first H values are stored.  The circular
// convolution is the same wherever the window lies, so it starts at row 0.  Consecutive blocks take
// the same columns of the nf fields, whose transfer rows then come from L2; columns fx and Wp - fx
// have the same one.
// Bound by L1 (75 % busy: most of it the 8 accesses of 16 bytes to shared memory per point pair, the
// rest transfer function, twiddles and data; 49 % issue): 60 us a 1920 x 1080 field, 105 us with
// scalar 4096-point transforms, whose halves of zeros were transformed too.  85 registers a thread
// (three blocks an SM instead of two) spill: 84 us.
template <int LM>
__global__ void OPT_BOUNDS(LM) k_cols(float2 *S, int H, int Hs, int Wp, int nf, FieldPlace f0, int fields_per_lambda, bool conj,
                                      const float4 *Ht, const float2 *__restrict__ tab)
{
    using F = Fft2<LM, false>;
    using B = Fft2<LM, true>;
    using P = Place<LM, false>;
    extern __shared__ ulonglong2 sm[];
    const int c = P::c(), t = P::t();
    ulonglong2 *buf = sm + c * F::SMEM;
    const int grp = blockIdx.x / nf, f = blockIdx.x - grp * nf;
    const int fx0 = grp * P::C + c;
    const bool ok = fx0 < Wp;
    const int fx = ok ? fx0 : 0;
    float2 *col = S + ((size_t)f * (Wp / 2) + (fx >> 1)) * Hs * 2 + (fx & 1);
    const RootOf<LM> w(tab, F::ROOTS, t);
    chain_next();
    chain_wait();
    c2 v[F::N];
    const Roots K = Roots::make();
#pragma unroll
    for (int e = 0; e < F::N; ++e) {
        const int n = F::template in_index<0>(t, e);
        float2 x = make_float2(0.0f, 0.0f), o = make_float2(0.0f, 0.0f);
        if (n < H) {
            x = col[2 * (size_t)n];
            const float2 r = w.at(n, e);
            o = make_float2(x.x * r.x - x.y * r.y, x.x * r.y + x.y * r.x);
        }
        v[e] = {pk(x.x, o.x), pk(x.y, o.y)};
    }
    F::template run<0, true>(v, t, buf, tab, K, P::bar);
    {
        const int lam = lambda_of(f0, f, fields_per_lambda), hrow = min(fx, Wp - fx);
        const float4 *h = Ht + ((size_t)lam * (Wp / 2 + 1) + hrow) * F::M;
        if (conj) {
#pragma unroll
            for (int e = 0; e < F::N; ++e) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(h + F::template out_index<F::NP - 1>(t, e));
                v[e] = cmul2<true>(v[e], q.x, q.y);
            }
        } else {
#pragma unroll
            for (int e = 0; e < F::N; ++e) {
                const ulonglong2 q = *reinterpret_cast<const ulonglong2 *>(h + F::template out_index<F::NP - 1>(t, e));
                v[e] = cmul2<false>(v[e], q.x, q.y);
            }
        }
    }
    B::template run<0, (F::NP == 1)>(v, t, buf, tab, K, P::bar);
    if (!ok) return;
#pragma unroll
    for (int e = 0; e < F::N; ++e) {
        const int n = B::template out_index<B::NP - 1>(t, e);
        if (n < H) {
            float er, orr, ei, oi;
            upk(v[e].re, er, orr);
            upk(v[e].im, ei, oi);
            const float2 r = w.at(n, e);
            col[2 * (size_t)n] = make_float2(er + (r.x * orr + r.y * oi), ei + (r.x * oi - r.y * orr));
        }
    }
}

// Pass 3: inverse FFT along x of the rows, of which the first W points are stored.
template <int LM>
__global__ void ROW_BOUNDS(LM) k_rows_out(const float4 *S, const RowOut out, int rows, int W, int H, int Hs,
                                          const float2 *__restrict__ tab)
{
    using B = Fft2<LM, true>;
    using P = Place<LM, true>;
    extern __shared__ ulonglong2 sm[];
    const int c = P::c(), t = P::t();
    ulonglong2 *buf = sm + c * B::SMEM;
    const int row = blockIdx.x * P::C + c;
    const bool ok = row < rows;
    const int f = ok ? row / H : 0, y = ok ? row - f * H : 0;
    chain_next();
    chain_wait();
    const float4 *s = S + (size_t)f * B::M * Hs + y;
    c2 v[B::N];
    const Roots K = Roots::make();
#pragma unroll
    for (int e = 0; e < B::N; ++e) {
        const float4 q = s[(size_t)B::template in_index<0>(t, e) * Hs];
        v[e] = {pk(q.x, q.z), pk(q.y, q.w)};
    }
    B::template run<0, true>(v, t, buf, tab, K, P::bar);
    const RootOf<LM> w(tab, B::ROOTS, t);
    const size_t base = (size_t)(ok ? row : 0) * W;
    float re = 0.0f, im = 0.0f, aa = 0.0f;
#pragma unroll
    for (int e = 0; e < B::N; ++e) {
        const int n = B::template out_index<B::NP - 1>(t, e);
        if (ok && n < W) {
            float er, orr, ei, oi;
            upk(v[e].re, er, orr);
            upk(v[e].im, ei, oi);
            const float2 r = w.at(n, e);
            const float2 a = make_float2(er + (r.x * orr + r.y * oi), ei + (r.x * oi - r.y * orr));
            if (out.mode == ROW_STEP) {
                // phi <- phi - lr dL/dphi, dL/dphi = -2 Im(u conj(G)), u = exp(i phi)
                const float p = out.phi[base + n];
                float sn, cs;
                sincosf(p, &sn, &cs);
                out.phi[base + n] = p + 2.0f * out.lr * (sn * a.x - cs * a.y);
            } else {
                out.field[base + n] = a;
                if (out.mode == ROW_DOTS) {
                    const float2 g = __ldg(out.target + base + n);
                    re += a.x * g.x + a.y * g.y;
                    im += a.x * g.y - a.y * g.x;
                    aa += a.x * a.x + a.y * a.y;
                }
            }
        }
    }
    if (out.mode == ROW_DOTS) {
        double d[3] = {(double)re, (double)im, (double)aa};
        block_sum<3>(d);
        if (threadIdx.x == 0) {
            out.part[blockIdx.x] = d[0];
            out.part[gridDim.x + blockIdx.x] = d[1];
            out.part[2 * gridDim.x + blockIdx.x] = d[2];
        }
    }
}

// calls f(std::integral_constant<int, lm>) for lm in [0, FFT2_MAX_LM]
template <class F>
cudaError_t with_lm(int lm, F f)
{
    switch (lm) {
    case 0: return f(std::integral_constant<int, 0>{});
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    case 9: return f(std::integral_constant<int, 9>{});
    case 10: return f(std::integral_constant<int, 10>{});
    case 11: return f(std::integral_constant<int, 11>{});
    case 12: return f(std::integral_constant<int, 12>{});
    default: return cudaErrorInvalidValue;
    }
}

// exp(i 2 pi z sqrt(1/lambda^2 - fx^2 - fy^2)) times 'scale' on the padded Wp x 2M grid, for fx up to
// Wp / 2 (the value depends on fx^2 only): Ht[lambda][fx][i] = the even and odd frequencies 2i and
// 2i + 1 along y as the column pass's lanes hold them, (E.re, O.re, E.im, O.im).  The value depends on
// fy^2 only as well: E[M - i] = E[i] and O[M - 1 - i] = O[i], so a thread computes i <= M / 2 and
// stores it at i and, with its neighbour's O[i - 1], at M - i.
constexpr int TRANSFER_BLOCK = 256;
struct TransferLambdas {
    float2 inv_lambda2[3];
};
__global__ void __launch_bounds__(TRANSFER_BLOCK) k_transfer(float4 *Ht, int Wp, int M, float2 fx_unit, float2 fy_unit,
                                                             const TransferLambdas L, float2 zdist, float scale)
{
    // double-float arithmetic (~48-bit significands): the phase runs to ~1e5 turns and its
    // fraction must hold ~1e-7
    __shared__ float2 odd[TRANSFER_BLOCK];
    const int fxi = blockIdx.y, lam = blockIdx.z;              // fx = 0 .. Wp / 2
    const df fx = mul_f(mkdf(fx_unit.x, fx_unit.y), (float)fxi);
    const df base = mkdf(L.inv_lambda2[lam].x, L.inv_lambda2[lam].y) - fx * fx;
    const df fyu = mkdf(fy_unit.x, fy_unit.y), z = mkdf(zdist.x, zdist.y);
    auto value = [&](int fyi) {                                // fy = 0 .. M, or a mirror of it
        const df fy = mul_f(fyu, (float)(fyi <= M ? fyi : 2 * M - fyi));
        const df a = base - fy * fy;
        float2 v = make_float2(0.0f, 0.0f);
        if (a.hi > 0.0f) {
            // square root: the approximate reciprocal root's product, corrected to float accuracy, then
            // by the residual a - x^2 (one FMA and the tail; what is left is below 2^-46 of the root)
            const float q = rsqrtf(a.hi), h = 0.5f * q, x0 = __fmul_rn(a.hi, q);
            const float x = __fmaf_rn(h, __fmaf_rn(-x0, x0, a.hi), x0);
            const float r = __fadd_rn(__fmaf_rn(-x, x, a.hi), a.lo);
            const float f = RealOps<df>::frac_f(z * quick_two_sum(x, __fmul_rn(h, r)));
            float sn, cs;
            sincospif(2.0f * f, &sn, &cs);
            v = make_float2(cs * scale, sn * scale);
        }
        return v;
    };
    float4 *row = Ht + ((size_t)lam * (Wp / 2 + 1) + fxi) * M;
    // the block's first thread only computes the odd value its neighbour needs
    const int i = blockIdx.x * (TRANSFER_BLOCK - 1) + (int)threadIdx.x - 1;
    const bool in = i >= 0 && i <= M / 2 && i < M;
    const float2 o = in ? value(2 * i + 1) : make_float2(0.0f, 0.0f);
    odd[threadIdx.x] = o;
    __syncthreads();
    if (threadIdx.x == 0 || !in) return;
    const float2 e = value(2 * i), om = odd[threadIdx.x - 1];
    row[i] = make_float4(e.x, o.x, e.y, o.y);
    if (i > 0 && M - i > M / 2) row[M - i] = make_float4(e.x, om.x, e.y, om.y);
}

// a double as a double-float pair (head, tail)
float2 to_df(double x)
{
    const float h = (float)x;
    return make_float2(h, (float)(x - (double)h));
}

int ilog2(int n)
{
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

bool pow2_in_range(int n) { return n >= 2 && n <= (1 << FFT_MAX_LOG) && (n & (n - 1)) == 0; }

template <class K> cudaError_t allow_smem(K kernel, int bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// a launch that may overlap the end of the one before it (chain_next)
template <class... P, class... A>
cudaError_t launch_next(void (*kernel)(P...), unsigned grid, int threads, int smem, cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute at;
    memset(&at, 0, sizeof at);
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof cfg);
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// scratch of one call from the context's pool, released on the stream
struct Scratch {
    char *p = nullptr;
    size_t used = 0;
    cudaStream_t s;
    explicit Scratch(cudaStream_t s_) : s(s_) {}
    cudaError_t get(size_t bytes, cudaMemPool_t pool) { return pool_alloc((void **)&p, bytes, pool, s); }
    template <class T> T *take(size_t n)
    {
        T *r = (T *)(p + used);
        used += (n * sizeof(T) + 255) & ~(size_t)255;
        return r;
    }
    cudaError_t release()
    {
        cudaError_t e = p ? cudaFreeAsync(p, s) : cudaSuccess;
        p = nullptr;
        return e;
    }
};

}  // namespace

namespace hpt {
// The twiddle tables live in the module, so that a captured call stays valid for as long as the
// process, whatever becomes of its context.
__device__ float2 g_twiddles[FFT2_TABLE_ENTRIES];

// For hpt_create: the twiddle tables (host doubles rounded to float) and the kernels' shared-memory
// limits, once per device, and the context's pool for the calls' scratch.  The pool keeps up to
// OPT_POOL_KEEP bytes between calls, so that a call after a synchronisation does not map its scratch
// anew (the device's default pool gives everything back at each synchronisation: 1.6 ms of a 4.9 ms
// call on 24 1080p fields, 3.9 of 6.6 on three of 3840 x 2160); what it keeps is given back when an
// allocation of the library would otherwise fail, and by hpt_destroy.
constexpr uint64_t OPT_POOL_KEEP = 1200ull << 20;
cudaError_t optics_setup(int device, const float2 **tab, cudaMemPool_t *pool)
{
    static OncePerDevice once;
    cudaError_t e = cudaGetSymbolAddress((void **)tab, g_twiddles);
    if (e != cudaSuccess) return e;
    e = once(device, [] {
        std::vector<float2> h((size_t)FFT2_TABLE_ENTRIES);
        for (int lm = 0; lm <= FFT2_MAX_LM; ++lm) {
            const int M = 1 << lm;
            float2 *r = &h[fft2_base(lm)];
            for (int n = 0; n < M; ++n) {
                const double a = -M_PI * n / M;
                r[n] = make_float2((float)cos(a), (float)sin(a));
            }
            for (int inv = 0; inv < 2; ++inv)
                for (int p = 1; p < fft2_npass(lm); ++p) {
                    const int R = fft2_radix(lm, inv, p), NS = fft2_ns(lm, inv, p);
                    float2 *q = &h[fft2_pass_off(lm, inv, p)];
                    for (int j = 1; j < R; ++j)
                        for (int k = 0; k < NS; ++k) {
                            const double a = -2.0 * M_PI * ((long long)j * k) / ((double)NS * R);
                            q[(j - 1) * NS + k] = make_float2((float)cos(a), (float)sin(a));
                        }
                }
        }
        cudaError_t e = cudaMemcpyToSymbol(g_twiddles, h.data(), h.size() * sizeof(float2));
        for (int lm = 0; lm <= FFT2_MAX_LM && e == cudaSuccess; ++lm)
            e = with_lm(lm, [&](auto L) {
                constexpr int l = decltype(L)::value;
                cudaError_t r = allow_smem(k_rows_in<l>, row_smem(l));
                if (r == cudaSuccess) r = allow_smem(k_cols<l>, blk_smem(l));
                if (r == cudaSuccess) r = allow_smem(k_rows_out<l>, row_smem(l));
                return r;
            });
        return e;
    });
    if (e != cudaSuccess) return e;
    cudaMemPoolProps props;
    memset(&props, 0, sizeof props);
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    e = cudaMemPoolCreate(pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = OPT_POOL_KEEP;
    return cudaMemPoolSetAttribute(*pool, cudaMemPoolAttrReleaseThreshold, &keep);
}
}  // namespace hpt

#define OPT_TRY(x)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (x);                                                                      \
        if (e_ != cudaSuccess) {                                                                   \
            char m_[256];                                                                          \
            snprintf(m_, sizeof m_, "%s: %s", #x, cudaGetErrorString(e_));                         \
            return internal_fail(HPT_ERR_CUDA, m_);                                                \
        }                                                                                          \
    } while (0)

namespace {

// The padded angular-spectrum step of W x H fields.
struct AsmPlan {
    int W, H, Hs, Wp, Hp, lx, ly;   // 2^lx = Wp / 2, 2^ly = Hp / 2
    const float2 *tab;
    float4 *S, *Ht;                 // spectra of one group of fields, transfer rows of every wavelength
    size_t spectrum() const { return (size_t)(Wp / 2) * Hs; }               // float4 per field
    size_t transfer() const { return (size_t)(Wp / 2 + 1) * (Hp / 2); }     // float4 per wavelength
    int row_blocks(int rows) const { return (rows + row_c(lx) - 1) / row_c(lx); }
};

bool asm_sizes(int W, int H, AsmPlan &P)
{
    P.W = W;
    P.H = H;
    P.Hs = (H + 1) & ~1;
    P.Wp = P.Hp = 2;
    while (P.Wp < 2 * W) P.Wp <<= 1;
    while (P.Hp < 2 * H) P.Hp <<= 1;
    if (!pow2_in_range(P.Wp) || !pow2_in_range(P.Hp)) return false;
    P.lx = ilog2(P.Wp) - 1;
    P.ly = ilog2(P.Hp) - 1;
    return true;
}

cudaError_t asm_transfer(const AsmPlan &P, const double *lambdas, int nl, double pitch, double z, cudaStream_t s)
{
    TransferLambdas L;
    memset(&L, 0, sizeof L);
    for (int l = 0; l < nl; ++l) L.inv_lambda2[l] = to_df(1.0 / (lambdas[l] * lambdas[l]));
    const int M = P.Hp / 2, cover = std::min(M, M / 2 + 1);   // i = 0 .. M / 2 below M
    k_transfer<<<dim3((cover + TRANSFER_BLOCK - 2) / (TRANSFER_BLOCK - 1), P.Wp / 2 + 1, nl), TRANSFER_BLOCK, 0, s>>>(
        P.Ht, P.Wp, M, to_df(1.0 / (P.Wp * pitch)), to_df(1.0 / (P.Hp * pitch)), L, to_df(z),
        1.0f / (float)((size_t)P.Wp * P.Hp));
    return cudaGetLastError();
}

// nf fields (consecutive W x H fields), the first being field f0 of fields_per_lambda to a wavelength
cudaError_t asm_group(const AsmPlan &P, const RowIn &in, const RowOut &out, int nf, long long f0, int fields_per_lambda, bool conj,
                      cudaStream_t s)
{
    const int rows = nf * P.H, rb = P.row_blocks(rows);
    cudaError_t e = with_lm(P.lx, [&](auto L) {
        constexpr int l = decltype(L)::value;
        return launch_next(k_rows_in<l>, rb, row_threads(l), row_smem(l), s, in, P.S, rows, P.W, P.H, P.Hs, P.tab);
    });
    if (e != cudaSuccess) return e;
    e = with_lm(P.ly, [&](auto L) {
        constexpr int l = decltype(L)::value, C = blk_c(l);
        return launch_next(k_cols<l>, ((P.Wp + C - 1) / C) * nf, blk_threads(l), blk_smem(l), s, (float2 *)P.S, P.H, P.Hs, P.Wp,
                          nf, field_place(f0, fields_per_lambda), fields_per_lambda, conj, P.Ht, P.tab);
    });
    if (e != cudaSuccess) return e;
    return with_lm(P.lx, [&](auto L) {
        constexpr int l = decltype(L)::value;
        return launch_next(k_rows_out<l>, rb, row_threads(l), row_smem(l), s, P.S, out, rows, P.W, P.H, P.Hs, P.tab);
    });
}

// ---- phase-only encoding -----------------------------------------------------------------
constexpr int RED_THREADS = 256;

// s = <A, T> / <A, A> from the nb partial sums of the row pass (one block), and, for iterations after
// the first, the loss of the iteration before from its partial sums
__global__ void __launch_bounds__(RED_THREADS) k_scale(const double *part, int nb, double *sc, const double *lpart, double *loss)
{
    chain_next();
    chain_wait();
    double d[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nb; b += RED_THREADS) {
        if (part) {
            d[0] += part[b];
            d[1] += part[nb + b];
            d[2] += part[2 * nb + b];
        }
        if (loss) d[3] += lpart[b];
    }
    block_sum<4>(d);
    if (threadIdx.x == 0) {
        if (part) {
            sc[0] = d[2] > 0.0 ? d[0] / d[2] : 0.0;
            sc[1] = d[2] > 0.0 ? d[1] / d[2] : 0.0;
        }
        if (loss) *loss = d[3];
    }
}

}  // namespace

extern "C" hpt_status hpt_asm_propagate(hpt_ctx *ctx, const void *in_dev, void *out_dev, int32_t W, int32_t H,
                                        int32_t n_lambda, int32_t K, const double *lambdas, double pitch, double z,
                                        void *stream)
{
    hpt_status st = internal_check(ctx);
    if (st) return st;
    if (!in_dev || !out_dev || !lambdas) return internal_fail(HPT_ERR_INVALID_ARG, "in_dev, out_dev or lambdas is NULL");
    if (W < 1 || H < 1 || n_lambda < 1 || n_lambda > 3 || K < 1)
        return internal_fail(HPT_ERR_INVALID_ARG, "need W, H, K >= 1 and 1 <= n_lambda <= 3");
    AsmPlan P;
    if (W > 4096 || H > 4096 || !asm_sizes(W, H, P))
        return internal_fail(HPT_ERR_UNSUPPORTED, "padded size above 8192 x 8192 (W, H <= 4096)");
    if (!(pitch > 0.0) || !std::isfinite(pitch) || !std::isfinite(z))
        return internal_fail(HPT_ERR_INVALID_ARG, "pitch must be finite and > 0, z finite");
    for (int l = 0; l < n_lambda; ++l)
        if (!(lambdas[l] > 0.0) || !std::isfinite(lambdas[l]))
            return internal_fail(HPT_ERR_INVALID_ARG, "wavelengths must be finite and > 0");
    OPT_TRY(cudaSetDevice(internal_ctx_device(ctx)));
    cudaMemPool_t pool;
    internal_optics(ctx, &P.tab, &pool);
    cudaStream_t s = (cudaStream_t)stream;
    // the fields of all wavelengths go through in groups
    const long long total = (long long)n_lambda * K;
    int G = group_items(total, P.spectrum() * sizeof(float4), GROUP_BYTES);
    Scratch scr(s);
    OPT_TRY(get_group(G, [&](int g) {
        return scr.get(((size_t)g * P.spectrum() + (size_t)n_lambda * P.transfer()) * sizeof(float4) + 512, pool);
    }));
    P.S = scr.take<float4>((size_t)G * P.spectrum());
    P.Ht = scr.take<float4>((size_t)n_lambda * P.transfer());
    cudaError_t e = asm_transfer(P, lambdas, n_lambda, pitch, z, s);
    if (e == cudaSuccess)
        e = for_groups(total, G, [&](long long f, int nf) {
            const size_t fo = (size_t)f * W * H;
            RowIn in{};
            in.field = (const float2 *)in_dev + fo;
            RowOut out{};
            out.field = (float2 *)out_dev + fo;
            return asm_group(P, in, out, nf, f, K, false, s);
        });
    cudaError_t e2 = scr.release();
    OPT_TRY(e);
    OPT_TRY(e2);
    return HPT_OK;
}

extern "C" hpt_status hpt_phase_encode(hpt_ctx *ctx, const void *target_dev, float *phi_dev, int32_t W, int32_t H,
                                       double lambda, double pitch, double z, int32_t iters, float lr, double *losses,
                                       void *stream)
{
    hpt_status st = internal_check(ctx);
    if (st) return st;
    if (!target_dev || !phi_dev) return internal_fail(HPT_ERR_INVALID_ARG, "target_dev or phi_dev is NULL");
    if (W < 1 || H < 1 || iters < 0) return internal_fail(HPT_ERR_INVALID_ARG, "need W, H >= 1 and iters >= 0");
    if (!(pitch > 0.0) || !(lambda > 0.0) || !std::isfinite(pitch) || !std::isfinite(lambda) || !std::isfinite(z) ||
        !std::isfinite(lr))
        return internal_fail(HPT_ERR_INVALID_ARG, "bad pitch, lambda, z or lr");
    AsmPlan P;
    if (W > 4096 || H > 4096 || !asm_sizes(W, H, P))
        return internal_fail(HPT_ERR_UNSUPPORTED, "padded size above 8192 x 8192 (W, H <= 4096)");
    OPT_TRY(cudaSetDevice(internal_ctx_device(ctx)));
    cudaMemPool_t pool;
    internal_optics(ctx, &P.tab, &pool);
    cudaStream_t s = (cudaStream_t)stream;
    const size_t n = (size_t)W * H;
    const int nb = P.row_blocks(H);
    Scratch scr(s);
    OPT_TRY(scr.get((P.spectrum() + P.transfer()) * sizeof(float4) + n * sizeof(float2) +
                        (4 * (size_t)nb + 2 + (size_t)std::max(iters, 1)) * sizeof(double) + 8 * 256,
                    pool));
    P.S = scr.take<float4>(P.spectrum());
    P.Ht = scr.take<float4>(P.transfer());
    float2 *A = scr.take<float2>(n);
    double *part = scr.take<double>(3 * (size_t)nb), *lpart = scr.take<double>(nb), *sc = scr.take<double>(2);
    double *dloss = scr.take<double>(std::max(iters, 1));
    const float2 *T = (const float2 *)target_dev;
    cudaError_t e = asm_transfer(P, &lambda, 1, pitch, z, s);
    RowIn phase{}, residual{};
    phase.mode = ROW_PHASE;
    phase.phi = phi_dev;
    residual.mode = ROW_RESIDUAL;
    residual.field = A;
    residual.target = T;
    residual.sc = sc;
    residual.part = lpart;
    RowOut dots{}, step{};
    dots.mode = ROW_DOTS;
    dots.field = A;
    dots.target = T;
    dots.part = part;
    step.mode = ROW_STEP;
    step.phi = phi_dev;
    step.lr = lr;
    for (int it = 0; it < iters && e == cudaSuccess; ++it) {
        e = asm_group(P, phase, dots, 1, 0, 1, false, s);
        if (e != cudaSuccess) break;
        e = launch_next(k_scale, 1, RED_THREADS, 0, s, part, nb, sc, lpart, it > 0 ? dloss + it - 1 : nullptr);
        if (e != cudaSuccess) break;
        // the adjoint of the propagation over z is the one over -z: the conjugate transfer function
        e = asm_group(P, residual, step, 1, 0, 1, true, s);
    }
    if (e == cudaSuccess && iters > 0)
        e = launch_next(k_scale, 1, RED_THREADS, 0, s, (const double *)nullptr, nb, sc, lpart, dloss + iters - 1);
    if (e == cudaSuccess && losses && iters > 0)
        e = cudaMemcpyAsync(losses, dloss, sizeof(double) * iters, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && losses && iters > 0) e = cudaStreamSynchronize(s);
    cudaError_t e2 = scr.release();
    OPT_TRY(e);
    OPT_TRY(e2);
    return HPT_OK;
}
