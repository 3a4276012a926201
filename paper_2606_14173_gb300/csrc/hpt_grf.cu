// The band-limited Gaussian random field phase maps of Eq. 4 (hpt_grf_build).
//
// One 2-D FFT of power-of-two sizes: every row transformed in shared memory by
// one block (Stockham autosort: radix-16 passes in registers, the remainder radix first, the
// first pass reading global memory and the last writing it in natural order, the passes in
// between in place in one bank-padded shared buffer), then every column the same way, a few
// adjacent columns per block read and written in place in the row-major array (no transposes).
// The spectrum is generated as the row pass loads it and the phase taken as the column pass stores
// it.  The data are complex64; the twiddle factors are rounded from double-precision values.
//
// The maps stay on these scalar transforms, not the packed half-length ones of the propagation
// (hpt_fft2.cuh): those gave the same accuracy and 88 us a 4096 x 2048 map against 97 (90 now), 1 % of a
// frame that builds its maps, but another rounding, which the phase magnifies without bound where the field
// is near zero, so that maps of a seed would no longer be the same bits.
#include <algorithm>
#include <type_traits>
#include <cmath>
#include <cstdio>
#include <cstring>

#include <cuda_runtime.h>

#include "hpt.h"
#include "hpt_device.cuh"
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

constexpr int FFT_MAX_LOG = 13;          // 8192 points: 68 KB of shared memory
constexpr int FFT_THREADS = 512;
#ifndef HPT_FFT_REGS
#define HPT_FFT_REGS 64                  // registers per thread the row kernels are compiled for
#endif
constexpr unsigned GRF_TAG = 0x47524600u;
constexpr size_t GROUP_BYTES = (size_t)300 << 20;

__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// tw[k] = exp(-2 pi i k / n), k < n
__global__ void k_twiddles(float2 *tw, int n)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    double s, c;
    sincospi(-2.0 * (double)k / (double)n, &s, &c);
    tw[k] = make_float2((float)c, (float)s);
}

// exp(-2 pi i m / 16), m < 8: the constants of the in-register radix-16 DFT
__device__ __forceinline__ float2 w16(int m)
{
    const float c[8] = {1.0f, 0.923879533f, 0.707106781f, 0.382683432f, 0.0f, -0.382683432f, -0.707106781f, -0.923879533f};
    const float s[8] = {0.0f, 0.382683432f, 0.707106781f, 0.923879533f, 1.0f, 0.923879533f, 0.707106781f, 0.382683432f};
    return make_float2(c[m], -s[m]);
}

// R-point DFT of v in registers (R = 2, 4, 8, 16): bit-reversed order, then log2 R radix-2
// stages; SIGN = -1 forward, +1 inverse.  The butterflies whose twiddle is 1 or -+i take no
// multiplication.
template <int R, int SIGN>
__device__ __forceinline__ void dft_reg(float2 *v)
{
    constexpr int B = R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : 4;
    float2 t[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        int r = 0;
#pragma unroll
        for (int b = 0; b < B; ++b) r |= ((i >> b) & 1) << (B - 1 - b);
        t[r] = v[i];
    }
#pragma unroll
    for (int half = 1; half < R; half *= 2) {
#pragma unroll
        for (int g = 0; g < R; g += 2 * half) {
#pragma unroll
            for (int pos = 0; pos < half; ++pos) {
                const int m = pos * (8 / half);        // twiddle exp(SIGN 2 pi i m / 16)
                float2 b = t[g + pos + half];
                if (m == 4) {
                    b = SIGN > 0 ? make_float2(-b.y, b.x) : make_float2(b.y, -b.x);
                } else if (m != 0) {
                    float2 w = w16(m);
                    if (SIGN > 0) w.y = -w.y;
                    b = cmul(w, b);
                }
                const float2 a = t[g + pos];
                t[g + pos] = make_float2(a.x + b.x, a.y + b.y);
                t[g + pos + half] = make_float2(a.x - b.x, a.y - b.y);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = t[i];
}

// Shared-memory index of point i of a row: one float2 of padding after every 16, so that the
// stride-16 stores of the first pass and the strided loads after it fall in distinct banks.
__device__ __forceinline__ int spad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int fft_smem_bytes(int n) { return (n + n / 16 + 1) * (int)sizeof(float2); }
// threads of a row's block: n / 16 (each holds 16 points of a pass), at least one warp
__host__ __device__ constexpr int fft_threads(int n) { return n / 16 > 32 ? (n / 16 < FFT_THREADS ? n / 16 : FFT_THREADS) : 32; }
// resident blocks per SM the row kernels are compiled for: 'regs' registers per thread
__host__ __device__ constexpr int fft_minb(int n, int regs)
{
    return 65536 / (regs * fft_threads(n)) < 1 ? 1 : (65536 / (regs * fft_threads(n)) > 32 ? 32 : 65536 / (regs * fft_threads(n)));
}
// radix of pass p of a 2^logn-point transform (the remainder radix first, then 16s), the number
// of passes, and the span Ns of the sub-transforms pass p combines
__host__ __device__ constexpr int fft_radix(int logn, int p) { return (p == 0 && (logn & 3)) ? (1 << (logn & 3)) : 16; }
__host__ __device__ constexpr int fft_npass(int logn) { return (logn >> 2) + ((logn & 3) ? 1 : 0); }
__host__ __device__ constexpr int fft_ns(int logn, int p) { return p == 0 ? 1 : fft_ns(logn, p - 1) * fft_radix(logn, p - 1); }

// Pass P of the Stockham transform of N = 2^LOGN points (radix R, span NS): element j reads
// x[j + r N/R] (r < R) through 'ld', multiplies it by exp(SIGN 2 pi i r (j mod NS) / (NS R))
// (the N-point twiddle table), takes the R-point DFT and writes
// y[(j - j mod NS) R + j mod NS + r NS] through 'st'.  Thread t takes j = t + m T (T threads,
// m < J; t = tid, the thread's index within the transform); with 'inplace' every thread holds
// its values in registers across a barrier before it stores, so that x and y may be the same buffer.
template <int LOGN, int P, int SIGN, class LD, class ST>
__device__ __forceinline__ void stockham_pass(const float2 *__restrict__ tw, LD ld, ST st, bool inplace, int tid)
{
    constexpr int N = 1 << LOGN, R = fft_radix(LOGN, P), NS = fft_ns(LOGN, P), T = fft_threads(N);
    constexpr int Q = N / R, TWS = N / (NS * R), J = (Q + T - 1) / T;
    constexpr bool RAGGED = J * T > Q;
    float2 v[J][R];
#pragma unroll
    for (int m = 0; m < J; ++m) {
        // past the row (small N only) a thread repeats the last element's loads and stores nothing
        const int j = RAGGED ? min(tid + m * T, Q - 1) : tid + m * T;
        const int k = j & (NS - 1);
#pragma unroll
        for (int r = 0; r < R; ++r) v[m][r] = ld(j + r * Q);
        if (NS > 1) {
            // twiddles w^r, w = exp(SIGN 2 pi i k / (NS R)): w, w^2, w^3 formed from the loaded w,
            // w^(4c) loaded for c >= 1 and multiplied by them (at most three complex products
            // per twiddle, ~1e-7 relative)
            float2 w1 = __ldg(tw + k * TWS);
            if (SIGN > 0) w1.y = -w1.y;
            const float2 w2 = cmul(w1, w1), w3 = cmul(w2, w1);
#pragma unroll
            for (int r = 1; r < R; ++r) {
                float2 w;
                if (r % 4 == 0 || r < 4) {
                    w = r == 1 ? w1 : r == 2 ? w2 : r == 3 ? w3 : __ldg(tw + r * k * TWS);
                    if (r >= 4 && SIGN > 0) w.y = -w.y;
                } else {
                    float2 b = __ldg(tw + (r & ~3) * k * TWS);
                    if (SIGN > 0) b.y = -b.y;
                    w = cmul(b, (r & 3) == 1 ? w1 : (r & 3) == 2 ? w2 : w3);
                }
                v[m][r] = cmul(v[m][r], w);
            }
        }
        dft_reg<R, SIGN>(v[m]);
    }
    if (inplace) __syncthreads();
#pragma unroll
    for (int m = 0; m < J; ++m) {
        const int j = tid + m * T;
        if (!RAGGED || j < Q) {
            const int k = j & (NS - 1);
            const int o = (j - k) * R + k;
#pragma unroll
            for (int r = 0; r < R; ++r) st(o + r * NS, v[m][r]);
        }
    }
}

// FFT of one row of 2^LOGN points by fft_threads(2^LOGN) threads: the passes from P on, the
// first reading through 'gld', the last writing through 'gst', the ones in between in place in
// the shared buffer 'buf' (padded by spad).  IN_SMEM / OUT_SMEM say that gld / gst touch 'buf'
// themselves.  tid: the thread's index within the transform (threadIdx.x when a block takes one
// row).  Ends with a barrier of the whole block.
template <int LOGN, int SIGN, bool IN_SMEM, bool OUT_SMEM, int P = 0, class LD, class ST>
__device__ __forceinline__ void row_fft(const float2 *tw, float2 *buf, LD gld, ST gst, int tid = threadIdx.x)
{
    constexpr int NP = fft_npass(LOGN);
    constexpr bool first = P == 0, last = P == NP - 1;
    constexpr bool src_smem = first ? IN_SMEM : true, dst_smem = last ? OUT_SMEM : true;
    constexpr bool inplace = (src_smem && dst_smem) || NP == 1;
    auto sld = [&](int i) { return buf[spad(i)]; };
    auto sst = [&](int i, float2 v) { buf[spad(i)] = v; };
    if constexpr (first && last) stockham_pass<LOGN, P, SIGN>(tw, gld, gst, inplace, tid);
    else if constexpr (first) stockham_pass<LOGN, P, SIGN>(tw, gld, sst, inplace, tid);
    else if constexpr (last) stockham_pass<LOGN, P, SIGN>(tw, sld, gst, inplace, tid);
    else stockham_pass<LOGN, P, SIGN>(tw, sld, sst, inplace, tid);
    __syncthreads();
    if constexpr (P + 1 < NP) row_fft<LOGN, SIGN, IN_SMEM, OUT_SMEM, P + 1>(tw, buf, gld, gst, tid);
}

#define FFT_BOUNDS(L) __launch_bounds__(fft_threads(1 << (L)), fft_minb(1 << (L), HPT_FFT_REGS))

// GRF pass 1 (Eq. 4): for each spectrum row ky < ny, the unit-modulus random spectrum
// exp(i xi) inside the elliptic passband 4 (kx^2 ny^2 + ky^2 nx^2) <= nx^2 ny^2 (integers, FFT
// order) and 0 outside it, xi = 2 pi u24(Philox(ix, iy, m, 'GRF'; seed)), generated as the
// first pass loads it, and its unnormalised inverse FFT along x.
template <int LOGN>
__global__ void FFT_BOUNDS(LOGN) k_grf_rows(float2 *out, int ny, int lny, unsigned m0, unsigned seed_lo, unsigned seed_hi,
                                            const float2 *__restrict__ tw)
{
    extern __shared__ float2 sm[];
    constexpr int nx = 1 << LOGN;
    const long long NX = nx, NY = ny;
    {
        // one row per block, the rows of a group of maps one after the other
        const int iy = blockIdx.x & (ny - 1);
        const unsigned m = m0 + (blockIdx.x >> lny);
        // the largest |kx| of the row inside the passband, exactly: 4 kx^2 ny^2 <= rest
        const long long ky = iy < ny / 2 ? iy : iy - ny;
        const long long rest = NX * NX * NY * NY - 4 * ky * ky * NX * NX, unit = 4 * NY * NY;
        long long km = (long long)sqrt((double)rest / (double)unit);
        while (km > 0 && km * km * unit > rest) --km;
        while ((km + 1) * (km + 1) * unit <= rest) ++km;
        const int kmax = (int)km;
        float2 *d = out + ((size_t)blockIdx.x << LOGN);
        row_fft<LOGN, +1, false, false>(tw, sm,
                                    [&](int ix) {
                                        float2 v = make_float2(0.0f, 0.0f);
                                        if ((ix < nx / 2 ? ix : nx - ix) <= kmax) {
                                            const uint4 o = philox(make_uint4((unsigned)ix, (unsigned)iy, m, GRF_TAG),
                                                                   seed_lo, seed_hi);
                                            float sn, cs;
                                            sincospif(2.0f * u24(o.x), &sn, &cs);
                                            v = make_float2(cs, sn);
                                        }
                                        return v;
                                    },
                                    [&](int i, float2 v) { d[i] = v; });
    }
}

// Column transforms without transposes: a block takes C adjacent columns of a row-major array,
// thread (c, t) = (threadIdx.x, threadIdx.y) being thread t of column c's transform, so that the
// lanes of a warp read and write C consecutive elements of each row (C x 8 bytes: whole 32-byte
// sectors for C >= 4).  Each column has its own shared buffer, C of them per block.
// columns per block by transform length, as measured on the GB300: two, except four for 2048
// points (eight 4096x2048 maps: 0.81 ms, against 0.91 with two and 0.99 with eight)
__host__ __device__ constexpr int cols_per_block(int logn) { return logn == 11 ? 4 : 2; }
// float2 elements between the shared buffers of two of C columns: at least the padded row, plus
// 8 (4 for eight columns), so that the columns a warp's lanes touch start in different banks
__host__ __device__ constexpr int col_stride(int n, int c) { return ((n + n / 16 + 1 + 15) / 16) * 16 + (c >= 8 ? 4 : 8); }
__host__ __device__ constexpr int cols_smem_bytes(int n, int c) { return c * col_stride(n, c) * (int)sizeof(float2); }
static_assert(cols_per_block(13) * fft_threads(1 << 13) <= 1024 && cols_smem_bytes(1 << 13, cols_per_block(13)) <= 227 * 1024,
              "column blocks of 8192 points exceed a block's threads or shared memory");

#define COLS_BOUNDS(L, C) __launch_bounds__((C) * fft_threads(1 << (L)), fft_minb(1 << (L), HPT_FFT_REGS * (C)))

// GRF pass 2 (Eq. 4): the unnormalised inverse FFT along y of C columns of the row pass's output
// B [ny][nx] per block, its phase (atan2) stored to phi [ny][nx] row-major.
template <int LOGN, int C>
__global__ void COLS_BOUNDS(LOGN, C) k_grf_cols(const float2 *__restrict__ B, float *__restrict__ phi, int nx, int lnx,
                                                const float2 *__restrict__ tw)
{
    extern __shared__ float2 sm[];
    const int c = threadIdx.x, t = threadIdx.y;
    const int g = blockIdx.x * C + c, ix = g & (nx - 1);      // nx >= C columns to each of the maps
    const size_t map = ((size_t)(g >> lnx) << lnx) << LOGN;
    const float2 *col = B + map + ix;
    float *out = phi + map + ix;
    float2 *buf = sm + c * col_stride(1 << LOGN, C);
    row_fft<LOGN, +1, false, false>(tw, buf, [&](int i) { return col[(size_t)i * nx]; },
                                    [&](int i, float2 v) { out[(size_t)i * nx] = atan2f(v.y, v.x); }, t);
}

// calls f(std::integral_constant<int, logn>) for logn in [1, FFT_MAX_LOG]
template <class F>
cudaError_t with_logn(int logn, F f)
{
    switch (logn) {
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
    case 13: return f(std::integral_constant<int, 13>{});
    default: return cudaErrorInvalidValue;
    }
}

int ilog2(int n)
{
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

bool pow2_in_range(int n) { return n >= 2 && n <= (1 << FFT_MAX_LOG) && (n & (n - 1)) == 0; }

// the kernels' shared-memory limits, which belong to a device
cudaError_t fft_setup(int device)
{
    static OncePerDevice once;
    return once(device, [] {
        for (int l = 1; l <= FFT_MAX_LOG; ++l) {
            cudaError_t e = with_logn(l, [&](auto L) {
                constexpr int ll = decltype(L)::value;
                const int smem = fft_smem_bytes(1 << ll);
                cudaError_t r = cudaFuncSetAttribute(k_grf_rows<ll>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
                constexpr int cc = cols_per_block(ll);
                const int csmem = cols_smem_bytes(1 << ll, cc);
                if (r == cudaSuccess) r = cudaFuncSetAttribute(k_grf_cols<ll, cc>, cudaFuncAttributeMaxDynamicSharedMemorySize, csmem);
                if (r == cudaSuccess) r = cudaFuncSetAttribute(k_grf_cols<ll, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                               cols_smem_bytes(1 << ll, 2));
                return r;
            });
            if (e != cudaSuccess) return e;
        }
        return cudaSuccess;
    });
}

}  // namespace

#define OPT_TRY(x)                                                                                  \
    do {                                                                                           \
        cudaError_t e_ = (x);                                                                      \
        if (e_ != cudaSuccess) {                                                                   \
            char m_[256];                                                                          \
            snprintf(m_, sizeof m_, "%s: %s", #x, cudaGetErrorString(e_));                         \
            return internal_fail(HPT_ERR_CUDA, m_);                                                \
        }                                                                                          \
    } while (0)

extern "C" hpt_status hpt_grf_build(hpt_ctx *ctx, uint64_t phase_seed, int32_t hologram_offset, int32_t K, int32_t nx,
                                    int32_t ny, double pitch, float *phi_dev, void *stream)
{
    hpt_status st = internal_check(ctx);
    if (st) return st;
    if (!phi_dev) return internal_fail(HPT_ERR_INVALID_ARG, "phi_dev is NULL");
    if (K < 1 || hologram_offset < 0) return internal_fail(HPT_ERR_INVALID_ARG, "K must be >= 1, hologram_offset >= 0");
    if (!pow2_in_range(nx) || !pow2_in_range(ny))
        return internal_fail(HPT_ERR_INVALID_ARG, "nx and ny must be powers of two in 2 .. 8192");
    if (!(pitch > 0.0) || !std::isfinite(pitch)) return internal_fail(HPT_ERR_INVALID_ARG, "pitch must be finite and > 0");
    OPT_TRY(cudaSetDevice(internal_ctx_device(ctx)));
    OPT_TRY(fft_setup(internal_ctx_device(ctx)));
    cudaStream_t s = (cudaStream_t)stream;
    const size_t n = (size_t)nx * ny;
    char *buf = nullptr;
    // the maps in groups of up to GROUP_BYTES of spectra: longer launches, whose last wave of blocks is a
    // smaller part
    int G = group_items(K, n * sizeof(float2), GROUP_BYTES);
    const float2 *tab;
    cudaMemPool_t pool;
    internal_optics(ctx, &tab, &pool);
    OPT_TRY(get_group(G, [&](int g) {
        return pool_alloc((void **)&buf, (size_t)g * n * sizeof(float2) + (size_t)(nx + ny) * sizeof(float2), pool, s);
    }));
    float2 *A = (float2 *)buf, *twx = A + (size_t)G * n, *twy = twx + nx;
    k_twiddles<<<(nx + 255) / 256, 256, 0, s>>>(twx, nx);
    if (ny != nx) k_twiddles<<<(ny + 255) / 256, 256, 0, s>>>(twy, ny);
    else twy = twx;
    // per group: spectra generated and transformed along x (row-major [ny][nx]), then the columns
    // transformed along y with the phase taken as they are stored
    const int lx = ilog2(nx), ly = ilog2(ny);
    const cudaError_t e = for_groups(K, G, [&](long long k, int g) {
        const cudaError_t er = with_logn(lx, [&](auto L) {
            constexpr int l = decltype(L)::value;
            k_grf_rows<l><<<(unsigned)g * ny, fft_threads(1 << l), fft_smem_bytes(1 << l), s>>>(
                A, ny, ly, (unsigned)(hologram_offset + k), (unsigned)phase_seed, (unsigned)(phase_seed >> 32), twx);
            return cudaGetLastError();
        });
        if (er != cudaSuccess) return er;
        return with_logn(ly, [&](auto L) {
            constexpr int l = decltype(L)::value;
            constexpr int cc = cols_per_block(l);
            float *dst = phi_dev + (size_t)k * n;
            const int cols = g * nx;
            if (nx >= cc)
                k_grf_cols<l, cc><<<cols / cc, dim3(cc, fft_threads(1 << l)), cols_smem_bytes(1 << l, cc), s>>>(A, dst, nx, lx, twy);
            else
                k_grf_cols<l, 2><<<cols / 2, dim3(2, fft_threads(1 << l)), cols_smem_bytes(1 << l, 2), s>>>(A, dst, nx, lx, twy);
            return cudaGetLastError();
        });
    });
    cudaError_t e2 = cudaFreeAsync(buf, s);
    OPT_TRY(e);
    OPT_TRY(e2);
    return HPT_OK;
}
