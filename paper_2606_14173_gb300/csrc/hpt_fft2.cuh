// Packed FFT core of the wave optics: pairs of power-of-two transforms of equal length, one in each
// half of a 64-bit register pair, so that every add, multiply and FMA of a pass is one packed
// instruction (fma.rn.f32x2 and its kin) for both.
//
// The two halves come from one transform of twice the length.  Forward, a zero-extended sequence of
// at most M = N / 2 points has as its even frequencies the M-point transform of x[n] and as its odd
// ones that of x[n] exp(-2 pi i n / N); back, the first M of N points are
// IFFT(even)[n] + exp(2 pi i n / N) IFFT(odd)[n].  So a padded transform never touches its zeros, and
// neither lane needs the other between the load and the store.
//
// M points are transformed by M / 16 threads (16 points of both lanes, 64 registers, each): Stockham
// passes of radix 16 with the remainder radix last (forward) or first (inverse), exchanged through
// one shared buffer of M 16-byte elements.  A thread's outputs of the forward's last pass are the
// inputs of the same thread in the inverse's first pass, so a convolution multiplies its spectrum in
// registers between them.
#pragma once
#include <cuda_runtime.h>

#include "hpt_pair.cuh"

namespace hpt {

struct c2 {   // two complex numbers, one per lane
    f2 re, im;
};

__device__ __forceinline__ c2 cadd(c2 a, c2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ c2 csub(c2 a, c2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// v * w, or v * conj(w)
template <bool CONJ>
__device__ __forceinline__ c2 cmul2(c2 v, f2 wr, f2 wi)
{
    if (CONJ) return {fma2(v.re, wr, mul2(v.im, wi)), sub2(mul2(v.im, wr), mul2(v.re, wi))};
    return {sub2(mul2(v.re, wr), mul2(v.im, wi)), fma2(v.re, wi, mul2(v.im, wr))};
}

// the cosines of pi / 8, pi / 4 and 3 pi / 8 in both halves of a register pair each
struct Roots {
    f2 c1, c2, c3;
    static __device__ __forceinline__ f2 twice(float x)
    {
        f2 r;
        asm volatile("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));   // kept in registers, not made anew at each use
        return r;
    }
    static __device__ __forceinline__ Roots make() { return {twice(0.923879533f), twice(0.707106781f), twice(0.382683432f)}; }
};

// a, b -> a + w b, a - w b with w = exp(-2 pi i m / 16) (INV: its conjugate), m < 8
template <bool INV>
__device__ __forceinline__ void butterfly(c2 &a, c2 &b, int m, const Roots &K)
{
    c2 w = b;
    bool nre = false, nim = false;    // the parts of w b come negated
    if (m == 4) {
        w = {b.im, b.re};             // -i b, or i b
        nre = INV;
        nim = !INV;
    } else if (m == 2) {              // (1 -+ i) / sqrt 2
        w = INV ? c2{mul2(sub2(b.re, b.im), K.c2), mul2(add2(b.re, b.im), K.c2)}
                : c2{mul2(add2(b.re, b.im), K.c2), mul2(sub2(b.im, b.re), K.c2)};
    } else if (m == 6) {              // (-1 -+ i) / sqrt 2
        w = INV ? c2{mul2(add2(b.re, b.im), K.c2), mul2(sub2(b.re, b.im), K.c2)}
                : c2{mul2(sub2(b.im, b.re), K.c2), mul2(add2(b.re, b.im), K.c2)};
        nre = INV;
        nim = !INV;
    } else if (m != 0) {
        // |cos|, |sin| of the root's angle; its cosine is negative for m > 4
        const f2 c = m == 1 || m == 7 ? K.c1 : K.c3, s = m == 1 || m == 7 ? K.c3 : K.c1;
        const bool neg = m > 4;
        // fwd: re = +-c b.re + s b.im, im = +-c b.im - s b.re; inv: re = +-c b.re - s b.im, im = +-c b.im + s b.re
        const f2 pr = mul2(b.re, c), pi = mul2(b.im, c);
        if (!INV) {
            w.re = neg ? sub2(mul2(b.im, s), pr) : fma2(b.im, s, pr);
            if (neg) { w.im = fma2(b.re, s, pi); nim = true; }
            else w.im = sub2(pi, mul2(b.re, s));
        } else {
            if (neg) { w.re = fma2(b.im, s, pr); nre = true; }
            else w.re = sub2(pr, mul2(b.im, s));
            w.im = neg ? sub2(mul2(b.re, s), pi) : fma2(b.re, s, pi);
        }
    }
    const c2 x = a;
    a = {nre ? sub2(x.re, w.re) : add2(x.re, w.re), nim ? sub2(x.im, w.im) : add2(x.im, w.im)};
    b = {nre ? add2(x.re, w.re) : sub2(x.re, w.re), nim ? add2(x.im, w.im) : sub2(x.im, w.im)};
}

// R-point DFT of both lanes in registers (R = 1, 2, 4, 8, 16): bit-reversed order, then radix-2
// stages; INV: the conjugate roots, unnormalised.
template <int R, bool INV>
__device__ __forceinline__ void dft2(c2 *v, const Roots &K)
{
    if constexpr (R > 1) {
        constexpr int B = R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : 4;
        c2 t[R];
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
                for (int pos = 0; pos < half; ++pos) butterfly<INV>(t[g + pos], t[g + pos + half], pos * (8 / half), K);
            }
        }
#pragma unroll
        for (int i = 0; i < R; ++i) v[i] = t[i];
    }
}

// ---- shape of an M = 2^LM point transform ---------------------------------------------------
constexpr int FFT2_MAX_LM = 12;
__host__ __device__ constexpr int fft2_points(int lm) { return lm >= 4 ? 16 : 1 << lm; }    // per thread and lane
__host__ __device__ constexpr int fft2_threads(int lm) { return lm >= 4 ? 1 << (lm - 4) : 1; }
__host__ __device__ constexpr int fft2_npass(int lm) { return lm == 0 ? 1 : (lm + 3) / 4; }
// radix of pass p: 16s with the remainder last (forward) or first (inverse)
__host__ __device__ constexpr int fft2_radix(int lm, bool inv, int p)
{
    if (lm == 0) return 1;
    const int rem = lm & 3, n = fft2_npass(lm);
    return rem && p == (inv ? 0 : n - 1) ? 1 << rem : 16;
}
__host__ __device__ constexpr int fft2_ns(int lm, bool inv, int p)
{
    int s = 1;
    for (int i = 0; i < p; ++i) s *= fft2_radix(lm, inv, i);
    return s;
}
// Twiddle tables, all lengths in one array: the split's roots exp(-2 pi i n / 2M), n < M, then for each
// pass p >= 1 of M points exp(-2 pi i r k / (NS R)) at [(r - 1) NS + k] (r = 1 .. R - 1, k < NS:
// neighbouring threads read neighbouring entries).  Duplicating an entry into both halves takes four
// moves; entries stored twice took twice the L1 wavefronts, of which the passes are short.
__host__ __device__ constexpr int fft2_pass_entries(int lm, bool inv, int p)
{
    return p == 0 ? 0 : (fft2_radix(lm, inv, p) - 1) * fft2_ns(lm, inv, p);
}
__host__ __device__ constexpr int fft2_len_entries(int lm)
{
    int e = 1 << lm;
    for (int p = 1; p < fft2_npass(lm); ++p) e += fft2_pass_entries(lm, false, p) + fft2_pass_entries(lm, true, p);
    return e;
}
__host__ __device__ constexpr int fft2_base(int lm)
{
    int b = 0;
    for (int l = 0; l < lm; ++l) b += fft2_len_entries(l);
    return b;
}
__host__ __device__ constexpr int fft2_pass_off(int lm, bool inv, int p)
{
    int b = fft2_base(lm) + (1 << lm);
    for (int d = 0; d < 2; ++d)
        for (int q = 1; q < fft2_npass(lm); ++q) {
            if ((d == 1) == inv && q == p) return b;
            b += fft2_pass_entries(lm, d == 1, q);
        }
    return b;
}
constexpr int FFT2_TABLE_ENTRIES = fft2_base(FFT2_MAX_LM + 1);

// Shared-memory place of point i when it is stored by pass p: padded by one element after every R of a
// first pass (whose stores lie R apart) and after every 16 otherwise, so that the eight lanes of a
// 16-byte access phase fall in distinct banks, storing and loading.
__host__ __device__ constexpr int fft2_log2(int r) { return r <= 1 ? 0 : 1 + fft2_log2(r / 2); }
__host__ __device__ constexpr int fft2_pad_shift(int lm, bool inv, int p) { return p == 0 ? fft2_log2(fft2_radix(lm, inv, 0)) : 4; }
// shared elements (16 bytes) of one transform: the padded points, plus four modulo eight, so that two
// transforms whose threads alternate in a warp start in different banks
__host__ __device__ constexpr int fft2_smem_elems(int lm)
{
    if (fft2_npass(lm) == 1) return 0;
    const int m = 1 << lm, sh = fft2_pad_shift(lm, true, 0);   // the inverse's first radix is the smaller one
    return ((m + (m >> sh) + 7) / 8) * 8 + 4;
}

// One thread's part (thread t) of an M-point transform of both lanes.
template <int LM, bool INV>
struct Fft2 {
    static constexpr int M = 1 << LM, T = fft2_threads(LM), N = fft2_points(LM), NP = fft2_npass(LM);
    static constexpr int SMEM = fft2_smem_elems(LM), ROOTS = fft2_base(LM);

    // the point index of element m (r-th input) of pass P's butterflies
    template <int P> static __device__ __forceinline__ int in_index(int t, int e)
    {
        constexpr int R = fft2_radix(LM, INV, P), Q = M / R;
        return t + (e / R) * T + (e % R) * Q;
    }
    template <int P> static __device__ __forceinline__ int out_index(int t, int e)
    {
        constexpr int R = fft2_radix(LM, INV, P), NS = fft2_ns(LM, INV, P);
        const int j = t + (e / R) * T, k = j & (NS - 1);
        return (j - k) * R + k + (e % R) * NS;
    }
    // twiddles and butterflies of pass P on the thread's N points
    template <int P> static __device__ __forceinline__ void butterflies(c2 *v, int t, const float2 *__restrict__ tab, const Roots &K)
    {
        constexpr int R = fft2_radix(LM, INV, P), NS = fft2_ns(LM, INV, P), J = N / R;
#pragma unroll
        for (int m = 0; m < J; ++m) {
            if constexpr (P > 0) {
                const int k = (t + m * T) & (NS - 1);
                constexpr int OFF = fft2_pass_off(LM, INV, P);
                const float2 *w = tab + OFF + k;
#pragma unroll
                for (int r = 1; r < R; ++r) {
                    const float2 q = __ldg(w + (r - 1) * NS);
                    v[m * R + r] = cmul2<INV>(v[m * R + r], pk(q.x, q.x), pk(q.y, q.y));
                }
            }
            dft2<R, INV>(v + m * R, K);
        }
    }
    // A pass's points lie a power of two apart, from a first point whose index modulo the padding's
    // period leaves room for every step's remainder: the padded place is that of the first point plus
    // a constant (the propagation tests go through every length).
    template <int P> static __device__ __forceinline__ void put(const c2 *v, int t, ulonglong2 *buf)
    {
        constexpr int R = fft2_radix(LM, INV, P), NS = fft2_ns(LM, INV, P), SH = fft2_pad_shift(LM, INV, P);
#pragma unroll
        for (int m = 0; m < N / R; ++m) {
            const int o = out_index<P>(t, m * R);
            ulonglong2 *b = buf + o + (o >> SH);
#pragma unroll
            for (int r = 0; r < R; ++r) b[r * NS + ((r * NS) >> SH)] = make_ulonglong2(v[m * R + r].re, v[m * R + r].im);
        }
    }
    template <int P> static __device__ __forceinline__ void get(c2 *v, int t, const ulonglong2 *buf)
    {
        constexpr int R = fft2_radix(LM, INV, P), Q = M / R, SH = fft2_pad_shift(LM, INV, P - 1);
#pragma unroll
        for (int m = 0; m < N / R; ++m) {
            const int i = in_index<P>(t, m * R);
            const ulonglong2 *b = buf + i + (i >> SH);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const ulonglong2 q = b[r * Q + ((r * Q) >> SH)];
                v[m * R + r].re = q.x;
                v[m * R + r].im = q.y;
            }
        }
    }
    // passes P .. NP - 1 on the values of pass P's inputs: leaves the last pass's outputs in v.
    // 'bar' synchronises the transform's threads; on entry the buffer may still be read by others
    // when FRESH is false.
    template <int P, bool FRESH, class BAR>
    static __device__ __forceinline__ void run(c2 *v, int t, ulonglong2 *buf, const float2 *__restrict__ tab, const Roots &K,
                                               BAR bar)
    {
        butterflies<P>(v, t, tab, K);
        if constexpr (P + 1 < NP) {
            if constexpr (!FRESH) bar();
            put<P>(v, t, buf);
            bar();
            get<P + 1>(v, t, buf);
            run<P + 1, false>(v, t, buf, tab, K, bar);
        }
    }
};

}  // namespace hpt
