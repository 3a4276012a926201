// Packed pairs of floats: two lanes in one 64-bit register, so that an add, a multiply or an FMA of
// both is one instruction (add.rn.f32x2 and its kin).  The host forms round the same, lane by lane: the
// tests compile the code above them with the host compiler.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace hpt {

typedef unsigned long long f2;   // (lane 0, lane 1)

#ifdef __CUDACC__
__device__ __forceinline__ f2 pk(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void upk(f2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b)
{
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
#else
inline unsigned __float_as_uint(float a)
{
    unsigned r;
    __builtin_memcpy(&r, &a, 4);
    return r;
}
inline float __uint_as_float(unsigned a)
{
    float r;
    __builtin_memcpy(&r, &a, 4);
    return r;
}
inline unsigned __byte_perm(unsigned x, unsigned y, unsigned s)
{
    const unsigned long long v = (unsigned long long)y << 32 | x;
    unsigned r = 0;
    for (int i = 0; i < 4; ++i) r |= (unsigned)((v >> (8 * ((s >> (4 * i)) & 7))) & 255) << (8 * i);
    return r;
}
inline f2 pk(float a, float b) { return (f2)__float_as_uint(b) << 32 | __float_as_uint(a); }
inline void upk(f2 v, float &a, float &b)
{
    a = __uint_as_float((unsigned)v);
    b = __uint_as_float((unsigned)(v >> 32));
}
inline f2 fma2(f2 a, f2 b, f2 c)
{
    float a0, a1, b0, b1, c0, c1;
    upk(a, a0, a1);
    upk(b, b0, b1);
    upk(c, c0, c1);
    return pk(__builtin_fmaf(a0, b0, c0), __builtin_fmaf(a1, b1, c1));
}
#endif

}  // namespace hpt
