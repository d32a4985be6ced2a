// fx64.cuh -- 64-bit fixed-point arithmetic on the 32-bit integer pipes.
//
// GB300 issues one FP64 warp instruction per 64 clocks and scheduler, but a
// 32 x 32 + 64 -> 64 bit integer multiply-add (IMAD.WIDE) per 5.6 and other
// 32-bit integer instructions per 2 (measured:
// profiles/integer_and_fp64_pipe_rates.md).  A product of two 62-bit fractions,
// correct to 2^-60 of its operands' range, takes three multiply-adds, so
// arithmetic that carries more bits than an FP64 mantissa runs about three
// times faster than the FP64 pipe wherever the range of the values is known.
//
// Two forms of a 64-bit value v:
//   raw       (hi, lo) of the two's complement number (non-negative values
//             below 2^63 multiply as unsigned halves);
//   balanced  v = hi 2^32 + lo with lo read as a SIGNED 32-bit number, so that
//             every partial product is signed x signed.
#pragma once

#include <stdint.h>

namespace fmm {
namespace fx {

typedef long long s64;
typedef unsigned long long u64;

// a * b + c
__device__ __forceinline__ s64 madw(int a, int b, s64 c)
{
    s64 d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
// The same written as a product and an addition: measured, a chain of them into
// one sum takes 4.6 clocks each, of madw 5.4.  Where several results meet in later
// additions the form with the addend can be the faster one (the sums of p2p_fx.cu).
__device__ __forceinline__ s64 madp(int a, int b, s64 c)
{
    s64 d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d + c;
}
__device__ __forceinline__ u64 madu(uint32_t a, uint32_t b, u64 c)
{
    u64 d;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d + c;
}

// a shift whose amount may pass the width (the result is then 0)
__device__ __forceinline__ uint32_t shl32(uint32_t a, uint32_t n)
{
    uint32_t d;
    asm("shl.b32 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(n));
    return d;
}

__device__ __forceinline__ int hi32(s64 v) { return (int)(v >> 32); }
__device__ __forceinline__ int lo32(s64 v) { return (int)v; }

// balanced halves (|v| < 2^62)
struct I2 {
    int h, l;
};
__device__ __forceinline__ I2 bal(s64 v)
{
    const int l = (int)v;
    return {(int)(v >> 32) + (int)((uint32_t)l >> 31), l};
}

constexpr s64 kHalfUlp = 0x80000000ll;     // rounds the cross products' sum
constexpr s64 kBias = 0x80000000ll;        // see bal_biased

// the balanced halves of v given v + 2^31 (the addend of a product chain, so it
// costs nothing): the upper half comes out rounded, the lower with its sign bit
// flipped
__device__ __forceinline__ I2 bal_biased(s64 vb) { return {hi32(vb), lo32(vb) ^ (int)0x80000000}; }

// add + a b / 2^64, rounded (error below one unit); |a|, |b| < 2^62.6
__device__ __forceinline__ s64 mulhi(I2 a, I2 b, s64 add = 0)
{
    const s64 c = madp(a.h, b.l, madp(a.l, b.h, kHalfUlp));
    return madp(a.h, b.h, add + (s64)hi32(c));
}
// a b / 2^62, rounded: two more bits where the product is known to stay below 2^62
__device__ __forceinline__ s64 mulhi_62(I2 a, I2 b)
{
    const s64 c = madp(a.h, b.l, madp(a.l, b.h, kHalfUlp / 4));
    return (madp(a.h, b.h, 0) << 2) + (c >> 30);
}
// add + (a0 b0 + a1 b1 + a2 b2) / 2^64, rounded; the halves' cross products must
// sum below 2^63
__device__ __forceinline__ s64 dot3hi(I2 a0, I2 b0, I2 a1, I2 b1, I2 a2, I2 b2, s64 add = 0)
{
    s64 c = madp(a0.h, b0.l, madp(a0.l, b0.h, kHalfUlp));
    c = madp(a1.h, b1.l, madp(a1.l, b1.h, c));
    c = madp(a2.h, b2.l, madp(a2.l, b2.h, c));
    return madp(a2.h, b2.h, madp(a1.h, b1.h, madp(a0.h, b0.h, add + (s64)hi32(c))));
}
// add + a b / 2^64 modulo 2^64, for 0 <= a, b < 2^63 (error below two units, downward)
__device__ __forceinline__ u64 mulhi_u(u64 a, u64 b, u64 add = 0)
{
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a, bh = (uint32_t)(b >> 32), bl = (uint32_t)b;
    const u64 c = madu(ah, bl, madu(al, bh, 0));
    return madu(ah, bh, add + (c >> 32));
}

// round(x 2^sc) modulo 2^64: exact unless bits fall below 2^0, whatever the
// size of x, so that differences of nearby values are right although each of
// them may exceed the range.  x finite.
__device__ __forceinline__ s64 fix64(double x, int sc)
{
    const s64 b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7ff);
    u64 m = (u64)b & 0xfffffffffffffull;
    if (ex) m |= 1ull << 52;
    const int sh = (ex ? ex : 1) - 1075 + sc;
    u64 v;
    if (sh >= 0) {
        v = sh < 64 ? m << sh : 0ull;
    } else {
        const int r = -sh;
        v = r <= 54 ? (m + (1ull << (r - 1))) >> r : 0ull;
    }
    return b < 0 ? -(s64)v : (s64)v;
}

}  // namespace fx
}  // namespace fmm
