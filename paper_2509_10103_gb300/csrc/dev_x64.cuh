// Block-floating 64-bit integer arithmetic for the kernels that carry FP64
// values but spend their time on the FP64 pipe.  That pipe executes one warp
// instruction per scheduler in 77 cycles on this GPU; a 32x32+64-bit integer
// multiply-add (IMAD.WIDE) takes 4.2, a 64-bit addition 2.2 and a 64-bit shift
// about 4 (measured, 16 warps per SM), so a product of two 64-bit fixed-point
// numbers, four multiply-adds, costs about a quarter of one FP64 FMA.
//
// A value is an integer v of at most 60 bits and the exponent E of its unit:
// x = v 2^E.  The values that meet in a sum share E, which follows their
// largest magnitude, so that sums are exact and only the final result is
// rounded (to nearest) when it becomes an FP64 number again.
// Multipliers are fixed-point with kXF fractional bits.  Both factors are
// split into a signed high and a signed low 32-bit digit, so every partial
// product is a signed 32x32 one.
#pragma once

#include <cuda_runtime.h>

namespace pnop {

constexpr int kXF = 58;  // fractional bits of a multiplier

// x < 2^60 in units of 2^E when E >= field - kXTop, field the exponent field of x
constexpr int kXTop = 1082;
constexpr int kXZero = -100000;  // unit of an empty window

// Loads of FP64 values as integers in units of 2^E, E >= -kXTop: the exponent
// field is moved by integer arithmetic, the conversion (to the nearest integer)
// is the FP64 pipe's, which the integer sweeps leave idle.  Values below
// 2^-1022 in that unit, zeros and subnormals are 0.
struct xunit {
    int e20, lim;  // E 2^20; high words up to lim (sign cleared) are 0
};
__device__ __forceinline__ xunit x_unit(int E) {
    xunit u;
    u.e20 = E * (1 << 20);
    u.lim = max(u.e20, 0) + 0xFFFFF;
    return u;
}
__device__ __forceinline__ long long x_load(double x, xunit u) {
    const int h = __double2hiint(x);
    const int hi = (h & 0x7FFFFFFF) > u.lim ? h - u.e20 : 0;
    return __double2ll_rn(__hiloint2double(hi, __double2loint(x)));
}
// v 2^E as FP64, for -1000 <= E <= 900 or v = 0; nan = 0x7FF80000 makes it NaN
__device__ __forceinline__ double x_store(long long v, int E, int nan) {
    const double d = __ll2double_rn(v);
    const int h = __double2hiint(d);
    return __hiloint2double((h ? h + E * (1 << 20) : 0) | nan, __double2loint(d));
}
// the same for any E (underflow to zero, overflow to infinity)
__device__ __forceinline__ double x_store_any(long long v, int E, int nan) {
    const double d = __ll2double_rn(v);
    const int h = __double2hiint(d), f = ((h >> 20) & 0x7FF) + E;
    if (nan) return __hiloint2double(nan, 0);
    if (v == 0 || f <= 0) return 0.0;
    if (f >= 2047) return __hiloint2double((h & (int)0x80000000) | 0x7FF00000, 0);
    return __hiloint2double(h + E * (1 << 20), __double2loint(d));
}
// v 2^-n to the nearest integer, n of either sign, |v| < 2^62 (the caller bounds
// left shifts)
struct xmove {
    int right, left;
    long long half;
    __device__ __forceinline__ explicit xmove(int n) {
        right = min(max(n, 0), 62);
        left = min(max(-n, 0), 62);
        half = (1ll << right) >> 1;
    }
    __device__ __forceinline__ long long operator()(long long v) const { return ((v + half) >> right) << left; }
};

// signed 32-bit digits: v = h 2^32 + l
struct xdig {
    int h, l;
};
__device__ __forceinline__ xdig x_split(long long v) {
    xdig d;
    d.l = (int)v;
    d.h = (int)((v + (1ll << 31)) >> 32);
    return d;
}
__device__ __forceinline__ long long x_join(xdig d) { return ((long long)d.h << 32) + (long long)d.l; }

// a b + c with 32-bit factors (written out: from C++ products the compiler made
// 64x64-bit ones of most)
__device__ __forceinline__ long long x_mad(int a, int b, long long c) {
    long long d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
}
__device__ __forceinline__ long long x_mul(int a, int b) {
    long long d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
}
// half a unit of what x_dot drops, in a register pair of its own (as a
// constant it is set up again for every row)
template <int F = kXF> __device__ __forceinline__ long long x_half() {
    long long d;
    asm volatile("mov.b64 %0, %1;" : "=l"(d) : "n"(1ll << (F - 33)));
    return d;
}
// sum of four products (multiplier digits c: x low, y high; value digits w),
// the last one ready last; two accumulators for the products of low digits,
// which reach 2^62 each
__device__ __forceinline__ long long x_dot4(int2 c0, xdig w0, int2 c1, xdig w1, int2 c2, xdig w2, int2 c3, xdig w3,
                                            long long half) {
    long long l0 = x_mad(c1.x, w1.l, x_mul(c0.x, w0.l)), l1 = x_mad(c3.x, w3.l, x_mul(c2.x, w2.l));
    long long m = x_mad(c0.y, w0.l, x_mad(c0.x, w0.h, half));
    m = x_mad(c1.y, w1.l, x_mad(c1.x, w1.h, m));
    m = x_mad(c2.y, w2.l, x_mad(c2.x, w2.h, m));
    m = x_mad(c3.y, w3.l, x_mad(c3.x, w3.h, m));
    const long long h = x_mad(c3.y, w3.h, x_mad(c2.y, w2.h, x_mad(c1.y, w1.h, x_mul(c0.y, w0.h))));
    m += (long long)(int)(l0 >> 32) + (long long)(int)(l1 >> 32);
    return (h << (64 - kXF)) + (m >> (kXF - 32));
}
// one product with F fractional bits
template <int F> __device__ __forceinline__ long long x_prod(int2 c, xdig w, long long half) {
    const long long l = x_mul(c.x, w.l);
    const long long m = x_mad(c.y, w.l, x_mad(c.x, w.h, half)) + (long long)(int)(l >> 32);
    return (x_mul(c.y, w.h) << (64 - F)) + (m >> (F - 32));
}
__device__ __forceinline__ int x_mag(xdig d) { return d.h ^ (d.h >> 31); }  // high digit of |v| (or |v| - 1)

}  // namespace pnop
