// 64-bit fixed-point complex arithmetic for the FP64 transforms.
//
// GB300's FP64 pipe retires 2 lanes per clock and SM (a warp's DFMA holds its
// scheduler's share for 64 cycles), its integer pipes 64-128.  The transforms
// of FP64 contexts therefore run on integers in block floating point: a warp
// (x and z passes) or a tile (y passes) shares one exponent, a value is
// x 2^ex with a 64-bit integer x, additions are exact and a complex product
// with a 60-bit twiddle takes 12 32x32+64-bit multiply-adds.  Before every
// radix-16 stage the values are shifted so that the largest sum of magnitudes
// that one butterfly combines fills FX_TOP bits, the most for which the stage
// cannot overflow: the largest of its 32 components is then at least about 2^54
// units.  A value enters the butterfly with an error of up to two units (half a
// unit from the shift, up to 1.5 from a twiddle product, which drops the low
// parts' products).  These errors are relative to the largest component of the
// warp or tile, FP64's to each value; measured against 80-bit arithmetic the
// potentials' error is 0.6-1.0 of that of FP64 transforms (grids of 16^3 to 64^3
// and 256 x 16 x 64).  Work arrays, H-hat and potentials stay FP64 in memory.
#pragma once

#include "pm_internal.cuh"

// Compute types of the transforms: FP32 values in FP32, FP64 values in block
// floating point; TW is the element of their twiddle tables.
struct fx2 { long long x, y; };
struct __align__(16) fxw { int rh, rl, ih, il; };   // w = (h 2^30 + l) 2^-60, l in [-2^29, 2^29)

template <typename T> struct comp_t;
template <> struct comp_t<float> { typedef float2 V; typedef float2 W; };
template <> struct comp_t<double> { typedef fx2 V; typedef fxw W; };

namespace pmfx {

constexpr int FX_Q = 60;      // fraction bits of twiddles and normalised factors

// The values of a stage are scaled so that the sum of the magnitudes that one
// butterfly combines, and with it every value it forms, stays below 2^FX_TOP
// (a product's operand must stay below 2^61, and the rotations by odd
// multiples of pi/4 add two components first).  The sum, rather than 16 times
// the largest, keeps the bits that a peaked spectrum leaves free.
constexpr int FX_TOP = 60;

__device__ __forceinline__ long long madw(int a, int b, long long c) { return (long long)a * b + c; }
// |x| < 2^61 as h 2^30 + l, 0 <= l < 2^30
__device__ __forceinline__ void split(long long x, int &h, int &l) {
    h = (int)(x >> 30);
    l = (int)x & 0x3fffffff;
}
// x w 2^-60 for a real factor w = (wh 2^30 + wl) 2^-60 (rounded; the product
// of the low parts, below one unit, is dropped)
__device__ __forceinline__ long long mulr(long long x, int wh, int wl) {
    int h, l;
    split(x, h, l);
    long long m = madw(h, wl, 1LL << 29);
    m = madw(l, wh, m);
    return madw(h, wh, m >> 30);
}
__device__ __forceinline__ fx2 cmulw(fx2 v, int rh, int rl, int ih, int il) {
    int xh, xl, yh, yl;
    split(v.x, xh, xl);
    split(v.y, yh, yl);
    const int nh = -ih, nl = -il;
    long long m = madw(xh, rl, 1LL << 29);
    m = madw(xl, rh, m);
    m = madw(yh, nl, m);
    m = madw(yl, nh, m);
    fx2 r;
    r.x = madw(yh, nh, madw(xh, rh, m >> 30));
    m = madw(xh, il, 1LL << 29);
    m = madw(xl, ih, m);
    m = madw(yh, rl, m);
    m = madw(yl, rh, m);
    r.y = madw(yh, rh, madw(xh, ih, m >> 30));
    return r;
}
// a factor q 2^-60 (|q| <= 2^60) as its two parts
__host__ __device__ __forceinline__ void wsplit(long long q, int &h, int &l) {
    h = (int)((q + (1LL << 29)) >> 30);
    l = (int)(q - ((long long)h << 30));
}
__device__ __forceinline__ fx2 cmulq(fx2 v, long long qr, long long qi) {
    int rh, rl, ih, il;
    wsplit(qr, rh, rl);
    wsplit(qi, ih, il);
    return cmulw(v, rh, rl, ih, il);
}

// Upper bound, in units of 2^35, of the magnitudes' sum over each group of R
// of the 16 values, the largest of the groups; the high words of |x| < 2^61
// are summed by eights, so that nothing overflows.
template <int R> __device__ __forceinline__ unsigned group_sum(const fx2 *v) {
    unsigned best = 0;
#pragma unroll
    for (int g = 0; g < 16 / R; ++g) {
        unsigned tot = 0, part = 0;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            part += (unsigned)abs((int)(v[g * R + r].x >> 32)) + (unsigned)abs((int)(v[g * R + r].y >> 32));
            if (r % 4 == 3 || r == R - 1) {
                tot += part >> 3;
                part = 0;
            }
        }
        best = max(best, tot);
    }
    return best + 12;   // what the high words and the shifts left out
}
// Bits of the largest of N values' components over the warp.
template <int N> __device__ __forceinline__ int warp_bits(const fx2 *v) {
    unsigned h = 0, l = 0;
#pragma unroll
    for (int e = 0; e < N; ++e) {
        const long long x = v[e].x ^ (v[e].x >> 63), y = v[e].y ^ (v[e].y >> 63);
        h |= (unsigned)(x >> 32) | (unsigned)(y >> 32);
        l |= (unsigned)x | (unsigned)y;
    }
    h = __reduce_or_sync(0xffffffffu, h);
    l = __reduce_or_sync(0xffffffffu, l);
    return h ? 64 - __clz((int)h) : 32 - __clz((int)l);
}
// Right shift that brings a group_sum below 2^top.
__device__ __forceinline__ int sum_shift(unsigned m, int top) { return 35 + 32 - __clz((int)m) - top; }

// Multiplies every component by 2^-s, s of either sign (rounded: truncation
// would add half a unit to every value, which the next stage sums into one).
template <int N> __device__ __forceinline__ void shift(fx2 *v, int s) {
    if (s > 0) {
        s = min(s, 62);
        const long long h = 1LL << (s - 1);
#pragma unroll
        for (int e = 0; e < N; ++e) {
            v[e].x = (v[e].x + h) >> s;
            v[e].y = (v[e].y + h) >> s;
        }
    } else if (s < 0) {
#pragma unroll
        for (int e = 0; e < N; ++e) {
            v[e].x = (long long)((unsigned long long)v[e].x << -s);
            v[e].y = (long long)((unsigned long long)v[e].y << -s);
        }
    }
}

// shift for integers of all 64 bits (the rounding bit is added after the
// shift: 2^(s-1) added before it would wrap within that of 2^63).
template <int N> __device__ __forceinline__ void shift_full(fx2 *v, int s) {
    if (s <= 0) return shift<N>(v, s);
#pragma unroll
    for (int e = 0; e < N; ++e) {
        v[e].x = (v[e].x >> s) + ((v[e].x >> (s - 1)) & 1);
        v[e].y = (v[e].y >> s) + ((v[e].y >> (s - 1)) & 1);
    }
}

// FP64 <-> fixed point by integer operations (the conversions run on the FP64
// pipe too).  hi word without sign: orders like |d|.
__device__ __forceinline__ unsigned dmag(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
// d as q 2^(em - 1022 - K) with |q| < 2^K, K in 53..63 (truncated; negative
// values one unit low, a zero's too).  em: group_em.
template <int K> __device__ __forceinline__ long long from_double(double d, int em) {
    const int hi = __double2hiint(d);
    const int e = (hi >> 20) & 0x7ff;
    const unsigned long long m = ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32 |
                                  (unsigned)__double2loint(d)) << (K - 53);
    return (long long)(m >> min(em - e, 63)) ^ (long long)(hi >> 31);
}
// x 2^ex for |x| < 2^61, rounded to nearest (a negative x one unit high).
// CHECK: ex may put the result out of range (then 0, infinity or, for
// FX_NAN, NaN); without, -1000 < ex < 900.  Never -0.0, of which from_double
// would make a unit.
template <bool CHECK> __device__ __forceinline__ double to_double(long long x, int ex) {
    int s = (int)(x >> 63);
    unsigned h = (unsigned)(x >> 32) ^ (unsigned)s, l = (unsigned)x ^ (unsigned)s;
    int E = 1023 + 62 - 1 + ex;   // biased exponent - 1 of a leading bit 62 (which adds it)
    if (h == 0) { h = l; l = 0; E -= 32; }
    const int n = __clz((int)h);   // at least 3 for the first word; a second word may fill all 32
    E -= n - 1;
    const unsigned long long a = (unsigned long long)h << 32 | l;
    unsigned long long m = (n > 0 ? a << (n - 1) : a >> 1) + 0x200u;
    m = (m >> 10) + ((unsigned long long)(unsigned)E << 52);
    if (h == 0) m = 0;
    if (CHECK) {
        if (ex > (1 << 15)) m = 0x7ff8000000000000ull;
        else if (E < 0) { m = 0; s = 0; }
        else if (E >= 2046) m = 0x7ff0000000000000ull;
    }
    return __hiloint2double((int)((unsigned)(m >> 32) | ((unsigned)s & 0x80000000u)), (int)(unsigned)m);
}
__device__ __forceinline__ bool in_range(int ex) { return ex > -1000 && ex < 900; }

__device__ __forceinline__ unsigned warp_max(unsigned m) { return __reduce_max_sync(0xffffffffu, m); }

// Exponent of values that held an infinity or a NaN (they come out as NaN).
constexpr int FX_NAN = 1 << 16;
constexpr int FX_LOW = -(1 << 16);   // below every exponent
constexpr int FX_ZERO = -900;        // the exponent given to zeros
// em and ex of a group whose largest dmag is m, converted with K bits.  em is
// at least 64, so that a zero, whose implicit bit from_double does not mask, is
// shifted out: the unit of a group below 2^-958 stays at 2^(-958 - K), and what
// is below it vanishes.  A group of zeros: em beyond every shift.
__device__ __forceinline__ int group_em(unsigned m) {
    const int e = (int)(m >> 20);
    return e > 64 ? e : m ? 64 : 1 << 13;
}
__device__ __forceinline__ bool group_zero(int em) { return em > 0x7ff; }
__device__ __forceinline__ int group_ex(int em, int K) { return em == 0x7ff ? FX_NAN : group_zero(em) ? FX_ZERO : em - 1022 - K; }
// What a factor converted with FX_Q bits adds to a product's exponent; a factor
// of zero takes every value below the FP64 range (and leaves FX_NAN beyond it).
__device__ __forceinline__ int factor_ex(int em) { return group_zero(em) ? -(1 << 14) : group_ex(em, FX_Q) + FX_Q; }

}  // namespace pmfx

// twiddle products (overloads of the FP32 helpers)
__device__ __forceinline__ fx2 cmul(fx2 a, fxw w) { return pmfx::cmulw(a, w.rh, w.rl, w.ih, w.il); }
__device__ __forceinline__ fx2 cconjmul(fx2 a, fxw w) { return pmfx::cmulw(a, w.rh, w.rl, -w.ih, -w.il); }
