// Block fixed-point complex arithmetic for the 64-bit convolution passes
// (internal).
//
// The FP64 pipe of this GPU issues two lanes a clock and SM, the integer pipe
// 64: measured in registers, 1.7 DFMA lanes a clock and SM against 55 lanes of
// 64-bit adds and 32 of 32 x 32 + 64-bit multiply-adds.  An FFT butterfly is
// mostly adds, so a transform on 64-bit integers with one exponent per
// transform runs several times faster than in FP64, and keeps more bits: the
// components of a pass's input stay below 2^58, so one unit in the last place
// is 2^-58 of the largest value, where FP64 rounds every result to 2^-53 of
// itself.
//
// A value is x 2^e with x a signed 64-bit integer and e shared by a transform
// (a block-wide reduction of the leading bits after each pass rescales it, so
// a pass loses no more bits than the data grew by).  Twiddles are Q62, held
// as two 31-bit halves so that a product is three 32-bit multiply-adds.
//
// Bounds: a radix-8 pass multiplies components by at most 8 sqrt(2) = 2^3.5,
// so inputs below 2^58 leave below 2^61.5.  A complex product's middle
// sum, with both operands split into centred halves (low halves at most 2^30)
// and |wr| + |wi| <= sqrt(2), is at most 2^30 sqrt(2) 2^31 + 2 |ah| 2^30 <
// 2^63 while the components are below 2^62.
#pragma once
#include "common.cuh"

struct __align__(16) fxc {
    long long x, y;
};

__device__ __forceinline__ fxc operator+(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fxc operator-(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }

constexpr int FX_TOP = 58;               // a pass's input components are below 2^FX_TOP
constexpr int FX_NAN = 1 << 28;          // exponent of data that held a NaN or an infinity
constexpr int FX_ZERO = -(1 << 28);      // exponent of an all-zero row pair

// a = ah 2^31 + al with |al| <= 2^30: centred, so that the dropped low product has no mean
struct FxSplit {
    int h, l;
};
__device__ __forceinline__ FxSplit fx_split(long long a) {
    return FxSplit{(int)((a + (1ll << 30)) >> 31), ((int)a << 1) >> 1};
}
__device__ __forceinline__ long long fx_mw(int a, int b) { return (long long)a * (long long)b; }

// a b 2^-62 rounded, b = (bh, bl) a Q62 real
__device__ __forceinline__ long long fx_rmul(long long a, int bh, int bl) {
    const FxSplit s = fx_split(a);
    const long long t = (1ll << 30) + fx_mw(s.h, bl) + fx_mw(s.l, bh);
    return (t >> 31) + fx_mw(s.h, bh);
}

// a w 2^-62, w = (re high, re low, im high, im low) a Q62 complex
__device__ __forceinline__ fxc fx_cmul(fxc a, int4 w) {
    const FxSplit x = fx_split(a.x), y = fx_split(a.y);
    const int nz = -w.z, nw = -w.w;
    const long long tr = (1ll << 30) + fx_mw(x.h, w.y) + fx_mw(x.l, w.x) + fx_mw(y.h, nw) + fx_mw(y.l, nz);
    const long long ti = (1ll << 30) + fx_mw(x.h, w.w) + fx_mw(x.l, w.z) + fx_mw(y.h, w.y) + fx_mw(y.l, w.x);
    fxc r;
    r.x = (tr >> 31) + fx_mw(x.h, w.x) + fx_mw(y.h, nz);
    r.y = (ti >> 31) + fx_mw(x.h, w.z) + fx_mw(y.h, w.x);
    return r;
}

// centred halves of a Q62 constant, |c| <= 2^62 - 1: c = high 2^31 + low with
// |low| <= 2^30, except that the high half of values within 2^30 of +-2^62
// would not fit (there: 2^31 - 1 and what is left)
__host__ __device__ constexpr int fx_high(long long c) {
    return c > (1ll << 62) - (1ll << 30) - 1 ? 0x7FFFFFFF
         : c < -(1ll << 62) + (1ll << 30) + 1 ? -0x7FFFFFFF : (int)((c + (1ll << 30)) >> 31);
}
__host__ __device__ constexpr int fx_low(long long c) { return (int)(c - (long long)fx_high(c) * (1ll << 31)); }

// cos(pi/4) in Q62
constexpr long long FX_SQRT1_2 = 3260954456333195553ll;

// x exp(-2 pi i M / 16) for the even M of butterflies up to radix 8
template <int M>
__device__ __forceinline__ fxc fx_rot16(fxc x) {
    static_assert(M % 2 == 0, "radix-16 rotations are not used in fixed point");
    constexpr int m = M & 15;
    if (m == 0) return x;
    if (m == 4) return fxc{x.y, -x.x};
    if (m == 8) return fxc{-x.x, -x.y};
    if (m == 12) return fxc{-x.y, x.x};
    constexpr int h = fx_high(FX_SQRT1_2), l = fx_low(FX_SQRT1_2);
    const long long s = fx_rmul(x.x + x.y, h, l), d = fx_rmul(x.y - x.x, h, l);   // x (1 - i)/sqrt 2
    if (m == 2) return fxc{s, d};
    if (m == 6) return fxc{d, -s};
    if (m == 10) return fxc{-s, -d};
    return fxc{-d, s};
}

// leading-bit mask of a component: bit b set iff its magnitude may reach 2^(32 + b)
__device__ __forceinline__ unsigned fx_mask(fxc a) {
    const int xh = (int)(a.x >> 32), yh = (int)(a.y >> 32);
    return (unsigned)((xh ^ (xh >> 31)) | (yh ^ (yh >> 31)));
}
// shift that brings data of this mask below 2^FX_TOP (negative: to the left)
__device__ __forceinline__ int fx_shift_of(unsigned mask) { return (32 - __clz(mask)) + 32 - FX_TOP; }

// a 2^-d, rounded, halves away from zero: rounding them all up would add the
// same sign to every element, which a transform collects in its zero
// frequency, where the Green's function is largest.  fx_round: d > 0;
// fx_align: d may be negative or beyond 63.
__device__ __forceinline__ long long fx_round(long long a, long long half, int d) { return (a + half + (a >> 63)) >> d; }
__device__ __forceinline__ long long fx_align1(long long a, int d) {
    if (d <= 0) return a << (-d);
    return d > 62 ? 0ll : fx_round(a, (1ll << d) >> 1, d);
}
__device__ __forceinline__ fxc fx_align(fxc a, int d) { return fxc{fx_align1(a.x, d), fx_align1(a.y, d)}; }

// a double as x 2^-s' with the shared exponent chosen so that the largest
// exponent field emax maps below 2^FX_TOP: value = result 2^(fx_exp(emax))
__device__ __forceinline__ int fx_exp(int emax) { return emax - 1022 - FX_TOP; }
__device__ __forceinline__ long long fx_from_double(double d, int emax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int ef = (int)((b >> 52) & 0x7FF), e = ef ? ef : 1;
    const long long m = (long long)((b & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull));
    const long long v = fx_align1(m, emax - e + 53 - FX_TOP);
    return (long long)b < 0 ? -v : v;
}

// x 2^e as the nearest double
__device__ __forceinline__ double fx_to_double(long long x, int e) {
    const long long s = x >> 63;
    unsigned long long a = (unsigned long long)((x ^ s) - s);
    if (a == 0) return 0.0;
    const int sh = __clzll((long long)a) - 1;             // |x| < 2^63: to [2^62, 2^63)
    a <<= sh;
    const int ef = e - sh + 62 + 1023;
    if (ef < 1 || ef > 2045) return ldexp((double)x, e);
    a += 0x1FF + ((a >> 10) & 1);                          // to nearest even; a carry moves into the exponent
    const unsigned long long bits = (a >> 10) + ((unsigned long long)(ef - 1) << 52);
    return __longlong_as_double((long long)(bits | ((unsigned long long)s & 0x8000000000000000ull)));
}
