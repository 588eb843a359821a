// Fixed-point arithmetic of the FP64 pair sums.
//
// This device issues 32 32x32+64-bit integer multiply-adds per clock and SM
// against 1.6 double-precision FMAs (measured), so the FP64 operators run
// their pair terms in 59 to 62-bit fixed point on the integer pipes: more
// significant bits than a double carries, at a fraction of the cost.  (The kernel
// tables are good to 2^-53.7, sigma_4 to 2^-51.9, of a value: fx_table.cu.)  The
// building blocks here are host and device code:
//
//   positions   in units of delta, 2^-ps grid, int64; differences are exact
//   fx_index    v = 1 + |y - x|^2 / delta^2 exactly, normalised; segment and
//               local variable s in [-1, 1) of the kernel tables
//   fx_poly     sigma_i(t) = s_i / rho^p of that segment (degree 7), as a
//               62-bit mantissa and an exponent: smoothed and bare kernels,
//               near and far pairs alike, without erf, exp or a square root
//   fx_dot      dot product of two vectors of 31-bit limbs (to 2^-105 of its
//               range), rounded once to a 61-bit mantissa and an exponent
//   fx_mul      62-bit product of two mantissas
//   fx_shift    mantissa and exponent to fixed point (64 + 32 bits)
//
// Vectors and mantissas are split as h 2^31 + l, 0 <= l < 2^31 (differences of
// vectors |l| < 2^31); mantissas stay below 2^62.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace ssd {

constexpr int kFxSegBits = 6;                   // segments per octave of v: 64
constexpr int kFxSeg = 1 << kFxSegBits;
constexpr int kFxMaxOct = 20;                   // octaves of v = 1 + t
constexpr int kFxEntry = 3;                     // 16-byte words of a table entry
constexpr int kFxBareEntries = 2 * kFxSeg;      // t^(-1/2) over two octaves of t
constexpr int kFxTabEntries = 4 * kFxMaxOct * kFxSeg + kFxBareEntries;
constexpr int kFxEBias = 8;                     // bias of the stored exponent
// extent / delta served: beyond 256 the position grid is coarser than 2^-54
// delta; below 1/16 all terms are small against the bounds that fix the units
constexpr double kFxMinExt = 0.0625, kFxMaxExt = 256.0;

// 32 x 32 + 64 bits: mad.wide.s32 (a x b in full, plus c), as one instruction
FX_HD int64_t fx_mw(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
    int64_t d;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
    return d;
#else
    return (int64_t)a * b + c;
#endif
}
FX_HD int64_t fx_mw(int a, int b) {
#ifdef __CUDA_ARCH__
    int64_t d;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(d) : "r"(a), "r"(b));
    return d;
#else
    return (int64_t)a * b;
#endif
}
FX_HD int fx_hi(int64_t x) { return (int)(x >> 32); }
FX_HD uint32_t fx_shl(uint32_t lo, uint32_t hi, uint32_t s) {   // high word of (hi:lo) << s, s < 32
#ifdef __CUDA_ARCH__
    return __funnelshift_l(lo, hi, s);
#else
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}
FX_HD int fx_clz(uint32_t x) {
#ifdef __CUDA_ARCH__
    return __clz(x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
// leading sign-extension bits: 32 for 0 and -1, else 32 - (significant bits without the sign)
FX_HD int fx_clzs(int x) {
#ifdef __CUDA_ARCH__
    uint32_t r;
    asm("bfind.shiftamt.s32 %0, %1;" : "=r"(r) : "r"(x));
    return (int)(r < 32u ? r : 32u);
#else
    return fx_clz((uint32_t)(x ^ (x >> 31)));
#endif
}

struct FxV { int h[3], l[3]; };                 // vector in limbs

FX_HD void fx_split(int64_t x, int &h, int &l) { h = (int)(x >> 31); l = (int)(x & 0x7fffffff); }

// round(v 2^(bits - e)) of a finite double |v| < 2^e, to nearest
FX_HD int64_t fx_fix(double v, int e, int bits) {
    union { double d; uint64_t u; } c;
    c.d = v;
    const int ex = (int)((c.u >> 52) & 0x7ff);
    const uint64_t m = (c.u & 0xfffffffffffffull) | (ex ? 0x10000000000000ull : 0ull);
    const int sh = (ex ? ex : 1) - 1075 - e + bits;
    uint64_t r;
    if (sh >= 0) r = m << (sh > 63 ? 63 : sh);
    else if (sh < -54) r = 0;
    else r = (m + (1ull << (-sh - 1))) >> (-sh);
    return (c.u >> 63) ? -(int64_t)r : (int64_t)r;
}

struct FxArgSeg { uint32_t idx; int sh, sl; };

// T = |d|^2 from the limbs (|d| < 2^61), v = T + one (one_hi = 2^(60 - 2 L): the
// value 1 in units of T's 2^62), and its segment.  oct0 = (2 + 2 L) 64.  The
// squares of the low limbs enter with 15 bits (within 2^17.6 of w's unit); 2^18
// added to w keeps v >= one where the limbs cancel, at 2^-72 of T's range.
FX_HD FxArgSeg fx_index(const FxV &d, int64_t one_hi, int oct0) {
    const int64_t t2 = fx_mw(d.h[2], d.h[2], fx_mw(d.h[1], d.h[1], fx_mw(d.h[0], d.h[0], one_hi)));
    const int64_t t1 = fx_mw(d.h[2], d.l[2], fx_mw(d.h[1], d.l[1], fx_mw(d.h[0], d.l[0], 1 << 18)));
    const uint32_t q0 = (uint32_t)(d.l[0] >> 16), q1 = (uint32_t)(d.l[1] >> 16), q2 = (uint32_t)(d.l[2] >> 16);
    const int64_t w = t1 + (int64_t)(uint64_t)(q0 * q0 + q1 * q1 + q2 * q2);
    const int64_t v = t2 + (w >> 30);
    const uint32_t vh = (uint32_t)(v >> 32), vl = (uint32_t)v, wl = (uint32_t)w << 2;
    const int lz = fx_clz(vh);
    const uint32_t mh = fx_shl(vl, vh, lz & 31), ml = fx_shl(wl, vl, lz & 31);
    FxArgSeg r;
    r.idx = (uint32_t)(oct0 - lz * kFxSeg) + (mh >> (31 - kFxSegBits));
    r.sh = (int)(fx_shl(ml, mh, kFxSegBits + 1) ^ 0x80000000u);
    r.sl = (int)((ml << kFxSegBits) & 0x7fffffffu);
    return r;
}

struct FxQ { int64_t m; int e; };               // m 2^-e (times a scale fixed by the context)

// c + p s, s = (sh 2^31 + sl) 2^-62, within 1.3 units and unbiased: the two
// truncations below drop 1.25 units on average, which the constant returns
// (sums over thousands of pairs of either sign would show the bias)
FX_HD int64_t fx_muladd(int64_t p, int sh, int sl, int64_t c) {
    const int ph = (int)(p >> 31), pl = (int)p & 0x7fffffff;
    const int64_t x = fx_mw(pl, sh, fx_mw(ph, sl, 0xA0000000ll));
    return fx_mw(ph, sh, fx_mw(fx_hi(x), 2, c));
}

struct FxI4 { int x, y, z, w; };
// kernel factor of a segment: sigma = m 2^-(61 + e), 2^61 <= m < 2^62 near the
// segment's top.  Entry: c0, c1 | c2, c3 (64 bits) | c4, c5, c6, (c7 << 8 | e + bias),
// c4 .. c7 in units of 2^U .. 2^(U-3), U = fx_unit(i) (c4 of sigma_4 needs the larger one)
constexpr int fx_unit(int i) { return i == 3 ? 9 : 7; }
template <int U>
FX_HD FxQ fx_poly(const FxI4 &e0, const FxI4 &e1, const FxI4 &e2, int sh, int sl) {
    const int64_t c0 = ((int64_t)e0.y << 32) | (uint32_t)e0.x, c1 = ((int64_t)e0.w << 32) | (uint32_t)e0.z;
    const int64_t c2 = ((int64_t)e1.y << 32) | (uint32_t)e1.x, c3 = ((int64_t)e1.w << 32) | (uint32_t)e1.z;
    const int p6 = e2.z + fx_hi(fx_mw(e2.w >> 8, sh, 1ll << 31));
    const int p5 = e2.y + fx_hi(fx_mw(p6, sh, 1ll << 31));
    const int p4 = e2.x + fx_hi(fx_mw(p5, sh, 1ll << 31));
    const int64_t p3 = c3 + (fx_mw(p4, sh) >> (31 - U));
    FxQ r;
    r.m = fx_muladd(fx_muladd(fx_muladd(p3, sh, sl, c2), sh, sl, c1), sh, sl, c0);
    r.e = (e2.w & 255) - kFxEBias;
    return r;
}

// a . b = m 2^(62 - e) in units of the product, |m| < 2^62; |a| < 2^61,
// |b| < 2^59, the products of the low limbs to 14 x 15 bits
FX_HD FxQ fx_dot(const FxV &a, const FxV &b) {
    const int64_t a2 = fx_mw(a.h[2], b.h[2], fx_mw(a.h[1], b.h[1], fx_mw(a.h[0], b.h[0])));
    int64_t a1 = fx_mw(a.h[2], b.l[2], fx_mw(a.h[1], b.l[1], fx_mw(a.h[0], b.l[0])));
    a1 = fx_mw(a.l[2], b.h[2], fx_mw(a.l[1], b.h[1], fx_mw(a.l[0], b.h[0], a1)));
    const int a0 = (a.l[0] >> 16) * (b.l[0] >> 17) + (a.l[1] >> 16) * (b.l[1] >> 17) + (a.l[2] >> 16) * (b.l[2] >> 17);
    const int64_t w = a1 + (int64_t)a0 * 4;
    FxQ r;
    r.e = fx_clzs(fx_hi(a2)) - 3;
    r.m = (int64_t)((uint64_t)a2 << r.e) + (w >> (31 - r.e));
    return r;
}

FX_HD int64_t fx_mul(int64_t a, int64_t b) {    // (a b) 2^-62
    return fx_muladd(a, (int)(b >> 31), (int)b & 0x7fffffff, 0);
}

struct FxF { int64_t h; uint32_t l; };          // h + l 2^-32

FX_HD FxF fx_shift(int64_t b, int sh) {         // b 2^-sh, 0 <= sh (clamped to 0 .. 95)
    const int s = sh < 0 ? 0 : (sh > 95 ? 95 : sh);
    const int g = s > 32 ? s - 32 : 0, r = s - g;    // r <= 32
    const int64_t bb = b >> g;
    FxF f;
    f.h = bb >> r;
#ifdef __CUDA_ARCH__
    f.l = __funnelshift_rc(0u, (uint32_t)bb, r);
#else
    f.l = r >= 32 ? (uint32_t)bb : (r == 0 ? 0u : (uint32_t)bb << (32 - r));
#endif
    return f;
}

FX_HD FxF fx_add(const FxF &a, const FxF &b) {
    FxF r;
    r.l = a.l + b.l;
    r.h = a.h + b.h + (r.l < a.l ? 1 : 0);
    return r;
}

// accumulator of sum_j f_j g_j over products of a number f in limbs of 25, 24
// and 24 bits (f.h 2^16 + the top 16 bits of f.l) and a number g in 31-bit
// limbs: one 64-bit sum per product weight, so nothing carries inside the
// loop.  With |f.h| < 2^56.7 and |g| < 2^61, 128 terms stay below 2^63.
struct FxMac { int64_t h, m1, m2, l1, l2; };

struct FxB { int b2, b1, b0; };
FX_HD FxB fx_limbs(const FxF &f) {              // to nearest: a truncated term would bias the sum
    const uint32_t l = f.l + 0x8000u;
    const int64_t h = f.h + (l < 0x8000u ? 1 : 0);
    FxB b;
    b.b2 = (int)(h >> 32);
    b.b1 = (int)((uint32_t)h >> 8);
    b.b0 = (int)fx_shl(l, (uint32_t)h, 16) & 0xffffff;
    return b;
}
FX_HD void fx_mac(FxMac &a, const FxB &b, int gh, int gl) {
    a.h = fx_mw(b.b2, gh, a.h);
    a.m1 = fx_mw(b.b1, gh, a.m1);
    a.m2 = fx_mw(b.b2, gl, a.m2);
    a.l1 = fx_mw(b.b0, gh, a.l1);
    a.l2 = fx_mw(b.b1, gl, a.l2);
}
// the sum is h 2^24 + fx_low in units of 2^55 of f's and g's last places
FX_HD int64_t fx_low(const FxMac &a) {
    const int64_t l = a.l1 + (a.l2 >> 7);
    return a.m1 + (a.m2 >> 7) + (l >> 24);
}
FX_HD double fx_value(const FxMac &a) { return (double)a.h * 16777216.0 + (double)fx_low(a); }

// Kernel tables of sigma_1 .. sigma_4 on v in [1, 2^kFxMaxOct), then t^(-1/2) on
// t in [1, 4): host array of kFxTabEntries entries, built once per process
// (fx_table.cu); NULL without the memory.
const FxI4 *fx_table_host();

}  // namespace ssd
