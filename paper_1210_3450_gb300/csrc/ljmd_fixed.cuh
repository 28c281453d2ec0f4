// Pair arithmetic of the FP64 form in 64-bit fixed point.
//
// GB300's FP64 pipe issues one warp instruction per 64 cycles of a scheduler, its
// integer multipliers one per 2-4, so the 17 FP64 instructions of a pair (about 1,090
// cycles per warp) cost several times what the same arithmetic costs in integers.
// Here a pair's force factor comes from products of 64-bit fixed-point numbers, each
// formed from 32 x 32 -> 64-bit multiply-adds of its halves, and the sums are kept as
// 96-bit integers: additions are exact, so a force does not depend on the order in
// which its pairs are added. No factor is rounded more coarsely than in FP64, at any
// distance in the range: against 113-bit arithmetic it errs (rms, relative to its 24 r^-8)
// by 0.06 to 0.8e-16 beyond r = 1.2 and by up to 1.3e-16 below, where the FP64 pipe's errs by
// 0.8 to 3.4e-16 and by up to 1.1e-15 (cutoffs 2.5 and 3.99), with a mean below 2e-17.
//
// Formats (value = integer x unit):
//   position, separation  unit 2^-60, modulo 2^64 (16 length units; a separation
//                         below 8 is recovered exactly from two wrapped positions,
//                         and an FP64 position of 2^-8 or more is held exactly)
//   r^2                   2^-56   (r^2 < 16)
//   y = 1 / r^2           2^-63   (r^2 >= kFixR2Min = 0.84: y < 1.1905)
//   y^2, y^3, y^4         2^-62, 2^-61, 2^-92 (96 bits: y^4 falls to 2^-16 at r = 4)
//   g / 24                2^-88   (96 bits; |g / 24| < 4.77)
//   force sums / 24       2^-84   (96 bits; 468 pairs of the largest force, 4.37,
//                         reach their range)
// Pairs closer than sqrt(0.84) take the FP64 pipe, for lists longer than kFixMaxList those
// closer than 1 (beyond it a force / 24 is below 1.081: 1,895 pairs reach the sums' range),
// for lists longer than kFixMaxLong all (fix_limit).
// Separations of kFixMaxSep and more may come out of the wrapped differences as shorter
// ones (and r^2 of 128 and more as a negative number), so a loop that hands every listed
// pair on, and not only those that passed a test on the shadows, must know that no listed
// pair comes that far apart.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

namespace ljmd {

constexpr int kFixMaxList = 448;                                // longest list summed in 96 bits ...
constexpr int kFixMaxLong = 1880;                               // ... without pairs closer than 1
constexpr unsigned kFixR2Min = 14092862u;                      // 0.84 in units of 2^-24 (r^2's high word)
constexpr double kFixMaxRc = 3.99;                              // r^2 < 16
constexpr double kFixMaxSep = 7.9;                              // separations below 8, r^2 < 128

// A number split into a signed high and a signed low half (the low half rounded to
// nearest): products of halves are signed 32 x 32 -> 64. fix_split takes the number
// plus kFixBias, so that the rounding costs no addition where the bias can be folded
// into a constant or an operand prepared once.
constexpr long long kFixBias = 0x80000000ll;
struct Fix2 {
  int h, l;
};
// The same with a third, signed part 2^-32 below.
struct Fix3 {
  int h, l, m;
};
// c2 / 3 in units of 2^-88 plus the biases of both lower parts.
struct FixC2 {
  long long hi;
  unsigned lo;
};
static __device__ __forceinline__ Fix2 fix_split(long long biased) {
  Fix2 s;
  s.l = (int)((unsigned)biased + 0x80000000u);
  s.h = (int)(biased >> 32);
  return s;
}
// FP64 to position units, rounded to nearest (integer operations only; modulo 2^64).
static __device__ __forceinline__ long long to_fix(double x) {
  const long long b = __double_as_longlong(x);
  const int sh = (int)((b >> 52) & 0x7FF) - (1075 - 60);
  const unsigned long long m = ((unsigned long long)b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  unsigned long long r;
  if (sh >= 0) r = sh < 64 ? m << sh : 0ull;
  else r = sh >= -54 ? ((m >> (-sh - 1)) + 1ull) >> 1 : 0ull;
  return b < 0 ? -(long long)r : (long long)r;
}

// The multiply-add chains below are written out: from the same sums in C++ the compiler
// makes 1.5 times the multiplier work (a 32 x 32 -> 64-bit multiply-add holds the
// multiplier for 4 cycles, four times a float one, and is what bounds the pair).

// r^2 of a separation (units 2^-56; the products of two low halves are below the unit).
// The constant is the mean of what is cut off, which with that of fix_rcp would leave every
// 1 / r^2 too large by 2e-17, and a virial of many pairs by what single ones average out.
static __device__ __forceinline__ unsigned long long fix_r2(const Fix2& x, const Fix2& y, const Fix2& z) {
  unsigned long long r;
  asm("{\n\t"
      ".reg .s64 s;\n\t"
      "mad.wide.s32 s, %1, %2, 0x60000000;\n\t"
      "mad.wide.s32 s, %3, %4, s;\n\t"
      "mad.wide.s32 s, %5, %6, s;\n\t"
      "shr.s64 s, s, 31;\n\t"
      "mad.wide.s32 s, %1, %1, s;\n\t"
      "mad.wide.s32 s, %3, %3, s;\n\t"
      "mad.wide.s32 %0, %5, %5, s;\n\t"
      "}"
      : "=l"(r)
      : "r"(x.h), "r"(x.l), "r"(y.h), "r"(y.l), "r"(z.h), "r"(z.l));
  return r;
}

// 1 / r^2 from a hardware float estimate and two Newton steps on exact integer
// residuals r^2 y - 1 (only their low 32 bits are formed: they are small). The
// estimate errs by less than 2^-21, the first step leaves 2^-27, the last a relative
// error near 2^-55.
static __device__ __forceinline__ unsigned long long fix_rcp(unsigned long long r2) {
  const unsigned rh = (unsigned)(r2 >> 32), rl = (unsigned)r2;
  float yf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(__uint2float_rn(rh)));
  const unsigned y0 = __float2uint_rn(yf * 4503599627370496.0f);            // 2^52: unit 2^-28
  const int e0 = (int)(rh * y0 + __umulhi(rl, y0));                         // unit 2^-52
  const unsigned y1 = (y0 << 3) - (unsigned)(__mulhi((int)y0, e0) >> 17);   // unit 2^-31
  const unsigned ry = (unsigned)(((unsigned long long)rl * y1 + 0x80000000ull) >> 32);
  const int e1 = (int)(0u - (rh * y1 + ry));                                // unit 2^-55
  unsigned long long y;                                                     // y1 + y1 e1
  asm("{\n\t"
      ".reg .s64 c;\n\t"
      ".reg .u32 c0, c1;\n\t"
      "mul.wide.s32 c, %2, %3;\n\t"  // unit 2^-85
      "shr.s64 c, c, 22;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "add.u32 c1, c1, %1;\n\t"
      "mov.b64 %0, {c0, c1};\n\t"
      "}"
      : "=l"(y)
      : "r"(y1), "r"((int)(y1 >> 1)), "r"(e1));
  return y;
}

// g / 24 = y^4 (1 - 2 y^3) + c2 / 3 (g: the factor 24 r^-8 - 48 r^-14 + 8 c2). With
// y < 1.1905 the cross terms of y y^2 stay below 2^64; y^2 is rounded (the constant holds
// the mean of the dropped square of the low half as well), and y^4 and the products keep
// what lies below the second half, without which pairs beyond r = 1.6 would be rounded
// more coarsely than in FP64 (5e-15 of 24 r^-8 at 2.4, 4.5e-13 at 3.9). The six products
// more (three here, one per sum) cost 0.09 ms of a pass over 2,048,000 particles (1.01 ms).
static __device__ __forceinline__ Fix3 fix_force_factor(unsigned long long y, const FixC2& c2) {
  Fix3 g;
  asm("{\n\t"
      ".reg .u64 c, p;\n\t"
      ".reg .s64 d, t;\n\t"
      ".reg .u32 y0, y1, a0, a1, b0, b1, c0, c1, z;\n\t"
      ".reg .s32 wh, wl, qh, ql, qm, d0, d1, sg;\n\t"
      "mov.b64 {y0, y1}, %3;\n\t"
      "mad.wide.u32 c, y1, y0, 0x6AAAAAAA;\n\t"  // y^2 (unit 2^-62)
      "shr.u64 c, c, 31;\n\t"
      "mad.wide.u32 p, y1, y1, c;\n\t"
      "mov.b64 {a0, a1}, p;\n\t"
      "mul.wide.u32 c, y1, a0;\n\t"            // y^3 (unit 2^-61)
      "mad.wide.u32 c, y0, a1, c;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "mov.u32 z, 0;\n\t"
      "mov.b64 c, {c1, z};\n\t"
      "mad.wide.u32 c, y1, a1, c;\n\t"
      "mov.b64 {b0, b1}, c;\n\t"
      "sub.cc.u32 b0, 0x80000000, b0;\n\t"     // w = 1 - 2 y^3 (unit 2^-60), split
      "subc.u32 wh, 0x10000000, b1;\n\t"
      "add.u32 wl, b0, 0x80000000;\n\t"
      "mul.hi.u32 c0, a0, a0;\n\t"             // q = y^4 (unit 2^-92), split: half the cross
      "shr.u32 c0, c0, 1;\n\t"                 // terms (unit 2^-91) with both biases
      "add.u32 c0, c0, 0x40000000;\n\t"
      "mov.u32 c1, 0x40000000;\n\t"
      "mov.b64 c, {c0, c1};\n\t"
      "mad.wide.u32 c, a1, a0, c;\n\t"
      "mov.b64 {c0, c1}, c;\n\t"
      "mad.lo.u32 qm, c0, 2, 0x80000000;\n\t"
      "shr.u64 c, c, 31;\n\t"
      "mad.wide.u32 p, a1, a1, c;\n\t"
      "mov.b64 {b0, qh}, p;\n\t"
      "add.u32 ql, b0, 0x80000000;\n\t"
      "mul.wide.s32 d, ql, wl;\n\t"            // q w: the parts of 2^-120,
      "mad.wide.s32 d, qm, wh, d;\n\t"
      "shr.s64 d, d, 32;\n\t"
      "mad.wide.s32 d, wl, qh, d;\n\t"         // 2^-88
      "mad.wide.s32 d, wh, ql, d;\n\t"
      "mad.wide.s32 t, wh, qh, %4;\n\t"        // and 2^-56
      "mov.b64 {d0, d1}, d;\n\t"
      "shr.s32 sg, d1, 31;\n\t"
      "mov.b64 {c0, c1}, t;\n\t"
      "add.cc.u32 d0, d0, %5;\n\t"
      "addc.cc.u32 c0, c0, d1;\n\t"
      "addc.u32 %0, c1, sg;\n\t"
      "add.u32 %1, c0, 0x80000000;\n\t"
      "add.u32 %2, d0, 0x80000000;\n\t"
      "}"
      : "=r"(g.h), "=r"(g.l), "=r"(g.m)
      : "l"(y), "l"(c2.hi), "r"(c2.lo));
  return g;
}

// A 96-bit number: 64 bits and the 32 below.
struct Fix96 {
  unsigned long long hi;
  unsigned lo;
};
// y^3 in units of 2^-93, and the square of an a < 2^31.4 / 2^32 of its range (a in units of
// 2^-u: units of 2^(32 - 2 u); y^3's high part in 2^-61 gives y^6 in 2^-90).
static __device__ __forceinline__ Fix96 fix_y3(unsigned long long y) {
  Fix96 r;
  asm("{\n\t"
      ".reg .u64 c, p;\n\t"
      ".reg .u32 y0, y1, a0, a1, c1, z;\n\t"
      "mov.b64 {y0, y1}, %2;\n\t"
      "mad.wide.u32 c, y1, y0, 0x6AAAAAAA;\n\t"  // y^2 (unit 2^-62), rounded as in fix_force_factor
      "shr.u64 c, c, 31;\n\t"
      "mad.wide.u32 p, y1, y1, c;\n\t"
      "mov.b64 {a0, a1}, p;\n\t"
      "mov.u32 z, 0;\n\t"
      "mul.hi.u32 c1, y0, a0;\n\t"
      "mov.b64 c, {c1, z};\n\t"
      "mad.wide.u32 c, y1, a0, c;\n\t"
      "mad.wide.u32 c, y0, a1, c;\n\t"
      "mov.b64 {%1, c1}, c;\n\t"
      "mov.b64 c, {c1, z};\n\t"
      "mad.wide.u32 %0, y1, a1, c;\n\t"
      "}"
      : "=l"(r.hi), "=&r"(r.lo)
      : "l"(y));
  return r;
}
static __device__ __forceinline__ Fix96 fix_sqr(unsigned long long a) {
  Fix96 r;
  asm("{\n\t"
      ".reg .u64 c;\n\t"
      ".reg .u32 a0, a1, c0, z;\n\t"
      "mov.b64 {a0, a1}, %2;\n\t"
      "mov.u32 z, 0;\n\t"
      "mul.hi.u32 c0, a0, a0;\n\t"
      "shr.u32 c0, c0, 1;\n\t"
      "mov.b64 c, {c0, z};\n\t"
      "mad.wide.u32 c, a1, a0, c;\n\t"  // half the cross terms
      "mov.b64 {c0, z}, c;\n\t"
      "shl.b32 %1, c0, 1;\n\t"
      "shr.u64 c, c, 31;\n\t"
      "mad.wide.u32 %0, a1, a1, c;\n\t"
      "}"
      : "=l"(r.hi), "=&r"(r.lo)
      : "l"(a));
  return r;
}

// Exact sum of 64- or 96-bit non-negative terms in 128 bits.
struct FixAcc {
  unsigned long long lo = 0ull, hi = 0ull;
  __device__ __forceinline__ void add(unsigned long long v) {
    lo += v;
    hi += lo < v ? 1ull : 0ull;
  }
  __device__ __forceinline__ void add(const Fix96& v) {
    const unsigned long long l = (v.hi << 32) | v.lo;
    lo += l;
    hi += (v.hi >> 32) + (lo < l ? 1ull : 0ull);
  }
  // Adds the sum of the lane o away (all 32 lanes of the warp call it).
  __device__ __forceinline__ void join(int o) {
    const unsigned long long l = __shfl_xor_sync(0xffffffffu, lo, o), h = __shfl_xor_sync(0xffffffffu, hi, o);
    lo += l;
    hi += h + (lo < l ? 1ull : 0ull);
  }
  // The sum x 2^-unit as FP64 (rounded to nearest, halves up; unit at most 900), by
  // integer operations.
  __device__ __forceinline__ double value(int unit) const {
    if ((lo | hi) == 0ull) return 0.0;
    const int z = hi ? __clzll((long long)hi) : 64 + __clzll((long long)lo);
    // the top 64 bits, normalised: sum = m 2^(64 - z)
    const unsigned long long m = z == 0 ? hi : z < 64 ? (hi << z) | (lo >> (64 - z)) : lo << (z - 64);
    const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);  // 53 bits; may round up to 2^53
    const int ex = 1023 + 52 + 11 + 64 - z - unit;
    return __longlong_as_double((long long)(((unsigned long long)(ex - 1) << 52) + r));
  }
};

// Exact sum of FP64 squares in 256 bits, units of 2^-160: squares of 2^-108 and more (a
// velocity component of 5e-17) keep all their bits, and 2^28 of the largest stay in range.
// Squares of 2^64 and more, and what is not finite, are only kept as the largest of them,
// which then stands for the sum.
struct SquareSum {
  unsigned long long w[4] = {0ull, 0ull, 0ull, 0ull};
  unsigned long long over = 0ull;
  static constexpr unsigned long long kOver = (1023ull + 64ull) << 52;  // 2^64
  __device__ __forceinline__ void add_words(unsigned long long a, unsigned long long b, unsigned long long c,
                                            unsigned long long d) {
    asm("add.cc.u64 %0, %0, %4;\n\t"
        "addc.cc.u64 %1, %1, %5;\n\t"
        "addc.cc.u64 %2, %2, %6;\n\t"
        "addc.u64 %3, %3, %7;"
        : "+l"(w[0]), "+l"(w[1]), "+l"(w[2]), "+l"(w[3])
        : "l"(a), "l"(b), "l"(c), "l"(d));
  }
  __device__ __forceinline__ void add(double v) {  // v: a square
    const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFull;
    if (b >= kOver) {
      over = b > over ? b : over;
      return;
    }
    const int sh = (int)(b >> 52) - (1075 - 160);
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int k = sh >> 6, r = sh & 63;
    unsigned long long lo = m << r, hi = r ? m >> (64 - r) : 0ull;
    if (sh < 0) {
      lo = sh > -64 ? m >> -sh : 0ull;
      hi = 0ull;
    }
    add_words(k <= 0 ? lo : 0ull, k == 1 ? lo : (k == 0 ? hi : 0ull), k == 2 ? lo : (k == 1 ? hi : 0ull),
              k == 2 ? hi : 0ull);
  }
  // Adds the sum of the lane o away (all 32 lanes of the warp call it).
  __device__ __forceinline__ void join(int o) {
    unsigned long long y[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) y[m] = __shfl_xor_sync(0xffffffffu, w[m], o);
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, over, o);
    add_words(y[0], y[1], y[2], y[3]);
    over = v > over ? v : over;
  }
  // Half the sum as FP64 (rounded to nearest).
  __device__ __forceinline__ double half() const {
    if (over) return 0.5 * __longlong_as_double((long long)over);
    FixAcc s;  // the top word that is not zero, and the next
    s.hi = w[3];
    s.lo = w[2];
    int unit = 161 - 128;
#pragma unroll
    for (int k = 2; k >= 0; --k) {  // (no index known only at run time: the words stay in registers)
      if (s.hi != 0ull) break;
      s.hi = w[k];
      s.lo = k > 0 ? w[k - 1] : 0ull;
      unit += 64;
    }
    return s.value(unit);
  }
};

// 96-bit sum of products g d (units 2^-84: g 2^-88, d 2^-60).
struct FixSum {
  unsigned lo = 0u;   // units of 2^-84
  long long hi = 0;   // units of 2^-52
  __device__ __forceinline__ void add(const Fix3& g, const Fix2& d) {
    asm("{\n\t"
        ".reg .s32 sg, c0, c1, h0, h1;\n\t"
        ".reg .s64 c;\n\t"
        "mul.wide.s32 c, %3, %6;\n\t"      // 2^-116
        "mad.wide.s32 c, %4, %5, c;\n\t"
        "shr.s64 c, c, 32;\n\t"
        "mad.wide.s32 c, %2, %6, c;\n\t"   // 2^-84
        "mad.wide.s32 c, %3, %5, c;\n\t"
        "mad.wide.s32 %1, %2, %5, %1;\n\t" // 2^-52
        "mov.b64 {c0, c1}, c;\n\t"
        "shr.s32 sg, c1, 31;\n\t"
        "mov.b64 {h0, h1}, %1;\n\t"
        "add.cc.u32 %0, %0, c0;\n\t"
        "addc.cc.u32 h0, h0, c1;\n\t"
        "addc.u32 h1, h1, sg;\n\t"
        "mov.b64 %1, {h0, h1};\n\t"
        "}"
        : "+r"(lo), "+l"(hi)
        : "r"(g.h), "r"(g.l), "r"(g.m), "r"(d.h), "r"(d.l));
  }
  // Adds the sum of the lane o away (all 32 lanes of the warp call it).
  __device__ __forceinline__ void join(int o) {
    const unsigned l = __shfl_xor_sync(0xffffffffu, lo, o);
    const long long h = __shfl_xor_sync(0xffffffffu, hi, o);
    const unsigned t = lo + l;
    hi += h + (t < l ? 1 : 0);
    lo = t;
  }
  // 24 x the sum as FP64, formed with integer operations (the FP64 pipe's conversions
  // would cost more than the pairs of three rounds).
  __device__ __forceinline__ double value24() const {
    unsigned long long h = (unsigned long long)hi;
    unsigned l = lo;
    if (hi < 0) {  // magnitude of the 96-bit sum
      l = 0u - l;
      h = ~h + (l == 0u ? 1ull : 0ull);
    }
    if (h == 0ull && l == 0u) return 0.0;
    const int z = h ? __clzll((long long)h) : 64 + __clz((int)l);  // leading zeros of 96 bits
    unsigned long long m;                                         // top 64 bits, normalised
    if (z == 0) m = h;
    else if (z < 32) m = (h << z) | (l >> (32 - z));
    else if (z < 64) m = (h << z) | ((unsigned long long)l << (z - 32));
    else m = (unsigned long long)l << (z - 32);
    m = (m >> 3) * 3ull;                  // in [3, 6) x 2^60: value m 2^(-84 + 32 - z + 3 + 3)
    const int up = (int)(m >> 62);        // 1: m in [2^62, 2^63)
    const int k = up ? 10 : 9;            // m >> k has 53 bits
    m = (m + (1ull << (k - 1))) >> k;     // may round up to 2^53: the addition below carries
    const int ex = 1023 + 52 + k - 46 - z;
    const unsigned long long b = ((unsigned long long)(ex - 1) << 52) + m;
    return __longlong_as_double((long long)(b | (hi < 0 ? 0x8000000000000000ull : 0ull)));
  }
};

// Separation qj - qi plus the periodic image `code` (two bits per axis: 1 adds L, 2
// subtracts it), split; qi comes minus kFixBias.
static __device__ __forceinline__ void fix_separation(const longlong4_32a& qi, const longlong4_32a& qj, unsigned code,
                                                      long long L, Fix2& fx, Fix2& fy, Fix2& fz) {
  long long dx = qj.x - qi.x, dy = qj.y - qi.y, dz = qj.z - qi.z;
  if (code) {
    dx += (code & 3u) == 1u ? L : ((code & 3u) == 2u ? -L : 0);
    dy += (code & 12u) == 4u ? L : ((code & 12u) == 8u ? -L : 0);
    dz += (code & 48u) == 16u ? L : ((code & 48u) == 32u ? -L : 0);
  }
  fx = fix_split(dx);
  fy = fix_split(dy);
  fz = fix_split(dz);
}
static __device__ __forceinline__ unsigned long long fix_separation2(const longlong4_32a& qi, const longlong4_32a& qj,
                                                                     unsigned code, long long L) {
  Fix2 fx, fy, fz;
  fix_separation(qi, qj, code, L, fx, fy, fz);
  return fix_r2(fx, fy, fz);
}

// The squared distance (its high word) from which a particle's pairs are taken in fixed
// point.
static __device__ __forceinline__ unsigned fix_limit(int listed) {
  return listed <= kFixMaxList ? kFixR2Min : listed <= kFixMaxLong ? 1u << 24 : ~0u;
}

// One pair: where r < rc, its force is added to the sums (qi, code, L as above; rc2 in
// units of 2^-56, c2 as for fix_force_factor). Returns true, with nothing added, for a pair closer than the range (the FP64 pipe takes it).
static __device__ __forceinline__ bool fix_pair(const longlong4_32a& qi, const longlong4_32a& qj, unsigned code,
                                                long long L, long long rc2, const FixC2& c2, FixSum& sx, FixSum& sy,
                                                FixSum& sz, unsigned limit = kFixR2Min) {
  Fix2 fx, fy, fz;
  fix_separation(qi, qj, code, L, fx, fy, fz);
  const unsigned long long r2 = fix_r2(fx, fy, fz);
  const bool far = (unsigned)(r2 >> 32) >= limit;
  if (far & ((long long)(r2 - (unsigned long long)rc2) < 0)) {
    const Fix3 g = fix_force_factor(fix_rcp(r2), c2);
    sx.add(g, fx);
    sy.add(g, fy);
    sz.add(g, fz);
  }
  return !far;
}

// Whether pairs listed within rc + skin may come kFixMaxSep apart before the list is built
// anew (either rule rebuilds once two particles may have moved `skin` against each other).
static inline bool fix_wide(double rc, double skin) { return !(rc + 2.0 * skin <= kFixMaxSep); }

// x >= 2^-8 in position units (host; exact).
static inline long long fix_host(double x) {
  int e = 0;
  const unsigned long long m = (unsigned long long)std::ldexp(std::frexp(x, &e), 53);  // x = m 2^(e - 53)
  const int sh = e - 53 + 60;
  return (long long)(sh >= 64 ? 0ull : sh >= 0 ? m << sh : m >> -sh);
}

// c2 / 3 for fix_force_factor (host; rounded to nearest). Cutoffs below the range of the
// pairs, whose c2 may not fit, have no pair that takes it.
static inline FixC2 fix_c2(double c2, double rc2) {
  __int128 v = 0;
  if (rc2 > 0.83) {
    int e = 0;
    const long long m = (long long)std::ldexp(std::frexp(c2, &e), 53);  // c2 = m 2^(e - 53)
    const int sh = e - 53 + 88;
    if (sh >= 0) {
      v = (__int128)m * ((__int128)1 << sh) + 1;
      v = (v - (v < 0 ? (v % 3 + 3) % 3 : v % 3)) / 3;  // floor((m 2^sh + 1) / 3)
    }
  }
  v += (__int128)kFixBias + ((__int128)kFixBias << 32);
  return FixC2{(long long)(v >> 32), (unsigned)v};
}

}  // namespace ljmd
