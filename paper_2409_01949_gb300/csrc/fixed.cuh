// Fixed-point arithmetic of the FP64-accurate feature evaluation.
//
// GB300 issues an FP64 warp instruction over 64 cycles of a sub-partition, a
// 32 x 32 + 64 bit integer multiply-add over a few, so a tanh in FP64 (about
// 50 such instructions with its argument) costs about 3000 cycles a warp and
// the integer form below about 200.  Every quantity of a feature is bounded
// (|x| <= 1 in a support, |w|, |b| <= the weight scale, |tanh| <= 1), so 62-bit
// fixed point loses nothing: the absolute error of the tanh is below 2^-57
// (2^-60 in the mean square), its argument's below 2^-59 times the weight scale (rounded up to a power of
// two), against 2^-54 and 2^-53 times the argument's terms in FP64.
//
// A value v is held as v = hi 2^31 + lo, 0 <= lo < 2^31, so that every partial
// product is one signed multiply-add; the lo x lo product (less than one unit
// after the shift, a quarter in the mean) is left out.
#pragma once

#include <math.h>
#include <stdint.h>

#if defined(__CUDACC__)
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN inline
struct int4 { int x, y, z, w; };
struct int2 { int x, y; };
#endif

namespace fx {

struct Val {
  int hi, lo;
};

// a b + c of 32-bit factors, one instruction on the device
FX_FN int64_t mad(int a, int b, int64_t c) {
#if defined(__CUDA_ARCH__)
  int64_t d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (int64_t)a * b + c;
#endif
}

FX_FN Val split(int64_t v) { return {(int)(v >> 31), (int)(v & 0x7fffffff)}; }

// c + a b / 2^62, to the nearest unit but for the lo x lo product: rounding down
// would put half a unit of the same sign on every one of the thousands of terms of
// a sum.  The quarter unit that the left-out product takes in the mean has one sign
// too: sums hold their terms in units well below their own last place.
FX_FN int64_t mul_add(Val a, Val b, int64_t c) {
  const int64_t cross = mad(a.hi, b.lo, mad(a.lo, b.hi, 1 << 30));
  return mad(a.hi, b.hi, c) + (cross >> 31);
}

// a b / 2^62, to the nearest unit, a half to either side by `odd`: where b has few
// bits halves are common, and a sum that rounds half of its terms each way has no
// bias
FX_FN int64_t mul_exact(Val a, Val b, int odd) {
  const int64_t low = (int64_t)(((uint64_t)(uint32_t)a.lo * (uint32_t)b.lo) >> 31);
  const int64_t cross = mad(a.hi, b.lo, mad(a.lo, b.hi, (1 << 30) - odd + low));
  return mad(a.hi, b.hi, cross >> 31);
}

// v / 2^n (n >= 0), rounded down
FX_FN int64_t down(int64_t v, int n) { return v >> (n < 63 ? n : 63); }

// The weight scale a as a power of two: weights and biases are at most
// 2^wexp(a) in magnitude.  Fixed point is used for kMinExp <= wexp <= kMaxExp:
// below, FP64's error (relative to its terms) is the smaller one; above, the
// interval index would run out of bits.
constexpr int kMinExp = -4, kMaxExp = 16;

// wexp(a), the least e with a <= 2^e (a > 0)
FX_FN int weight_exp(double a) {
  int e;
  const double m = frexp(a, &e);
  return m == 0.5 ? e - 1 : e;
}

// A feature's argument s = w0 x0 + w1 x1 + b with w in units of 2^(wexp - 61),
// x in units of 2^-61 and b in units of 2^(wexp - 60); s has b's unit and at
// most three terms, so it stays below 2^62.
FX_FN int64_t argument(Val w0, Val x0, Val w1, Val x1, int64_t b, bool two) {
  int64_t cross = mad(w0.hi, x0.lo, mad(w0.lo, x0.hi, 1 << 30));
  int64_t s = mad(w0.hi, x0.hi, b);
  if (two) {
    cross = mad(w1.hi, x1.lo, mad(w1.lo, x1.hi, cross));
    s = mad(w1.hi, x1.hi, s);
  }
  return s + (cross >> 31);
}

// tanh(s) in units of 2^-61, s in units of 2^(wexp - 60); `shift` = 54 - wexp is
// the width of an interval of 1/64.  tab holds `rows` rows of the table
// (tanh_table.py), the last of them for everything past the others.
FX_FN int64_t tanh61(int64_t s, int shift, const int4* tab, int rows) {
  const uint64_t m = (uint64_t)(s < 0 ? -s : s);
  // |s| < 2^62 and 38 <= shift <= 58: the interval is in the upper word
  const uint32_t mh = (uint32_t)(m >> 32), ml = (uint32_t)m;
  const uint32_t ju = mh >> (shift - 32);
  const int j = ju < (uint32_t)rows ? (int)ju : rows - 1;
  // the place in the interval as r in [-1, 1), units of 2^-62: the bits below
  // `shift`, from bit 62 down, less 2^62
  const int up = 63 - shift;
  const uint32_t vl = ml << up;
  const uint32_t vh = (((mh << up) | (ml >> (32 - up))) & 0x7fffffffu) - 0x40000000u;
  const Val r = {(int)((vh << 1) | (vl >> 31)), (int)(vl & 0x7fffffffu)};
  const int4 a = tab[3 * j], b = tab[3 * j + 1], d = tab[3 * j + 2];
  auto word = [](int lo, int hi) { return (int64_t)(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); };
  // c4 and up fit 32 bits, and the high half of r is enough for them
  int t = (int)(((int64_t)d.z * r.hi) >> 31) + d.y;                // c6 r + c5
  t = (int)(((int64_t)t * r.hi) >> 31) + d.x;                      // ... r + c4
  int64_t v = (((int64_t)t * r.hi) >> 31) + word(b.z, b.w);        // ... r + c3
  v = mul_add(split(v), r, word(b.x, b.y));
  v = mul_add(split(v), r, word(a.z, a.w));
  v = mul_add(split(v), r, word(a.x, a.y));
  return s < 0 ? -v : v;
}

constexpr int kTanhRows = 64 * 22 + 1;   // tanh_table.py: 64 a unit up to 22, and the closing row

// rows that arguments up to (dim + 1) 2^wexp reach, the closing row included
FX_FN int tanh_rows(int dim, int wexp) {
  const int64_t n = wexp >= 0 ? (int64_t)(dim + 1) * 64 << wexp : ((int64_t)(dim + 1) * 64 >> -wexp) + 1;
  return n + 1 < kTanhRows ? (int)n + 1 : kTanhRows;
}

}  // namespace fx
