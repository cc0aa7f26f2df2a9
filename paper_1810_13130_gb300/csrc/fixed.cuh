// Fixed-point contractions with a float tail: the element operator in integer arithmetic.
//
// GB300 runs 2 FP64 operations per clock and SM; its integer pipe multiplies 32 x 32 bits
// into 64 sixteen times as fast, its FP32 pipe is 64 times as fast.  So a contraction is
// carried out in 55-bit integers with an FP32 tail below them: faster than the FP64 pipe
// and at least as accurate.  All values of an element's part (real or imaginary) of one
// orbital share a power of two:
//   value x = (V + f) 2^E,    V a 64-bit integer, |V| < 2^55, f a float of a few units;
//   coefficient c = C 2^-63,  C = h 2^32 + l, |c| < 1, l signed.
// With V = vh 2^32 + vl (vl signed; taken from V + 2^31, whose high word is vh)
//   C V 2^-64 = h vh + (h vl + l vh) 2^-32 + (l 2^-32)(vl 2^-32),
// half the product: every contraction halves the unit's exponent count by one (E grows by
// 1), which keeps h in 32 bits.  A dot product sums h vh and mid = sum (h vl + l vh)
// exactly in 64 bits (three wide multiply-adds per term); the integer part is
// sum h vh + (mid >> 32), rounded to nearest.  What is left goes to the tail in FP32: the
// fraction of mid 2^-32, sum (c / 2) f and the low products, each to about 2^-23 of a unit.
// What a stage loses is fixed in units, so the values have to fill their 55 bits: a vector
// with one large entry loses three bits per contraction (the element operator was off by up
// to 4e-15 at p = 8), and is raised once on the way (fx_raise).  Relative error of the whole
// element operator in the 2-norm, p = 1..8, against extended precision, over dense vectors,
// ones that fall off by up to 69 e-folds along the element and ones with a single large
// entry, with mild and with steep potentials: 2.3e-17 .. 1.6e-16 (little more than the rounding
// of the result), FP64 contractions 6.8e-17 .. 7.7e-15, and for every vector at most 0.75
// times theirs.
//
// Range: with row sums sum |c| = R, |sum h vl| <= R 2^62 and |sum l vh| <= 5 2^31 2^(56 - 32)
// R^2, so |mid| < 2^63 for R <= 1.54, the largest row sum (the transposed interpolation of
// p = 2); the integer parts keep |V| < 2^55 / 2 * R.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

namespace tdks {

struct FxC {      // coefficient c 2^63 = h 2^32 + l, and c / 2, l 2^-32 as floats
  int h, l;
  float c, cl;
};
struct FxL {      // the limbs alone
  int h, l;
};

constexpr int kFxBits = 55;   // |V| < 2^55 on input

// c 2^63 -> limbs (|c| < 1)
__host__ __device__ __forceinline__ FxC fx_coef(long long c) {
  const long long h = (c >> 32) + ((c >> 31) & 1);
  const int l = (int)(unsigned)c;
  return FxC{(int)h, l, (float)c * 0x1p-64f, (float)l * 0x1p-32f};
}

__host__ __device__ __forceinline__ float fx_bits_float(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  __builtin_memcpy(&f, &b, 4);
  return f;
#endif
}
__host__ __device__ __forceinline__ unsigned fx_float_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  unsigned b;
  __builtin_memcpy(&b, &f, 4);
  return b;
#endif
}
// 1 + w 2^-32, cut to 23 bits
__host__ __device__ __forceinline__ float fx_frac1(unsigned w) { return fx_bits_float((w >> 9) + 0x3f800000u); }

// operand: V = h 2^32 + l (l signed), its tail f, and g = 1.5 + l 2^-32
struct FxV {
  int h, l;
  float f, g;
};
constexpr long long kFxHalf = 1ll << 31;
// from V + 2^31
__host__ __device__ __forceinline__ FxV fx_operand(long long vb, float f) {
  const unsigned w = (unsigned)vb;
  return FxV{(int)(vb >> 32), (int)(w ^ 0x80000000u), f, fx_frac1(w)};
}
// a b + c; as one instruction also where b is known to be non-negative (the compiler would
// extend such an operand without sign and multiply 64 x 64 bits)
__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)a * (long long)b + c;
#endif
}

// A dot product: term() for every term, close(), then top() for every term.  The tail
// constant k of a row is -1.5 (1 + sum of its cl): operands bring g = 1.5 + l 2^-32, the
// fraction of mid comes as 1 + fraction, and mid starts at one half.
struct FxDot {
  long long mid = kFxHalf, hi = 0;
  float f = 0.0f;
  __host__ __device__ __forceinline__ void term(FxC c, const FxV& x) {
    mid = fx_mad(c.l, x.h, fx_mad(c.h, x.l, mid));
    f = fmaf(c.cl, x.g, fmaf(c.c, x.f, f));
  }
  __host__ __device__ __forceinline__ void close(float k) {
    hi = mid >> 32;
    f += fx_frac1((unsigned)mid) + k;
  }
  __host__ __device__ __forceinline__ void top(FxC c, const FxV& x) { hi = fx_mad(c.h, x.h, hi); }
};

// sum u r of two sets of values: dh 2^64 + (dm + da) 2^32 + dl 2^10, exact but for the
// rounding of da (the tails' products with the other value's high word; the rest of them is
// below 2^-54 of u r) and the cut of dl.
struct FxInner {
  long long dh = 0, dm = 0, dl = 0;
  float da = 0.0f;
  __host__ __device__ __forceinline__ void add(long long u, float uf, long long r, float rf) {
    const FxV a = fx_operand(u + kFxHalf, 0.0f), b = fx_operand(r + kFxHalf, 0.0f);
    da = fmaf((float)a.h, rf, fmaf((float)b.h, uf, da));
    dm = fx_mad(a.h, b.l, fx_mad(a.l, b.h, dm));
    dh = fx_mad(a.h, b.h, dh);
    dl += fx_mad(a.l, b.l, 0) >> 10;
  }
};

// Folded operator: coefficients in the layout of tdks_internal.h (CS of them), tail
// constants of the even, odd and middle rows (KS).
template <int N>
struct FxOp {
  static constexpr int h = N / 2, CS = 2 * h * h + 2 * h + 1, KS = 2 * h + 1;
};

// M (v, f) / 2 for a centrosymmetric N x N operator; c(i), k(i) its coefficients and tail
// constants; out(q, V, F) takes output q as soon as it is formed (all inputs have been
// read by then, so it may overwrite them in place).
template <int N, class CF, class KF, class OF>
__host__ __device__ __forceinline__ void fx_apply(CF c, KF k, const long long (&v)[N], const float (&f)[N], OF out) {
  constexpr int h = N / 2;
  constexpr int hh = h > 0 ? h : 1;
  FxV e[hh], o[hh], m{0, 0, 0.0f, 0.0f};
#pragma unroll
  for (int i = 0; i < h; ++i) {
    e[i] = fx_operand(v[i] + v[N - 1 - i] + kFxHalf, f[i] + f[N - 1 - i]);
    o[i] = fx_operand(v[i] - v[N - 1 - i] + kFxHalf, f[i] - f[N - 1 - i]);
  }
  if (N & 1) m = fx_operand(v[h] + kFxHalf, f[h]);
#pragma unroll
  for (int q = 0; q < h; ++q) {
    FxDot a, b;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      a.term(c(q * h + i), e[i]);
      b.term(c(h * h + q * h + i), o[i]);
    }
    if (N & 1) a.term(c(2 * h * h + q), m);
    a.close(k(q));
    b.close(k(h + q));
#pragma unroll
    for (int i = 0; i < h; ++i) {
      a.top(c(q * h + i), e[i]);
      b.top(c(h * h + q * h + i), o[i]);
    }
    if (N & 1) a.top(c(2 * h * h + q), m);
    out(q, a.hi + b.hi, a.f + b.f);
    out(N - 1 - q, a.hi - b.hi, a.f - b.f);
  }
  if (N & 1) {
    FxDot a;
#pragma unroll
    for (int i = 0; i < h; ++i) a.term(c(2 * h * h + h + i), e[i]);
    a.term(c(2 * h * h + 2 * h), m);
    a.close(k(2 * h));
#pragma unroll
    for (int i = 0; i < h; ++i) a.top(c(2 * h * h + h + i), e[i]);
    a.top(c(2 * h * h + 2 * h), m);
    out(h, a.hi, a.f);
  }
}

// Tail constant i (ke, ko, km order) of the folded rows whose cl are given by c(i).
template <int N, class CF>
__host__ __device__ __forceinline__ float fx_tail_const(CF c, int i) {
  constexpr int h = N / 2;
  float s = 0.0f;
  if (i < h) {
    for (int j = 0; j < h; ++j) s += c(i * h + j).cl;
    if (N & 1) s += c(2 * h * h + i).cl;
  } else if (i < 2 * h) {
    for (int j = 0; j < h; ++j) s += c(h * h + (i - h) * h + j).cl;
  } else {
    for (int j = 0; j < h; ++j) s += c(2 * h * h + h + j).cl;
    s += c(2 * h * h + 2 * h).cl;
  }
  return -1.5f - 1.5f * s;
}

// y -> V and its tail at the block exponent eb (biased exponent of the block's largest |y|,
// in [64, 2046]): |V| < 2^kFxBits, cut towards zero; the bits below one unit, to 2^-32 of it,
// go to the tail.  An entry 2^-k of the largest has only 55 - k bits in V: without the tail
// the element operator was off by up to 1e-13 on vectors that fall off steeply inside an
// element, by 2e-16 .. 7e-15 with FP64 contractions.  Subnormal y give 0.
__host__ __device__ __forceinline__ long long fx_from_bits(unsigned hw, unsigned lw, int eb, float& f) {
  const int e = (int)((hw >> 20) & 0x7ffu);
  const unsigned long long m = (((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32) | lw) << (kFxBits - 53);
  int d = eb - e;
  d = (e == 0 || d > 95) ? 95 : d;
  const unsigned long long v = d < 64 ? m >> d : 0;
  const unsigned w = d == 0 ? 0u : d < 64 ? (unsigned)((m << (64 - d)) >> 32) : (unsigned)(m >> 32) >> (d - 64);
  const float t = (float)w * 0x1p-32f;
  const bool neg = (hw & 0x80000000u) != 0;
  f = neg ? -t : t;
  return neg ? -(long long)v : (long long)v;
}

// The values of a block raised to use the bits that the contractions so far have left free:
// the shift for big, the OR of fx_magnitude of all of them (at most 18, 0 for a block of
// zeros; raised values stay below 2^54 + 2^23), and the raise of one value, |f| < 8.
__host__ __device__ __forceinline__ unsigned fx_magnitude(long long v) {
  const int h = (int)(v >> 32);
  return (unsigned)(h ^ (h >> 31)) | (unsigned)((unsigned)v != 0u);
}
__host__ __device__ __forceinline__ int fx_free_bits(unsigned big) {
#ifdef __CUDA_ARCH__
  const int z = __clz((int)big);
#else
  const int z = big ? __builtin_clz(big) : 32;
#endif
  return z == 32 ? 0 : (z - 10 < 18 ? z - 10 : 18);
}
__host__ __device__ __forceinline__ void fx_raise(long long& v, float& f, int s) {
  const float g = f * fx_bits_float((unsigned)(127 + s) << 23);
  const float m = g + 12582912.0f;                   // 1.5 2^23 + nearest integer, |g| < 2^21
  v = (long long)((unsigned long long)v << s) + ((int)fx_float_bits(m) - 0x4b400000);
  f = g - (m - 12582912.0f);
}

// c (hi + lo) scale to the nearest integer, scale a power of two
__host__ __device__ __forceinline__ long long fx_scaled(double c, double hi, double lo, double scale) {
  const double q = c * hi, r = fma(c, hi, -q) + c * lo;
#ifdef __CUDA_ARCH__
  return __double2ll_rn(q * scale) + __double2ll_rn(r * scale);
#else
  return llrint(q * scale) + llrint(r * scale);
#endif
}

// Products of two numbers in fixed point, |V| < 2^kFxPBits, each with the exponent eb of the
// largest entry of its row or column; the bits below a unit are cut.  At 55 bits, which need no
// carry(), the 2-norm of a fast-diagonalization product was off by up to six times an FP64
// chain's error (steep or peaked columns); at 58 it is at most 0.84 times the chain's or one
// rounding, 2^-53, whichever is larger (axes of 3 to 255 nodes; host test).
constexpr int kFxPBits = 58;
constexpr int kFxK = 255;   // terms: K 2^52 and the carries < 2^61
__host__ __device__ __forceinline__ FxV fx_factor(unsigned hw, unsigned lw, int eb) {
  const int e = (int)((hw >> 20) & 0x7ffu);
  const unsigned long long m = (((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32) | lw) << (kFxPBits - 53);
  const int d = eb - e;
  const long long v = e == 0 || d > 63 ? 0 : (long long)(m >> (d & 63));
  return fx_operand(((hw & 0x80000000u) ? -v : v) + kFxHalf, 0.0f);
}
// sum a b in units of 2^64: h h' and h l' + l h' exactly (carry() at least every 16 terms), l l'
// in FP32
struct FxSum {
  long long mid = 0, hi = 0;
  float f = 0.0f;
  // lf, lg: l 2^-32 of a and b
  __host__ __device__ __forceinline__ void add(int ah, int al, float lf, int bh, int bl, float lg) {
    mid = fx_mad(ah, bl, fx_mad(al, bh, mid));
    hi = fx_mad(ah, bh, hi);
    f = fmaf(lf, lg, f);
  }
  __host__ __device__ __forceinline__ void carry() {
    hi += mid >> 32;
    mid &= 0xffffffffll;
  }
  // the sum 2^s, s its free bits (at most 20), |.| < 2^62
  __host__ __device__ __forceinline__ long long value(int& s) const {
    const long long t = hi + (mid >> 32), m = t ^ (t >> 63);
#ifdef __CUDA_ARCH__
    const int z = __clzll(m);
#else
    const int z = m ? __builtin_clzll((unsigned long long)m) : 64;
#endif
    s = z - 2 < 20 ? z - 2 : 20;
    const float fr = f * fx_bits_float((unsigned)(127 + s) << 23);
#ifdef __CUDA_ARCH__
    const int r = __float2int_rn(fr);
#else
    const int r = (int)lrintf(fr);
#endif
    return (long long)((unsigned long long)t << s) + (long long)((unsigned)mid >> (32 - s)) + r;
  }
};

#ifdef __CUDACC__
__device__ __forceinline__ double pow2(int e) {   // 2^e, e clamped to the normal range
  e = e < -1022 ? -1022 : (e > 1023 ? 1023 : e);
  return __hiloint2double((e + 1023) << 20, 0);
}

// V 2^e -> double, correctly rounded, |V| < 2^62, e in [-1074, 939], eb = e << 20 (two
// additions, the first exact)
__device__ __forceinline__ double fx_to_double(long long v, int eb) {
  const unsigned hi = (unsigned)((unsigned long long)v >> 32) ^ 0x80000000u;
  const double dh = __hiloint2double(0x45300000 + eb, (int)hi);            // 2^e (2^84 + (vh + 2^31) 2^32)
  const double dl = __hiloint2double(0x43300000 + eb, (int)(unsigned)v);   // 2^e (2^52 + vl)
  const double cc = __hiloint2double(0x45300000 + eb, (int)0x80100000u);   // 2^e (2^84 + 2^63 + 2^52)
  return (dh - cc) + dl;
}
#endif

}  // namespace tdks
