// Register-resident FFTs on block fixed-point data: the FP64-class arithmetic of the table-form
// P(dt) kernel (k_theta_fx.cu).
//
// Why.  GB300 issues 1.7 FP64 FMAs per clock and SM (measured) against 60 64-bit integer adds and
// 24 wide integer multiply-adds.  A vector that one thread transforms is therefore held as 64-bit
// integers with one common binary exponent:
//   value_n = x_n 2^E,   |Re x_n|, |Im x_n| <= 2^57 on entry of a transform of length <= 32,
// so that the largest output of the transform (modulus <= 32 * 2^57.5) still fits.  Additions are
// exact; a product with a twiddle constant of 64 fractional bits is off by less than two units of
// 2^E, i.e. 2^-56 of the vector's largest entry, and on average by less than a quarter of one, where
// an FP64 FMA rounds at 2^-53 of each result.  Between transforms a vector keeps its exponent and the number of magnitude bits it
// uses, and the next transform aligns what it gathers to 57 bits again.
//
// A rotation by an angle up to 45 degrees is done by three lifting steps
//   x += a y, y += s x, x += a y,  a = -tan(phi/2), s = sin(phi)
// (Daubechies and Sweldens, "Factoring wavelet transforms into lifting steps", J. Fourier Anal.
// Appl. 1998, apply the factorisation to rotations): three products instead of four, and every
// constant stays below one half after 1 - s replaces an s above it.
#pragma once

#include <cstdint>
#include <type_traits>

namespace chasm {
namespace {

using i64 = long long;
using u64 = unsigned long long;

// ---- constants with 64 fractional bits, evaluated at compile time ----
using fx128 = unsigned __int128;
constexpr u64 kFxPi61 = 0x6487ED5110B4611AULL;   // pi 2^61 (pi = 3.243F6A88 85A308D3 ... hex)
constexpr u64 fx_mulq(u64 a, u64 b) { return (u64)(((fx128)a * b) >> 64); }
constexpr u64 fx_divq(u64 a, u64 b) {   // a / b with 64 fractional bits, a < b
  return (u64)((((fx128)a) << 64) / b);
}
// 2 pi k / m for 0 < k / m <= 1/8, 64 fractional bits (at most pi / 4 < 1)
constexpr u64 fx_angle(int k, int m) { return (u64)((((fx128)kFxPi61) * 16 * (unsigned)k) / (unsigned)m); }
constexpr u64 fx_sin_series(u64 x) {
  const u64 x2 = fx_mulq(x, x);
  u64 t = x, s = x;
  for (int i = 1; i < 14; ++i) {
    t = fx_mulq(t, x2) / (unsigned)((2 * i) * (2 * i + 1));
    s = (i & 1) ? s - t : s + t;
  }
  return s;
}
constexpr u64 fx_vers_series(u64 x) {   // 1 - cos x
  const u64 x2 = fx_mulq(x, x);
  u64 t = x2 / 2, s = t;
  for (int i = 2; i < 14; ++i) {
    t = fx_mulq(t, x2) / (unsigned)((2 * i - 1) * (2 * i));
    s = (i & 1) ? s + t : s - t;
  }
  return s;
}
constexpr u64 fx_sin(int k, int m) { return fx_sin_series(fx_angle(k, m)); }
constexpr u64 fx_vers(int k, int m) { return fx_vers_series(fx_angle(k, m)); }
// sin, 1 - cos and tan(phi / 2) of phi = 2 pi K / M, 0 < K / M <= 1/8
template <int K, int M>
struct FxK {
  static constexpr u64 sin = fx_sin(K, M);
  static constexpr u64 vers = fx_vers(K, M);
  static constexpr u64 cos = (u64)0 - vers;
  static constexpr u64 tanh = fx_divq(fx_vers(K, M), fx_sin(K, M));
};

template <int B, int E, int S = 1, class F>
__device__ __forceinline__ void xfor(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    xfor<B + S, E, S>(f);
  }
}

// ---- products ----
// a b in 64 bits.  On the device written as its two halves: the compiler issues one wide product for
// them, and four instructions for the C expression of the same product.
__device__ __forceinline__ i64 fx_wide(int a, int b) {
#ifdef __CUDA_ARCH__
  int hi;
  unsigned lo;
  i64 r;
  asm("mul.hi.s32 %0, %1, %2;" : "=r"(hi) : "r"(a), "r"(b));
  asm("mul.lo.s32 %0, %1, %2;" : "=r"(lo) : "r"(a), "r"(b));
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(lo), "r"(hi));
  return r;
#else
  return (i64)a * (i64)b;
#endif
}
// High words of products, rounded to nearest: the half goes through the low words, so that zero stays
// zero and each product is one wide multiply-add.  (Rounded down, the errors of a transform's products
// have one sign and add up in single outputs: the largest error of Theta at N_k = 32 was up to 2.6 times
// that of an FP64 transform, now 0.84 to 0.94 times; and the separate high products and additions took
// longer: P(dt) at 16^3 x 32^3 36.8 -> 35.5 ms.)
// a b / 2^32, signed and unsigned
__device__ __forceinline__ int fx_hi(int a, int b) {
#ifdef __CUDA_ARCH__
  int t;
  asm("{\n .reg .u32 l;\n mad.lo.cc.u32 l, %1, %2, 0x80000000;\n madc.hi.s32 %0, %1, %2, 0;\n}" : "=r"(t) : "r"(a), "r"(b));
  return t;
#else
  return (int)(((i64)a * b + 0x80000000LL) >> 32);
#endif
}
__device__ __forceinline__ unsigned fx_hiu(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  unsigned t;
  asm("{\n .reg .u32 l;\n mad.lo.cc.u32 l, %1, %2, 0x80000000;\n madc.hi.u32 %0, %1, %2, 0;\n}" : "=r"(t) : "r"(a), "r"(b));
  return t;
#else
  return (unsigned)(((u64)a * b + 0x80000000ULL) >> 32);
#endif
}
// (a b + c d) / 2^32 modulo 2^32, a and b signed
__device__ __forceinline__ int fx_hi2(int a, int b, unsigned c, unsigned d) {
#ifdef __CUDA_ARCH__
  int t;
  asm("{\n .reg .u32 l, h;\n mad.lo.cc.u32 l, %1, %2, 0x80000000;\n madc.hi.s32 h, %1, %2, 0;\n"
      " mad.lo.cc.u32 l, %3, %4, l;\n madc.hi.u32 %0, %3, %4, h;\n}"
      : "=r"(t)
      : "r"(a), "r"(b), "r"(c), "r"(d));
  return t;
#else
  return (int)(unsigned)(((u64)((i64)a * b) + (u64)c * d + 0x80000000ULL) >> 32);
#endif
}
// A constant w = C / 2^64 as 2^-32 (wh + wl / 2^32) with a signed low word.
__host__ __device__ constexpr int fx_low(u64 c) { return (int)(unsigned)c; }
__host__ __device__ constexpr unsigned fx_high(u64 c) { return (unsigned)((c >> 32) + (((unsigned)c) >> 31)); }
// Whether the cross terms of x w, wh times the low word of x and wl times its signed high word, add up
// inside one signed word (over 2^32) for every |x| < 2^62.7: below wh, and at most |wl| 2^30.7 / 2^32
// (2^30.7 < 0x67f80000), and one for the rounding.
__host__ __device__ constexpr bool fx_one_word(u64 c) {
  const i64 wl = fx_low(c);
  const u64 cross = (u64)(wl < 0 ? -wl : wl) * 0x67f80000ULL >> 32;
  return fx_high(c) + cross + 1 < (1ULL << 31);
}
// x w for a constant w = C / 2^64 < 1/2; |x| < 2^62.7.  The constant's low word is taken as signed; its
// product with the low word of x, below half a unit and on average below a quarter, is left out.  Where
// the constant allows it (fx_one_word) the cross terms are added before they are rounded: within a unit of
// the exact product, 1.5 otherwise.
template <u64 C>
__device__ __forceinline__ i64 fx_mulc(i64 x) {
  static_assert(C < (1ULL << 63) - (1ULL << 32), "constants below one half");
  constexpr int wl = fx_low(C);
  constexpr unsigned wh = fx_high(C);
  const int xh = (int)(x >> 32);
  const unsigned xl = (unsigned)x;
  if constexpr (fx_one_word(C)) return fx_wide((int)wh, xh) + (i64)fx_hi2(wl, xh, wh, xl);
  else return fx_wide((int)wh, xh) + (i64)(u64)fx_hiu(wh, xl) + (i64)fx_hi(wl, xh);
}
// a +- x w, 0 <= w <= 1 given as C / 2^64
template <bool NEG, u64 C>
__device__ __forceinline__ i64 fx_fma(i64 a, i64 x) {
  if constexpr (C < (1ULL << 63) - (1ULL << 32)) {
    const i64 p = fx_mulc<C>(x);
    return NEG ? a - p : a + p;
  } else {   // x w = x - x (1 - w)
    const i64 p = fx_mulc<(u64)0 - C>(x);
    return NEG ? (a - x) + p : (a + x) - p;
  }
}
// x w
template <u64 C>
__device__ __forceinline__ i64 fx_mul(i64 x) {
  if constexpr (C < (1ULL << 63) - (1ULL << 32)) return fx_mulc<C>(x);
  else return x - fx_mulc<(u64)0 - C>(x);
}
struct fxc {
  i64 re, im;
};

// z e^{-2 pi i K / M} (INV: e^{+2 pi i K / M}), 8 | M
template <int K_, int M, bool INV>
__device__ __forceinline__ fxc fx_rot(fxc z) {
  constexpr int K = ((INV ? K_ : -K_) % M + M) % M;   // by the angle +2 pi K / M
  constexpr int q = (K + M / 8 - 1) / (M / 4);        // quarter turns taken out: rest in (-M/8, M/8]
  constexpr int r = K - q * (M / 4);
  constexpr int a = r < 0 ? -r : r;
  if constexpr (8 * a == M) {          // 45 degrees: (x -+ y) / sqrt 2, 1 / sqrt 2 = 1 - vers
    constexpr u64 V = FxK<1, 8>::vers;
    const i64 d = r > 0 ? z.re - z.im : z.re + z.im;
    const i64 s = r > 0 ? z.re + z.im : z.im - z.re;
    z = {d - fx_mulc<V>(d), s - fx_mulc<V>(s)};
  } else if constexpr (a != 0) {
    constexpr u64 T = FxK<a, M>::tanh, S = FxK<a, M>::sin;
    z.re = fx_fma<(r > 0), T>(z.re, z.im);
    z.im = fx_fma<(r < 0), S>(z.im, z.re);
    z.re = fx_fma<(r > 0), T>(z.re, z.im);
  }
  if constexpr ((q & 3) == 1) return {-z.im, z.re};
  else if constexpr ((q & 3) == 2) return {-z.re, -z.im};
  else if constexpr ((q & 3) == 3) return {z.im, -z.re};
  else return z;
}

// ---- vectors with a common exponent ----
// magnitude bits to which the entries of a vector are aligned before a transform (the outputs of
// two inverse halves are added: one bit less)
constexpr int kFxBits = 57;

__device__ __forceinline__ void mag_or(unsigned& m, i64 x) {
  const int h = (int)(x >> 32);
  m |= (unsigned)(h ^ (h >> 31));
}
// number of bits that hold the magnitudes whose high words were or-ed into m
__device__ __forceinline__ int mag_bits(unsigned m) { return 64 - __clz((int)m); }

// A double as an integer on the scale of a vector whose largest exponent field is em (fields as
// fx_field gives them, em >= 1): kFxBits bits below the largest entry, magnitudes rounded down.
// fx_exponent(em) is the exponent of the integers; em = 0x7ff means that an entry is not finite.
__device__ __forceinline__ int fx_field(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }
__device__ __forceinline__ int fx_exponent(int em) { return em - 1023 - (kFxBits - 1); }
__device__ __forceinline__ i64 fx_from_double(double v, int em) {
  const int hi = __double2hiint(v), e = fx_field(v);
  const unsigned mh = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
  u64 m = ((u64)mh << 32 | (unsigned)__double2loint(v)) << (kFxBits - 53);
  m >>= min(63, em - max(e, 1));
  const i64 sg = (i64)(hi >> 31);
  return ((i64)m ^ sg) - sg;
}
// 2^e for e in [-900, 900]
__device__ __forceinline__ double pow2_mid(int e) { return __hiloint2double((e + 1023) << 20, 0); }

// x y / 2^64 for a symbol value y in its stored form, rounded: high word, and the low word as a signed
// number (the high word holds its carry)
__device__ __forceinline__ i64 fx_mulsym(i64 x, i64 y) {
  const int xh = (int)(x >> 32), yh = (int)(y >> 32), yl = (int)y;
  const unsigned xl = (unsigned)x;
  // the cross terms, signed high times unsigned low word (below 2^30 in magnitude: |yh| <= 2^30), and
  // signed times signed (below 2^29.7)
  const int t = fx_hi2(yl, xh, (unsigned)yh, xl) - (int)(xl & (unsigned)(yh >> 31));
  return fx_wide(xh, yh) + (i64)t;
}

// ---- transforms ----
// DFT_4 in place, natural order: X_j = sum_n x_n e^{-2 pi i jn/4}
__device__ __forceinline__ void fx_dft4(fxc& a, fxc& b, fxc& c, fxc& d) {
  const fxc s = {a.re + c.re, a.im + c.im}, t = {a.re - c.re, a.im - c.im};
  const fxc u = {b.re + d.re, b.im + d.im}, v = {b.re - d.re, b.im - d.im};
  a = {s.re + u.re, s.im + u.im};
  b = {t.re + v.im, t.im - v.re};
  c = {s.re - u.re, s.im - u.im};
  d = {t.re - v.im, t.im + v.re};
}

// DFT_M (M = 4, 8, 16) of x[0..M), natural order in and out, by radix 4: 4 rotations by 45 degrees
// and 4 others at M = 16 (radix 2: 6 and 4)
template <int M>
__device__ __forceinline__ void fx_dft(fxc* x) {
  static_assert(M == 4 || M == 8 || M == 16, "DFT lengths");
  if constexpr (M == 4) {
    fx_dft4(x[0], x[1], x[2], x[3]);
  } else {
    constexpr int R = M / 4;   // M = 4 R: DFT_4 over n = i + R m, twiddle, DFT_R over i
    xfor<0, R>([&](auto I) {
      constexpr int i = decltype(I)::value;
      fx_dft4(x[i], x[i + R], x[i + 2 * R], x[i + 3 * R]);   // x[i + R k2]
      xfor<1, 4>([&](auto K) {
        constexpr int k2 = decltype(K)::value;
        x[i + R * k2] = fx_rot<i * k2, M, false>(x[i + R * k2]);
      });
    });
    fxc y[M];
    xfor<0, 4>([&](auto K) {
      constexpr int k2 = decltype(K)::value;
      if constexpr (R == 4) {
        fx_dft4(x[4 * k2], x[4 * k2 + 1], x[4 * k2 + 2], x[4 * k2 + 3]);
        xfor<0, 4>([&](auto J) { y[k2 + 4 * decltype(J)::value] = x[4 * k2 + decltype(J)::value]; });
      } else {
        const fxc a = x[2 * k2], b = x[2 * k2 + 1];
        y[k2] = {a.re + b.re, a.im + b.im};
        y[k2 + 4] = {a.re - b.re, a.im - b.im};
      }
    });
    xfor<0, M>([&](auto J) { x[decltype(J)::value] = y[decltype(J)::value]; });
  }
}

// A transform of length N (8, 16, 32) is two of length N / 2 (fft_fx_core) and one radix-2 step
// before it (fft_fx_pre: x in time order) or after it (fft_fx_post: x out in time order); the
// frequencies sit at x[j] = X_{fx_freq(j)}, the even ones first.  ODD: the odd outputs of a
// zero-padded length-2N transform, X_q = sum_n x_n e^{-2 pi i (2q + 1) n / (2N)}, or the sum over
// such frequencies: its radix-2 step holds the twist e^{-i pi n / N} in its own rotations.  All
// transforms have the sign of e^{-i...}; the other sign is this one on (im, re).
// On entry |Re|, |Im| <= 2^57 (N = 32); the outputs stay below 2^63.
template <int N>
__host__ __device__ constexpr int fx_freq(int j) { return 2 * (j % (N / 2)) + j / (N / 2); }

template <int N, bool ODD>
__device__ __forceinline__ void fft_fx_pre(fxc (&x)[N]) {
  constexpr int M = N / 2;
  xfor<0, M>([&](auto I) {
    constexpr int n = decltype(I)::value;
    const fxc a = x[n], b = x[n + M];
    if constexpr (ODD) {
      x[n] = fx_rot<n, 2 * N, false>(fxc{a.re + b.im, a.im - b.re});            // a - i b
      x[n + M] = fx_rot<3 * n, 2 * N, false>(fxc{a.re - b.im, a.im + b.re});    // a + i b
    } else {
      x[n] = {a.re + b.re, a.im + b.im};
      x[n + M] = fx_rot<n, N, false>(fxc{a.re - b.re, a.im - b.im});
    }
  });
}
template <int N>
__device__ __forceinline__ void fft_fx_core(fxc (&x)[N]) {
  fx_dft<N / 2>(x);
  fx_dft<N / 2>(x + N / 2);
}
template <int N, bool ODD>
__device__ __forceinline__ void fft_fx_post(fxc (&x)[N]) {
  constexpr int M = N / 2;
  xfor<0, M>([&](auto I) {
    constexpr int n = decltype(I)::value;
    if constexpr (ODD) {
      const fxc a = fx_rot<n, 2 * N, false>(x[n]), b = fx_rot<3 * n, 2 * N, false>(x[n + M]);
      x[n] = {a.re + b.re, a.im + b.im};
      x[n + M] = {a.im - b.im, b.re - a.re};   // -i (a - b)
    } else {
      const fxc a = x[n], b = fx_rot<n, N, false>(x[n + M]);
      x[n] = {a.re + b.re, a.im + b.im};
      x[n + M] = {a.re - b.re, a.im - b.im};
    }
  });
}

}  // namespace
}  // namespace chasm
