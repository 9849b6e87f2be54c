// The constant products of fft_fx.cuh on the host, against exact 128-bit products: the twiddle
// constants of every transform length and constants whose cross terms are as large as any can be,
// at the ends of the accepted range of x and at seeded values; and the product with a stored symbol
// value.  Exit status 0 when every product is within two units, a product with zero is zero and the
// mean error over the seeded values is below 0.6 units: errors of one sign would add up in a transform's
// outputs (a quarter is what the products of the low words, left out, may amount to, another quarter the
// ties of a constant whose low word is 2^31, rounded up; the mean's standard deviation is below 0.007;
// both high words rounded down: 0.75 at least).  Symbol values of either sign: below 0.05.
#include <cstdio>
#include <cmath>
#include <cstring>
#include <cstdint>
#include <algorithm>

#define __device__
#define __host__
#define __forceinline__ inline
using std::max;
using std::min;
static inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static inline int __double2hiint(double v) {
  unsigned long long b;
  std::memcpy(&b, &v, 8);
  return (int)(b >> 32);
}
static inline int __double2loint(double v) {
  unsigned long long b;
  std::memcpy(&b, &v, 8);
  return (int)b;
}
static inline double __hiloint2double(int h, int l) {
  const unsigned long long b = (unsigned long long)(unsigned)h << 32 | (unsigned)l;
  double v;
  std::memcpy(&v, &b, 8);
  return v;
}

#include "../../paper_2205_02380_gb300/csrc/fft_fx.cuh"

using namespace chasm;

static int bad = 0;

// got minus the exact x c / 2^64
static double error(i64 got, i64 x, __int128 c) {
  const __int128 p = (__int128)x * c;
  return (double)(got - (i64)(p >> 64)) - std::ldexp((double)(u64)p, -64);
}

template <u64 C>
void check() {
  if constexpr (C < (1ULL << 63) - (1ULL << 32)) {
    const i64 top = (i64)std::floor(std::exp2(62.7));
    u64 r = 88172645463325252ULL;
    double sum = 0.0;
    if (fx_mulc<C>(0) != 0) ++bad;
    for (int n = 0; n < 4400; ++n) {
      r ^= r << 13;
      r ^= r >> 7;
      r ^= r << 17;
      i64 x = (i64)(r % (u64)top) * ((n & 1) ? -1 : 1);
      if (n < 400) x = top - (i64)(r >> 60) * (n < 200 ? 1 : 0x7fffffffLL);
      if (n < 400 && (n & 1)) x = -x;
      if (n < 100) x |= 0xffffffffLL;   // the largest low word (also with the largest high word)
      if (x > top || x < -top) x = x < 0 ? -top : top - (1LL << 32) + ((1LL << 32) - 1 - (top & 0xffffffffLL));
      const i64 want = (i64)(((__int128)x * (__int128)C) >> 64);
      const i64 got = fx_mulc<C>(x);
      if (got - want > 2 || want - got > 2) {
        if (bad++ < 5) std::printf("C %016llx x %lld: %lld, not %lld\n", (unsigned long long)C, x, got, want);
        return;
      }
      if (n >= 400) sum += error(got, x, (__int128)C);
    }
    if (std::fabs(sum / 4000) > 0.6) {
      if (bad++ < 5) std::printf("C %016llx: mean error %.3f units\n", (unsigned long long)C, sum / 4000);
    }
  }
}

// y: a magnitude of at most 2^62, stored as fx_mulsym reads it
static void check_symbol() {
  const i64 top = (i64)std::floor(std::exp2(62.7));
  u64 r = 1181783497276652981ULL;
  double sum = 0.0;
  for (int n = 0; n < 100000; ++n) {
    u64 v[2];
    for (u64& q : v) {
      r ^= r << 13;
      r ^= r >> 7;
      r ^= r << 17;
      q = r;
    }
    i64 x = (i64)(v[0] % (u64)top) * ((n & 1) ? -1 : 1), y = (i64)(v[1] >> 2) * ((n & 2) ? -1 : 1);
    if (n < 64) {   // the ends
      x = (n & 1) ? -top : top;
      y = (n & 2) ? -(1LL << 62) : 1LL << 62;
      if (n & 4) y += (n & 2) ? 0x7fffffffLL : -0x7fffffffLL;
    }
    const int lo = (int)(unsigned)(u64)y;
    const i64 stored = (i64)((u64)(y - lo) | (unsigned)lo);
    const double e = error(fx_mulsym(x, stored), x, (__int128)y);
    if (std::fabs(e) > 2.0) {
      if (bad++ < 5) std::printf("x %lld y %lld: error %.3f\n", x, y, e);
      return;
    }
    if (fx_mulsym(0, stored) != 0) ++bad;
    if (n >= 64) sum += e;
  }
  if (std::fabs(sum / 1e5) > 0.05) {
    ++bad;
    std::printf("symbol products: mean error %.3f units\n", sum / 1e5);
  }
}

template <int K, int M>
void angle() {
  if constexpr (K >= 1) {
    check<FxK<K, M>::sin>();
    check<(u64)0 - FxK<K, M>::sin>();
    check<FxK<K, M>::vers>();
    check<(u64)0 - FxK<K, M>::cos>();
    check<FxK<K, M>::tanh>();
    angle<K - 1, M>();
  }
}

int main() {
  angle<1, 8>();
  angle<2, 16>();
  angle<4, 32>();
  angle<8, 64>();
  angle<16, 128>();
  // high words around one third and up to one half, with the largest low words of either sign
  check<0x555555547fffffffULL>();
  check<0x5555555380000000ULL>();
  check<0x5555555480000000ULL>();
  check<0x5000000080000000ULL>();
  check<0x4c0000007fffffffULL>();
  check<0x4b0000007fffffffULL>();
  check<0x7ffffffe7fffffffULL>();
  check<0x7ffffffd80000001ULL>();
  check<0x7ffffffe00000000ULL>();
  check<0x000000007fffffffULL>();
  check<0x0000000080000000ULL>();
  check_symbol();
  return bad ? 1 : 0;
}
