// The constant products of fft_fx.cuh on the host, against exact 128-bit products: the twiddle
// constants of every transform length and constants whose cross terms are as large as any can be,
// at the ends of the accepted range of x and at seeded values.  Exit status 0 when every product is
// within two units.
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

template <u64 C>
void check() {
  if constexpr (C < (1ULL << 63) - (1ULL << 32)) {
    const i64 top = (i64)std::floor(std::exp2(62.7));
    u64 r = 88172645463325252ULL;
    for (int n = 0; n < 4000; ++n) {
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
    }
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
  return bad ? 1 : 0;
}
