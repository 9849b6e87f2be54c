// The k-passes of the quadratic potential in double precision (Eq. 5.1): the exact shift along k_d
// (Strang) and the spectral k-derivative (LPC1), one k-dimension per launch, by transforms of length
// N in block fixed point (fft_fx.cuh).
//
// As circulants (one FP64 FMA per entry of an N x N matrix) these passes were bound by the FP64
// pipe, 1.7 FMAs per clock and SM: 5.1 ms per shift at 121 x 5^2 x 32^3, 20 times the time HBM
// needs to read and write f.  A thread transforms two real lines as one complex line, each line on
// its own exponent (the passes are real operators, so the lines do not mix), multiplies by the
// pass's spectrum and transforms back: three shifts 16.2 -> 2.36 ms (HBM alone 0.7).  Now two warps per
// scheduler (254 registers) wait for their own results (2.5 warps per issue), with the FP64 pipe, which
// converts back, 68 % busy and the integer pipe 37 %; the pass along k3 (51 % and 26 %) waits for shared
// memory as well.
//
// Errors: 57 bits below a line's largest entry on entry, about 3 units of the last one from each
// transform and one from the spectrum: 2^-54 of the line's largest entry, where the sum of N
// FP64 products is off by about 2^-53 of its root mean square times sqrt(N).
//
// A line with a non-finite entry takes the circulant sum, entry by entry, in FP64.
#include <cmath>

#include "internal.hpp"
#include "fft_fx.cuh"

namespace chasm {
namespace {

struct KPassParams {
  const double* in;
  const double* add;     // the derivative: out = add + scale D in; null: out = scale D in
  double* out;           // the shift: out = in, in place
  int64_t nxp;
  int nx1, nx2, nx3, dim;
  const double* rows;    // circulant first columns: the shift per x_d index [id][N], the derivative [N]
  const i64* spec;       // spectra in the same order, entries of fx_mulsym: [id][N][2] re, im, or [N]
  double rate, x_lo, h, center, coef;   // the derivative: scale of x_d index i is rate (x_lo + i h - center) coef
  double unit;                          // of its spectrum
};

// out_j = add_j + scale sum_l c_{j-l} u_l for one line, u from src, stride apart; kept out of the
// kernels' registers
template <int N>
__device__ __noinline__ void circulant_line(const double* src, const double* add, double* dst, int64_t stride,
                                            int64_t out_stride, const double* c, double scale) {
  double o[N];
#pragma unroll 1
  for (int j = 0; j < N; ++j) {
    double acc = 0.0;
#pragma unroll 1
    for (int l = 0; l < N; ++l) acc = fma(c[(j - l) & (N - 1)], src[l * stride], acc);
    o[j] = scale * acc;
  }
#pragma unroll 1
  for (int j = 0; j < N; ++j) dst[j * out_stride] = add ? add[j * out_stride] + o[j] : o[j];
}

// SHIFT: complex spectrum with the x index; else the derivative's i xi.  ROWS: the lines are
// contiguous (dim = 2) and staged through shared memory, a pair of lines per row.
template <int N, bool SHIFT, bool ROWS>
__global__ void __launch_bounds__(ROWS ? 64 : 128) k_kpass_fx(const KPassParams p) {
  constexpr int N2 = N * N, PAIRS = N2 / 2, RW = N + 1;   // pairs per x point; staging row in 16-byte units
  __shared__ double2 tile[ROWS ? 64 * RW : 1];
  const int64_t pair = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = p.nxp * PAIRS;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t pair0 = pair - lane;                       // the warp's first pair
  const int here = (int)min((int64_t)32, total - pair0);   // its pairs
  if (here <= 0) return;
  const bool on = lane < here;
  const int64_t xp = (on ? pair : pair0) / PAIRS;
  const int r = (int)((on ? pair : pair0) % PAIRS) * 2;    // first line of the pair
  const int i1 = (int)(xp / ((int64_t)p.nx2 * p.nx3)), i2 = (int)((xp / p.nx3) % p.nx2), i3 = (int)(xp % p.nx3);
  const int id = p.dim == 0 ? i1 : (p.dim == 1 ? (SHIFT ? p.nx1 : 0) + i2 : (SHIFT ? p.nx1 + p.nx2 : 0) + i3);
  int64_t base, stride;
  if (p.dim == 0) {
    base = xp * N * N2 + r;
    stride = N2;
  } else if (p.dim == 1) {
    base = xp * N * N2 + (int64_t)(r / N) * N2 + r % N;
    stride = N;
  } else {
    base = (xp * N2 + r) * N;
    stride = 1;
  }
  double2* row = tile + threadIdx.x * (ROWS ? RW : 0);
  double2* wt = tile + warp * (ROWS ? 32 * RW : 0);
  if constexpr (ROWS) {
    const double2* g = reinterpret_cast<const double2*>(p.in) + pair0 * N;
    for (int u = lane; u < here * N; u += 32) wt[(u / N) * RW + u % N] = g[u];
    __syncwarp();
  }
  fxc x[N];
  int em0 = 1, em1 = 1;
  {
    double2 v[N];
#pragma unroll
    for (int n = 0; n < N; ++n) {
      if constexpr (ROWS) {
        const double* l = reinterpret_cast<const double*>(row);
        v[n] = make_double2(l[n], l[N + n]);
      } else {
        v[n] = on ? *reinterpret_cast<const double2*>(p.in + base + n * stride) : make_double2(0.0, 0.0);
      }
      em0 = max(em0, fx_field(v[n].x));
      em1 = max(em1, fx_field(v[n].y));
    }
#pragma unroll
    for (int n = 0; n < N; ++n) x[n] = {fx_from_double(v[n].x, em0), fx_from_double(v[n].y, em1)};
  }
  fft_fx_pre<N, false>(x);
  fft_fx_core<N>(x);
  unsigned m = 0;
  const i64* sp = p.spec + (SHIFT ? (int64_t)id * 2 * N : 0);
#pragma unroll
  for (int n = 0; n < N; ++n) {
    i64 re, im;
    if constexpr (SHIFT) {
      const i64 c = __ldg(sp + 2 * fx_freq<N>(n)), s = __ldg(sp + 2 * fx_freq<N>(n) + 1);
      re = fx_mulsym(x[n].re, c) - fx_mulsym(x[n].im, s);
      im = fx_mulsym(x[n].re, s) + fx_mulsym(x[n].im, c);
    } else {
      const i64 w = __ldg(sp + fx_freq<N>(n));
      re = -fx_mulsym(x[n].im, w);
      im = fx_mulsym(x[n].re, w);
    }
    mag_or(m, re);
    mag_or(m, im);
    x[n] = {im, re};   // (im, re): the inverse transform by the forward one
  }
  const int sh = max(0, mag_bits(m) - kFxBits);
#pragma unroll
  for (int n = 0; n < N; ++n) x[n] = {x[n].re >> sh, x[n].im >> sh};
  fft_fx_core<N>(x);
  fft_fx_post<N, false>(x);

  // back to FP64: 2^(exponent + 2 + sh) / N, the products being quarters (62-bit spectra); in two
  // factors where it is not well inside the normal numbers
  constexpr int LG = N == 8 ? 3 : (N == 16 ? 4 : 5);
  const double scale = SHIFT ? 1.0 : p.rate * (p.x_lo + id * p.h - p.center) * p.coef;
  const double mult = SHIFT ? 1.0 : scale * p.unit;
  const int e0 = fx_exponent(em0) + 2 + sh - LG, e1 = fx_exponent(em1) + 2 + sh - LG;
  const int a0 = max(-800, min(800, e0)), a1 = max(-800, min(800, e1));
  const double f0 = mult * pow2_mid(a0), f1 = mult * pow2_mid(a1);
  const double g0 = pow2_mid(max(-900, min(900, e0 - a0))), g1 = pow2_mid(max(-900, min(900, e1 - a1)));
  const bool bad0 = on && em0 == 0x7ff, bad1 = on && em1 == 0x7ff;
  const double* c = p.rows + (SHIFT ? (int64_t)id * N : 0);
#pragma unroll
  for (int n = 0; n < N; ++n) {
    double u = (double)x[n].im, w = (double)x[n].re;
    if (a0 != e0) u *= g0;
    if (a1 != e1) w *= g1;
    if constexpr (ROWS) {
      double* l = reinterpret_cast<double*>(row);
      if (!bad0) l[n] = u;
      if (!bad1) l[N + n] = w;
    } else {
      const int64_t o = base + n * stride;
      if (on && !bad0 && !bad1) {
        double2 b = make_double2(0.0, 0.0);
        if (!SHIFT && p.add) b = *reinterpret_cast<const double2*>(p.add + o);
        *reinterpret_cast<double2*>(p.out + o) = make_double2(fma(f0, u, b.x), fma(f1, w, b.y));
      } else if (on) {
        if (!bad0) p.out[o] = fma(f0, u, !SHIFT && p.add ? p.add[o] : 0.0);
        if (!bad1) p.out[o + 1] = fma(f1, w, !SHIFT && p.add ? p.add[o + 1] : 0.0);
      }
    }
  }
  if constexpr (!ROWS) {
    if (bad0) circulant_line<N>(p.in + base, SHIFT ? nullptr : p.add ? p.add + base : nullptr, p.out + base, stride, stride, c, scale);
    if (bad1) circulant_line<N>(p.in + base + 1, SHIFT ? nullptr : p.add ? p.add + base + 1 : nullptr, p.out + base + 1, stride, stride, c, scale);
  } else {
    double* l = reinterpret_cast<double*>(row);
    if (bad0) circulant_line<N>(l, nullptr, l, 1, 1, c, scale);
    if (bad1) circulant_line<N>(l + N, nullptr, l + N, 1, 1, c, scale);
    row[N] = make_double2(bad0 ? 1.0 : f0, bad1 ? 1.0 : f1);   // the two lines' scales
    __syncwarp();
    double2* g = reinterpret_cast<double2*>(p.out) + pair0 * N;
    const double2* ad = !SHIFT && p.add ? reinterpret_cast<const double2*>(p.add) + pair0 * N : nullptr;
    for (int u = lane; u < here * N; u += 32) {
      const double2 v = wt[(u / N) * RW + u % N], f = wt[(u / N) * RW + N];
      const double k = u % N < N / 2 ? f.x : f.y;
      const double2 b = ad ? ad[u] : make_double2(0.0, 0.0);
      g[u] = make_double2(fma(k, v.x, b.x), fma(k, v.y, b.y));
    }
  }
}

template <int N, bool SHIFT>
cudaError_t launch_n(const KPassParams& p, cudaStream_t s) {
  const int64_t pairs = p.nxp * (N * N / 2);
  if (p.dim == 2) k_kpass_fx<N, SHIFT, true><<<(unsigned)((pairs + 63) / 64), 64, 0, s>>>(p);
  else k_kpass_fx<N, SHIFT, false><<<(unsigned)((pairs + 127) / 128), 128, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace

// a number of magnitude at most one with 62 fractional bits, in the stored form of fx_mulsym
int64_t fx_spec_entry(double v) {
  const int64_t w = (int64_t)std::llrint(std::ldexp(v, 62));
  const int32_t lo = (int32_t)(uint32_t)(uint64_t)w;
  return (int64_t)((uint64_t)(w - lo) | (uint32_t)lo);
}

cudaError_t launch_kshift_fx(const Handle& H, void* f, int dim, const void* rows, const void* spec, cudaStream_t s) {
  if (!rows || !spec) return cudaErrorInvalidValue;
  KPassParams p{};
  p.in = static_cast<const double*>(f);
  p.out = static_cast<double*>(f);
  p.nxp = H.g.nxp;
  p.nx1 = H.g.nx[0];
  p.nx2 = H.g.nx[1];
  p.nx3 = H.g.nx[2];
  p.dim = dim;
  p.rows = static_cast<const double*>(rows);
  p.spec = static_cast<const i64*>(spec);
  switch (H.g.nk) {
    case 8: return launch_n<8, true>(p, s);
    case 16: return launch_n<16, true>(p, s);
    case 32: return launch_n<32, true>(p, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_kderiv_fx(const Handle& H, const void* in, const void* add, void* out, int dim, double coef,
                             cudaStream_t s) {
  if (!H.d_kderiv) return cudaErrorInvalidValue;
  KPassParams p{};
  p.in = static_cast<const double*>(in);
  p.add = static_cast<const double*>(add);
  p.out = static_cast<double*>(out);
  p.nxp = H.g.nxp;
  p.nx1 = H.g.nx[0];
  p.nx2 = H.g.nx[1];
  p.nx3 = H.g.nx[2];
  p.dim = dim;
  p.rows = static_cast<const double*>(H.d_kderiv);
  p.spec = reinterpret_cast<const i64*>(p.rows + H.g.nk);
  p.rate = H.kappa / H.hbar;
  p.x_lo = H.g.x_lo[dim];
  p.h = H.g.h[dim];
  p.center = H.center[dim];
  p.coef = coef;
  p.unit = M_PI * (H.g.nk / 2 - 1) / H.g.lk;   // the largest kept |xi|
  switch (H.g.nk) {
    case 8: return launch_n<8, false>(p, s);
    case 16: return launch_n<16, false>(p, s);
    case 32: return launch_n<32, false>(p, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace chasm
