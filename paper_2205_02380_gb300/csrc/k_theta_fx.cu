// P-flow of the Coulomb operator in the real form (Sec. 4), double precision: block fixed-point
// arithmetic on the integer pipe (fft_fx.cuh).
//
// The operator, its embedding (twofold padding along k1 and k2, negacyclic along k3, only the k3
// frequencies nu3 = 2j + 1/2 kept), the symbol table and the four Horner stages per x point are
// those of the single-precision kernels (k_theta_xs.cu, k_theta_pk.cu); f, the Horner base, the
// iterates and the result are FP64 and the update v = base + c_s Theta is an FP64 FMA.  In
// between, every transformed vector is a thread's registers full of 64-bit integers with a common
// exponent.
//
// Bound.  The FP64 pipe (1.7 FMAs per clock and SM, measured) held the FP64 form of this kernel at
// 94 % of what its 6.7e6 FP64 instructions per x point and stage allow at N_k = 32.  The integer
// form issues 1.00e6 warp instructions per x point and stage (N_k = 16: 1.15e5), which at four per
// clock and SM would take 13.0 ms at 16^3 x 32^3 (5.1 ms at 24^3 x 16^3); it issues in 39 % (47 %) of
// the cycles, with the integer pipe at 39 % (45 %) and the multipliers at 32 % (36 %) (ncu).  At
// N_k = 32 64-bit vectors of 32 complex values leave registers for two warps per scheduler, which
// wait for their own results (1.24 warps per issue), for the L2-resident spectrum and the symbol
// (0.67), for shared memory (0.47) and for instructions (0.47).  At N_k = 16 eight groups fit (all
// slabs of an x point at once; four groups: 12.3 ms below): four warps per scheduler, which wait at
// the block's barriers between the phases (1.61), for their own results (1.34) and for the pipes
// (1.09).  P(dt): 224.3 -> 35.5 ms at 16^3 x 32^3, 77.7 -> 11.0 ms at 24^3 x 16^3.
//
// Errors.  A vector enters a transform with 57 bits below its largest entry and leaves it with an
// error of about 3 units of the last of them, so each of the eight transforms of a stage adds
// about 2^-55 of the vector's largest entry, where the FP64 transform adds about 2^-53 of its
// root mean square; the symbol is kept with 62 bits per column.  Products are rounded to nearest: errors
// of one sign add up.  Against Theta in 80 bits from the same T, twelve seeded problems with N_k = 8, 16
// and 32: relative L2 error 0.96 to 1.00 times that of FP64 transforms.
//
// Per x point (one CTA, persistent loop over x points), per Horner stage:
//   Phase B   groups of two warps, 32 / N slabs each: rows forward along k2, columns forward along
//             k1, times sigma, columns back, rows back.  A padded transform of length 2N is two
//             transforms of length N (even outputs from x, odd ones from x e^{-i pi n/N}); one warp
//             of the group does the even halves, the other the odd ones with their twists, and
//             they swap after the first half of the columns, so both carry the same load and no
//             lane idles in a twist.  The halves of an inverse transform are added through the slab
//             buffer.
//   Phase CA  lines along k3: inverse, Theta, Horner update, and for all but the last stage the
//             forward transform of the new iterate.
// Inverse transforms run the forward code on (im, re), and all steps of both phases go through one
// copy of it: the instruction cache and the registers do not hold two.
// Layouts: spectrum G[j][k2][k1] (k1 fastest: a warp's rows and its lines along k3 are both
// consecutive), in shared memory for N <= 16 and in an L2-resident scratch otherwise; slab buffer
// V[row][2N + 1] per slab; exponents beside them, one per vector.
//
// A non-finite value anywhere in an x point's iterate makes the whole x point NaN, as a transform
// in floating point does.
#include "internal.hpp"
#include "fft_reg.cuh"
#include "fft_fx.cuh"
#include "group_bar.cuh"

namespace chasm {
namespace {

struct FxParams {
  const double* in;    // stage-0 input u_0 = in + cin2 in2 (in2 may be null)
  const double* base;  // Horner base base + cbase2 base2 (base2 may be null), or null (0)
  const double* in2;
  const double* base2;
  double cin2, cbase2;
  double* out;         // result of the last stage; may alias in, in2, base and base2
  int64_t nxp;
  const i64* sig;      // [nxp][N][2N][2N] symbol, fixed point (fx_symbol)
  int64_t sig_xs;      // elements per x point of sig (0: one table for every x point)
  const int16_t* sigx; // [nxp][N][2][2N] its exponents
  int64_t sigx_xs;
  int nst;             // stages, 1..4
  double coef[4];      // c_s per stage
  fxc* G;              // per-CTA spectrum scratch when it is not in shared memory
  int* late;           // set when a wait ran out (chasm_moments reports it)
};

template <int N>
struct FxCfg {
  static constexpr int L = 2 * N;
  static constexpr int SPW = 32 / N;                 // slabs per group
  static constexpr int NG = N == 8 ? 2 : (N == 16 ? 8 : 4);   // groups of two warps
  static constexpr int NT = 64 * NG;
  static constexpr int NW = NT / 32;
  static constexpr bool GSM = N <= 16;               // spectrum in shared memory
  static constexpr int VR = L + 1;                   // slab-buffer row (odd: conflict-free 16-byte columns)
  static constexpr int VSZ = SPW * N * VR;           // slab buffers of a group
  static constexpr int TROW = N / 2 + 1;             // line staging row, 16-byte units
  static constexpr size_t v_bytes = (size_t)NG * VSZ * sizeof(fxc);
  static constexpr size_t g_bytes = GSM ? (size_t)N * N * N * sizeof(fxc) : 0;
  // exA, exG [N][N]; ex1, ex2 [NG][64]; exP [NG][64]; etA, etG [N]; flag [2] (and two spare); three barriers per group
  static constexpr size_t e_bytes = (2 * N * N + 2 * NG * 64) * sizeof(int2) + (NG * 64 + 2 * N + 4) * sizeof(int) + NG * 24;
  static constexpr size_t smem_bytes = v_bytes + g_bytes + e_bytes;
  static_assert(NG * VSZ * sizeof(fxc) / NW >= 32 * TROW * 16, "line staging fits the slab buffers");
};

template <int N>
__device__ __forceinline__ int seg_max(int v) {   // over the aligned groups of N lanes
#pragma unroll
  for (int o = N / 2; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// exponent to which vectors with exponents E and top bits E + b are aligned (never below an E: a
// shift to the left would add no information)
__device__ __forceinline__ int align_exp(int emax, int topmax, int bits) { return max(emax, topmax - bits); }
__device__ __forceinline__ int shift_of(int et, int e) { return min(63, et - e); }

template <bool GSM>
__device__ __forceinline__ fxc g_get(const fxc* p, uint64_t pol) {
  if constexpr (GSM) {
    return *p;
  } else {
    fxc v;
    asm volatile("ld.global.L2::cache_hint.v2.b64 {%0, %1}, [%2], %3;" : "=l"(v.re), "=l"(v.im) : "l"(p), "l"(pol) : "memory");
    return v;
  }
}
template <bool GSM>
__device__ __forceinline__ void g_put(fxc* p, fxc v, uint64_t pol) {
  if constexpr (GSM) *p = v;
  else asm volatile("st.global.L2::cache_hint.v2.b64 [%0], {%1, %2}, %3;" ::"l"(p), "l"(v.re), "l"(v.im), "l"(pol) : "memory");
}
__device__ __forceinline__ i64 ld_sym(const i64* p, uint64_t pol) {
  i64 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.b64 %0, [%1], %2;" : "=l"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ void prefetch_l2(const void* src, unsigned bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// The lines of one warp (N doubles each, line of lane t at src + off(t)) into a staging buffer,
// row t the line of lane t, so that every global access of the warp covers whole lines;
// src2 != null: src + c2 src2.
template <int N, bool X2, class Off>
__device__ __forceinline__ void stage_lines(const double* src, const double* src2, double c2, Off&& off, double2* T) {
  constexpr int Q = N / 2, TR = FxCfg<N>::TROW, PER = 32 / Q;   // 16-byte pieces per line, lines per access
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int t = q * PER + lane / Q, e = lane % Q;
    double2 v = __ldcs(reinterpret_cast<const double2*>(src + off(t)) + e);
    if (X2 && src2) {
      const double2 w = __ldcs(reinterpret_cast<const double2*>(src2 + off(t)) + e);
      v.x = fma(c2, w.x, v.x);
      v.y = fma(c2, w.y, v.y);
    }
    T[t * TR + e] = v;
  }
  __syncwarp();
}
template <int N>
__device__ __forceinline__ void clear_line(double* row) {
#pragma unroll
  for (int n = 0; n < N; ++n) row[n] = 0.0;
}
template <int N, class Off>
__device__ __forceinline__ void unstage_lines(double* dst, Off&& off, const double2* T) {
  constexpr int Q = N / 2, TR = FxCfg<N>::TROW, PER = 32 / Q;
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const int t = q * PER + lane / Q, e = lane % Q;
    __stcs(reinterpret_cast<double2*>(dst + off(t)) + e, T[t * TR + e]);
  }
  __syncwarp();
}

// The k3 twist e^{-i pi n / (2N)} of a real line (in shared memory), as integers with kFxBits
// bits below the line's largest entry, whose exponent field is em; returns their exponent,
// 1 << 30 when an entry is not finite.
template <int N>
__device__ __forceinline__ int quantise_line(const double* row, int em, fxc (&x)[N]) {
  xfor<0, N>([&](auto I) {
    constexpr int n = decltype(I)::value;
    asm volatile("" ::: "memory");
    const double v = row[n];
    const i64 w = fx_from_double(v, em);
    if constexpr (n == 0) {
      x[n] = {w, 0};
    } else {
      // angle in (0, pi/2): cos and sin of it, each from an angle of at most pi/4
      constexpr bool up = 8 * n > 4 * N;   // beyond pi/4: cos and sin of the complement
      constexpr int k = up ? N - n : n;
      constexpr u64 c = up ? FxK<k, 4 * N>::sin : FxK<k, 4 * N>::cos;
      constexpr u64 s = up ? FxK<k, 4 * N>::cos : FxK<k, 4 * N>::sin;
      x[n] = {fx_mul<c>(w), -fx_mul<s>(w)};
    }
  });
  return em == 0x7ff ? 1 << 30 : fx_exponent(em);
}

// sin phi Re z + cos phi Im z (the real part of -i e^{i phi} ... with the symbol's factor i taken
// out), or cos phi Re z - sin phi Im z for a real spectrum; phi = pi n / (2N)
template <int N, int n, bool REAL>
__device__ __forceinline__ i64 untwist(i64 re, i64 im) {
  if constexpr (n == 0) {
    return REAL ? re : im;
  } else {
    constexpr bool up = 8 * n > 4 * N;
    constexpr int k = up ? N - n : n;
    constexpr u64 c = up ? FxK<k, 4 * N>::sin : FxK<k, 4 * N>::cos;
    constexpr u64 s = up ? FxK<k, 4 * N>::cos : FxK<k, 4 * N>::sin;
    return REAL ? fx_mul<c>(re) - fx_mul<s>(im) : fx_mul<c>(im) + fx_mul<s>(re);
  }
}

// ex[i][k1] (exponent, top bit) of the N vectors gathered for each k1 -> ex[i][k1].x = shift of
// vector i, et[k1] = their common exponent; eight threads per k1
template <int N>
__device__ __forceinline__ void align_all(int2* ex, int* et, int bits) {
  const int t = threadIdx.x;
  if (t < 8 * N) {
    const int k1 = t / 8, p = t % 8;
    int em = -(1 << 29), tm = -(1 << 29);
#pragma unroll
    for (int i = p; i < N; i += 8) {
      em = max(em, ex[i * N + k1].x);
      tm = max(tm, ex[i * N + k1].y);
    }
    em = seg_max<8>(em);
    tm = seg_max<8>(tm);
    const int e = align_exp(em, tm, bits);
#pragma unroll
    for (int i = p; i < N; i += 8) ex[i * N + k1].x = shift_of(e, ex[i * N + k1].x);
    if (p == 0) et[k1] = e;
  }
}

// Shared memory of a CTA and a thread's place in it.
template <int N>
struct FxShared {
  fxc* V;                       // the group's slab buffers
  fxc* G;                       // spectrum
  int2 *exA, *exG, *ex1, *ex2;  // lines [k2][k1], slab rows [j][k1], the group's rows and columns
  int *exP, *etA, *etG, *flag;
  unsigned bar;                 // the group's barriers: read, written, both (8 bytes each)
  double2* T;                   // the warp's line staging (in the slab buffers)
  int warp, lane, grp, wb, ln, sub;
  __device__ __forceinline__ FxShared(unsigned char* smem, fxc* Gglobal) {
    using C = FxCfg<N>;
    const int tid = threadIdx.x;
    warp = tid >> 5;
    lane = tid & 31;
    grp = warp >> 1;
    wb = warp & 1;              // second warp of the group
    ln = lane % N;
    sub = lane / N;
    V = reinterpret_cast<fxc*>(smem) + grp * C::VSZ;
    G = C::GSM ? reinterpret_cast<fxc*>(smem + C::v_bytes) : Gglobal + (size_t)blockIdx.x * (N * N * N);
    exA = reinterpret_cast<int2*>(smem + C::v_bytes + C::g_bytes);
    exG = exA + N * N;
    ex1 = exG + N * N + grp * 64;
    ex2 = exG + N * N + C::NG * 64 + grp * 64;
    int* q = reinterpret_cast<int*>(exG + N * N + 2 * C::NG * 64);
    exP = q + grp * 64;
    etA = q + C::NG * 64;
    etG = etA + N;
    flag = etG + N;
    bar = sm_addr(flag + 4) + grp * 24;
    T = reinterpret_cast<double2*>(smem + (size_t)warp * (C::v_bytes / C::NW / 16 * 16));
  }
};

// The transforms of a stage, in the order of their data: Phase B per group of slabs (rows forward,
// the first and the second half of the columns forward and back, rows back), Phase CA per group
// of lines (back, forward).
enum FxBar { kRead = 0, kWritten = 8, kBoth = 16 };
enum FxStep { kRowF, kColF0, kColB0, kColF1, kColB1, kRowB, kLineB, kLineF };

// The halves of a transform are exchanged through the slab buffer three times per group of slabs
// (columns twice, rows): the odd half signals that it has read its input (barrier kRead), the even
// half then puts its result there and signals that (kWritten), the odd half adds its own.  Each
// barrier's phases are told apart by their parity: a phase's one arrival follows its partner's wait
// for the phase before.  `turn` counts the exchanges.
// One phase of stage st (st = -1: only the forward lines of the input) on x point xp.  All steps go
// through one copy of the transform's middle part: a copy per step would not fit the
// instruction cache, and two of them already cost 400 bytes of spilled registers (53.8 against
// 49.3 ms at 16^3 x 32^3).
// REAL: real spectrum of an even kernel (the plain TKM convolution).
template <int N, bool X2, bool REAL>
__device__ __forceinline__ void fx_phase(const FxParams& p, int64_t xp, int st, bool lines, int& turn) {
  using C = FxCfg<N>;
  constexpr int L = C::L, SPW = C::SPW, NG = C::NG, NW = C::NW, VR = C::VR, N2 = N * N, N3 = N * N * N;
  constexpr bool GSM = C::GSM;
  constexpr bool FW = N == 8;   // P(dt) at 24^3 x 8^3 1.425 -> 1.410 ms, at 24^3 x 16^3 11.03 -> 11.34
  extern __shared__ __align__(16) unsigned char smem[];
  const FxShared<N> S(smem, p.G);
  const uint64_t pol = l2_keep_policy(), spol = l2_stream_policy();
  const bool last = st == p.nst - 1, bad = *S.flag != 0;
  double cs = p.coef[0];   // static indexing keeps the parameter block out of local memory
#pragma unroll
  for (int q = 1; q < 4; ++q)
    if (q == st) cs = p.coef[q];
  if (!REAL) cs = -cs;
  if (bad) cs = __longlong_as_double(0x7ff8000000000000LL);
  double* row = reinterpret_cast<double*>(S.T + S.lane * C::TROW);   // this lane's line
  const int first = lines ? (st < 0 ? kLineF : kLineB) : kRowF;
  const int final = lines ? (last ? kLineB : kLineF) : kRowB;
  const int nitem = lines ? N2 / 32 : N / SPW;   // items: groups of 32 lines, groups of slabs
#pragma unroll 1
  for (int item = lines ? S.warp : S.grp; item < nitem; item += lines ? NW : NG) {
    const int s0 = item * SPW;
    if (!lines && S.lane == 0 && S.wb == 0) {   // the symbol slabs this group needs next, into L2
      const int sn = s0 + NG * SPW < N ? s0 + NG * SPW : S.grp * SPW;
      const int64_t xn = s0 + NG * SPW < N || st + 1 < p.nst ? xp : xp + gridDim.x;
      if (xn < p.nxp)
        prefetch_l2(p.sig + xn * p.sig_xs + sn * (int64_t)(L * L), SPW * L * L * sizeof(i64));
    }
    // global offset of the line of lane t in a line item: k1 = t % N, k2 = item SPW + t / N
    auto off = [&](int t) { return (size_t)xp * N3 + ((size_t)(t % N) * N + item * SPW + t / N) * N; };
    fxc x[N];
    int E = 0, em = 1;
#pragma unroll 1
    for (int step = first; step <= final; ++step) {
      const bool odd = !lines && (step < 3) == (S.wb == 1);   // this warp's half of the padded transform
      const bool inv = step == kColB0 || step == kColB1 || step == kRowB || step == kLineB;
      const int rnd = step >= kColF1;
      const int cc = S.lane + 32 * rnd, sc = cc / L, c = cc % L;
      if (step == kRowF) {
        const fxc* g = S.G + (size_t)(s0 + S.sub) * N2 + S.ln;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const fxc v = g_get<GSM>(g + n * N, pol);
          const int s = S.exA[n * N + S.ln].x;
          x[n] = {v.re >> s, v.im >> s};
        }
        E = S.etA[S.ln];
      } else if (step == kColF0 || step == kColF1) {
        const int2 e = S.ex1[(sc * 2 + c / N) * N + S.ln];
        E = align_exp(seg_max<N>(e.x), seg_max<N>(e.y), kFxBits);
        const int sh = shift_of(E, e.x);
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const fxc v = S.V[(sc * N + n) * VR + c];
          const int s = __shfl_sync(0xffffffffu, sh, (S.lane & ~(N - 1)) + n);
          x[n] = {v.re >> s, v.im >> s};
        }
        if (odd) mb_arrive(S.bar + kRead);   // the columns' entries are read: their place may be written
      } else if (step == kRowB) {
        const int2 e0 = S.ex2[S.sub * L + S.ln], e1 = S.ex2[S.sub * L + N + S.ln];
        E = align_exp(seg_max<N>(max(e0.x, e1.x)), seg_max<N>(max(e0.y, e1.y)), kFxBits - 1);
        const int sh = shift_of(E, odd ? e1.x : e0.x);
        const fxc* row = S.V + (S.sub * N + S.ln) * VR + (odd ? N : 0);
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const fxc v = row[fx_freq<N>(n)];
          const int s = __shfl_sync(0xffffffffu, sh, (S.lane & ~(N - 1)) + fx_freq<N>(n));
          x[n] = {v.re >> s, v.im >> s};
        }
        if (odd) mb_arrive(S.bar + kRead);
      } else if (step == kLineB) {
        if (p.base) stage_lines<N, X2>(p.base, p.base2, p.cbase2, off, S.T);
        else clear_line<N>(row);
        const fxc* g = S.G + (size_t)(item * SPW + S.sub) * N + S.ln;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const fxc q = g_get<GSM>(g + (size_t)fx_freq<N>(n) * N2, pol);
          const int s = S.exG[fx_freq<N>(n) * N + S.ln].x;
          x[n] = {q.im >> s, q.re >> s};
        }
        E = S.etG[S.ln];
      } else if (step == kLineF) {
        if (st < 0) {   // u_0 (with in2: the LPC1 predictor)
          stage_lines<N, X2>(p.in, p.in2, p.cin2, off, S.T);
          em = 1;
#pragma unroll
          for (int n = 0; n < N; ++n) em = max(em, fx_field(row[n]));
        }
        E = quantise_line<N>(row, em, x);
        if (E == 1 << 30) *S.flag = 1;
        __syncwarp();
      }
      if (!inv) {
        if (odd) fft_fx_pre<N, true>(x);
        else fft_fx_pre<N, false>(x);
      }
      fft_fx_core<N>(x);
      if (inv) {
        if (odd) fft_fx_post<N, true>(x);
        else fft_fx_post<N, false>(x);
      }

      if (step == kRowF) {
        fxc* row = S.V + (S.sub * N + S.ln) * VR + (odd ? N : 0);
        unsigned m = 0;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          mag_or(m, x[n].re);
          mag_or(m, x[n].im);
          row[fx_freq<N>(n)] = x[n];
        }
        S.ex1[(S.sub * 2 + (odd ? 1 : 0)) * N + S.ln] = make_int2(E, E + mag_bits(m));
        mb_arrive(S.bar + kBoth);
        mb_wait<FW>(S.bar + kBoth, 0, S.flag);
      } else if (step == kColF0 || step == kColF1) {
        const int64_t j = s0 + sc;
        const i64* sg = p.sig + xp * p.sig_xs + ((j * L + (odd ? N : 0)) * L + c);
        const int es = p.sigx[xp * p.sigx_xs + (j * 2 + (odd ? 1 : 0)) * L + c];
        unsigned m = 0;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          const i64 w = ld_sym(sg + (size_t)fx_freq<N>(n) * L, spol);
          const i64 re = fx_mulsym(x[n].re, w), im = fx_mulsym(x[n].im, w);
          mag_or(m, re);
          mag_or(m, im);
          x[n] = {im, re};   // (im, re): the inverse transform by the forward one
        }
        const int s = max(0, mag_bits(m) - kFxBits);
#pragma unroll
        for (int n = 0; n < N; ++n) x[n] = {x[n].re >> s, x[n].im >> s};
        E += es + 64 + s;
      } else if (step == kColB0 || step == kColB1) {
        fxc* col = S.V + (size_t)sc * N * VR + c;
        if (!odd) {
          mb_wait<FW>(S.bar + kRead, turn, S.flag);
#pragma unroll
          for (int n = 0; n < N; ++n) col[n * VR] = x[n];
          S.exP[cc] = E;
          mb_arrive(S.bar + kWritten);
        } else {
          mb_wait<FW>(S.bar + kWritten, turn, S.flag);
          const int ep = S.exP[cc], et = max(ep, E) + 1;
          const int s0_ = shift_of(et, ep), s1_ = shift_of(et, E);
          unsigned m = 0;
#pragma unroll
          for (int n = 0; n < N; ++n) {
            const fxc q = col[n * VR];
            const fxc r = {(x[n].re >> s1_) + (q.re >> s0_), (x[n].im >> s1_) + (q.im >> s0_)};
            mag_or(m, r.re);
            mag_or(m, r.im);
            col[n * VR] = r;
          }
          S.ex2[cc] = make_int2(et, et + mag_bits(m));
        }
        ++turn;
        if (step == kColB1) {
          mb_arrive(S.bar + kBoth);
          mb_wait<FW>(S.bar + kBoth, 1, S.flag);
        }
      } else if (step == kRowB) {
        fxc* row = S.V + (S.sub * N + S.ln) * VR;
        if (!odd) {
#pragma unroll
          for (int n = 0; n < N; ++n) row[n] = x[n];
          mb_arrive(S.bar + kWritten);
          mb_wait<FW>(S.bar + kRead, turn, S.flag);
        } else {
          mb_wait<FW>(S.bar + kWritten, turn, S.flag);
          fxc* g = S.G + (size_t)(s0 + S.sub) * N2 + S.ln;
          unsigned m = 0;
#pragma unroll
          for (int n = 0; n < N; ++n) {
            const fxc q = row[n];
            const fxc r = {x[n].im + q.im, x[n].re + q.re};
            mag_or(m, r.re);
            mag_or(m, r.im);
            g_put<GSM>(g + n * N, r, pol);
          }
          S.exG[(s0 + S.sub) * N + S.ln] = make_int2(E, E + mag_bits(m));
        }
        ++turn;
      } else if (step == kLineB) {
        // c 2^E as one factor where 2^E is well inside the normal numbers, else in two
        const int em_ = max(-800, min(800, E));
        const double c2 = cs * pow2_mid(em_), rest = pow2_mid(max(-900, min(900, E - em_)));
        em = 1;
        xfor<0, N>([&](auto I) {
          constexpr int n = decltype(I)::value;
          double th = (double)untwist<N, n, REAL>(x[n].im, x[n].re);
          if (em_ != E) th *= rest;
          const double v = fma(c2, th, row[n]);
          em = max(em, fx_field(v));
          row[n] = v;
          asm volatile("" ::: "memory");   // one entry after the other: there are no registers to spare
        });
        if (last) unstage_lines<N>(p.out, off, S.T);
      } else {   // kLineF
        fxc* g = S.G + (size_t)(item * SPW + S.sub) * N + S.ln;
        unsigned m = 0;
#pragma unroll
        for (int n = 0; n < N; ++n) {
          mag_or(m, x[n].re);
          mag_or(m, x[n].im);
          g_put<GSM>(g + (size_t)fx_freq<N>(n) * N2, x[n], pol);
        }
        S.exA[(item * SPW + S.sub) * N + S.ln] = make_int2(E, E + mag_bits(m));
      }
    }
  }
}

template <int N, bool X2, bool REAL>
__global__ void __launch_bounds__(FxCfg<N>::NT, 1) k_theta_fx(const FxParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  const FxShared<N> S(smem, p.G);
  if (threadIdx.x < FxCfg<N>::NG) {
    const unsigned b = sm_addr(S.flag + 4) + threadIdx.x * 24;
    mb_init(b + kRead, 1);
    mb_init(b + kWritten, 1);
    mb_init(b + kBoth, 2);
  }
  // flag[0]: this x point becomes NaN; flag[1]: an exchange never came, no results from then on rather
  // than wrong ones
  if (threadIdx.x == 0) S.flag[1] = 0;
  int turn = 0;
  for (int64_t xp = blockIdx.x; xp < p.nxp; xp += gridDim.x) {
    if (threadIdx.x == 0) S.flag[0] = S.flag[1];
    __syncthreads();
#pragma unroll 1
    for (int ph = 1; ph < 2 * p.nst + 2; ++ph) {   // lines of the input, then slabs and lines per stage
      const int st = ph / 2 - 1;
      const bool lines = ph & 1;
      fx_phase<N, X2, REAL>(p, xp, st, lines, turn);
      __syncthreads();
      if (st < p.nst - 1 || !lines) {
        align_all<N>(lines ? S.exA : S.exG, lines ? S.etA : S.etG, kFxBits);
        __syncthreads();
      }
    }
  }
  if (threadIdx.x == 0 && S.flag[1]) *p.late = 1;
}

// sigma (FP64, [x][j][s1][s2]) -> fixed point in place: the N values of a column (one parity of
// s1, one s2) get the exponent that puts the largest at 2^61..2^62; the low word is stored as a
// signed number with its carry in the high word (fx_mulsym).  One thread per column; a warp's
// loads are consecutive in s2.
__global__ void k_fx_symbol(i64* __restrict__ sig, int16_t* __restrict__ ex, int N, int64_t ncol) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ncol) return;
  const int L = 2 * N;
  const int s2 = (int)(t % L);
  const int64_t r = t / L;   // (x, j, half)
  i64* col = sig + r * (int64_t)N * L + s2;
  int em = 1;
  for (int n = 0; n < N; ++n) em = max(em, (int)(((u64)col[(int64_t)n * L] >> 52) & 0x7ff));
  for (int n = 0; n < N; ++n) {
    const u64 b = (u64)col[(int64_t)n * L];
    const int e = (int)((b >> 52) & 0x7ff);
    const u64 m = ((b & 0xfffffffffffffULL) | (e ? 0x10000000000000ULL : 0)) << 9;
    const int s = min(63, em - max(e, 1));
    const i64 w = (i64)b < 0 ? -(i64)(m >> s) : (i64)(m >> s);
    const int lo = (int)(unsigned)w;
    col[(int64_t)n * L] = (i64)(((u64)(unsigned)((w - lo) >> 32)) << 32 | (unsigned)lo);
  }
  ex[t] = (int16_t)(em - 1023 - 61);
}

template <int N>
void plan_fx_n(int64_t nxp, int num_sms, ThetaPlan* pl) {
  using C = FxCfg<N>;
  cudaFuncSetAttribute(k_theta_fx<N, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem_bytes);
  cudaFuncSetAttribute(k_theta_fx<N, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem_bytes);
  cudaFuncSetAttribute(k_theta_fx<N, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::smem_bytes);
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_theta_fx<N, false, false>, C::NT, C::smem_bytes) != cudaSuccess || nb < 1)
    nb = 1;
  pl->cluster = 0;
  pl->blocks = (int)std::min<int64_t>(nxp, (int64_t)nb * num_sms);
  pl->scratch_bytes = C::GSM ? 0 : (size_t)pl->blocks * N * N * N * sizeof(fxc);
}

template <int N>
cudaError_t launch_fx_n(const Handle& H, const void* in, const void* base, void* out, int nst,
                        const double* coef, const XsExtra& x, cudaStream_t s) {
  using C = FxCfg<N>;
  FxParams p;
  p.in = static_cast<const double*>(in);
  p.base = static_cast<const double*>(base);
  p.in2 = static_cast<const double*>(x.in2);
  p.base2 = static_cast<const double*>(x.base2);
  p.cin2 = x.cin2;
  p.cbase2 = x.cbase2;
  p.out = static_cast<double*>(out);
  p.nxp = H.g.nxp;
  const int64_t per = (int64_t)N * C::L * C::L;
  p.sig = static_cast<const i64*>(x.sig ? x.sig : H.d_sig);
  p.sigx = reinterpret_cast<const int16_t*>(p.sig + (x.sig ? 1 : H.g.nxp) * per);
  p.sig_xs = x.sig ? 0 : per;
  p.sigx_xs = x.sig ? 0 : (int64_t)N * 2 * C::L;
  p.nst = nst;
  for (int q = 0; q < 4; ++q) p.coef[q] = q < nst ? coef[q] : 0.0;
  p.G = static_cast<fxc*>(H.d_scratch);
  p.late = late_word(H);
  if (x.real_symbol) {
    if (x.in2 || x.base2) return cudaErrorInvalidValue;
    k_theta_fx<N, false, true><<<H.theta.blocks, C::NT, C::smem_bytes, s>>>(p);
  } else if (x.in2 || x.base2) {
    k_theta_fx<N, true, false><<<H.theta.blocks, C::NT, C::smem_bytes, s>>>(p);
  } else {
    k_theta_fx<N, false, false><<<H.theta.blocks, C::NT, C::smem_bytes, s>>>(p);
  }
  return cudaGetLastError();
}

}  // namespace

size_t fx_symbol_extra_bytes(int nk, int64_t nxp) { return (size_t)nxp * nk * 4 * nk * sizeof(int16_t); }

cudaError_t fx_symbol(void* sig, int nk, int64_t nxp, cudaStream_t s) {
  const int64_t ncol = nxp * nk * 4 * nk;
  i64* t = static_cast<i64*>(sig);
  int16_t* ex = reinterpret_cast<int16_t*>(t + ncol * nk);
  k_fx_symbol<<<(unsigned)((ncol + 255) / 256), 256, 0, s>>>(t, ex, nk, ncol);
  return cudaGetLastError();
}

void theta_fx_plan(int nk, int64_t nxp, int num_sms, ThetaPlan* pl) {
  if (nk == 8) plan_fx_n<8>(nxp, num_sms, pl);
  else if (nk == 16) plan_fx_n<16>(nxp, num_sms, pl);
  else plan_fx_n<32>(nxp, num_sms, pl);
}

cudaError_t launch_theta_fx(const Handle& H, const void* in, const void* base, void* out, int nst,
                            const double* coef, cudaStream_t s, const XsExtra& x) {
  switch (H.g.nk) {
    case 8: return launch_fx_n<8>(H, in, base, out, nst, coef, x, s);
    case 16: return launch_fx_n<16>(H, in, base, out, nst, coef, x, s);
    case 32: return launch_fx_n<32>(H, in, base, out, nst, coef, x, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace chasm
