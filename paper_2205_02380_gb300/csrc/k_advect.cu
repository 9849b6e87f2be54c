// Spatial advection A(tau): f(x, k) <- f(x - hbar k tau / m, k)   (Eq. 2.6, Sec. 3)
//
// The tensor-product spline of Eq. 3.9 and the 64-tap evaluation of Eq. 3.10 are computed in
// sum-factorised form: the 3-D operator is (E1 S1)(E2 S2)(E3 S3), where S_d is the PMBC-closed
// 1-D spline transform along x_d (Eq. 3.5 closure + Hermite-closed tridiagonal solve, step (5) of
// Sec. 3.1.2) and E_d the 4-tap evaluation at the feet x_j - alpha_d h_d (Eqs. 3.7-3.8).  Operators
// acting on different dimensions commute, so three in-place passes, one per x-dimension, give
// exactly the 64-term sum (up to rounding order) without ever storing the (N+3)^3 coefficient
// tensor.
//
// One thread owns one line: fixed k (the contiguous index, so a warp reads consecutive k and every
// load/store is a coalesced transaction) and fixed other two x indices; in the FP32 register
// kernel a thread owns the lines of two adjacent k and moves both with 8-byte accesses (each warp
// access 256 contiguous bytes, as in FP64).  The thread loads its nx values, forms the PMBC
// closure phi_L, phi_R, runs the constant-LU Thomas sweep, evaluates the 4-tap stencil and writes
// the nx new values back over the old ones (no other thread touches the line, so in place is
// safe).
//
// Closure precision.  FP64 form: native FP64.  FP32-mixed form: the closure dot products are
// accumulated in compensated FP32-pair arithmetic (error-free products by FMA, Knuth's two-sum;
// about 48 significant bits), i.e. at FP64-class precision without the FP64 pipe, which on GB300
// delivers 1/64 of the FP32 rate and otherwise bounds this pass.  Everything else is FP32.
//
// One kernel for the three dimensions of the smallest grids (k_advect_box), and per dimension:
// k_advect_reg keeps the line in registers (integer shift in [-2, 1], the usual case
// since |alpha| < 1; line length a compile-time constant from {16, 24, 32, 48, 64}, and in FP32
// any length up to 64, in classes of four); k_advect_smem is the general fallback with the line
// in shared memory (column layout, element e of thread t at e*B + t, conflict-free).
// FP32 lengths between the constants ran in shared memory before, bound by its round trips: A(tau)
// on 20^3, 36^2 x 16 and 60^2 x 16 x 32^3 at 2.37, 3.11 and 2.79 TB/s per pass, now 5.63, 5.35 and
// 5.03 (32 points: 6.11).  FP64 is bound by the FP64 pipe, where the padded slots cost more than
// shared memory does: ragged registers 661, 807 and 868 GB/s, shared memory 985, 907 and 893.
#include <cstring>

#include "internal.hpp"

namespace chasm {
namespace {

template <typename T>
struct AdvParams {
  T* f;
  int64_t n_lines;
  int64_t kvol;       // nk^3
  int64_t s_d;        // stride along the advected dimension
  int64_t s_a, s_b;   // strides of the two other x dimensions
  int n;              // points along the advected dimension
  int n_b;            // extent of the second "other" dimension
  int kdiv;           // k_d = (kidx / kdiv) % nk
  int nk;
  int J;              // stencil length (<= n); the coefficient arrays are zero-padded to n
  double h;
  float hf, h2f;      // h and 2h rounded to FP32 (FP32-mixed closure terms)
  const T* clos;      // closure coefficients (see ClosureFmt)
  const T* cprime;    // Thomas c'_i, i = 0..N
  const T* mult;      // Thomas 1/(b_i - a_i c'_{i-1}), i = 0..N
  const T* w;         // [nk][4] (b4, b3, b2, b1)
  const int* ns;      // [nk] floor(alpha)
};

// ---- closure accumulators ----
// FP64: c+ at clos[j], c- at clos[n + j].
// FP32: c+ hi/lo at clos[j], clos[n + j]; c- hi/lo at clos[2n + j], clos[3n + j].
struct DF {           // unevaluated sum hi + lo
  float hi, lo;
};
__device__ __forceinline__ void df_acc(DF& s, float x, float chi, float clo) {
  const float p = x * chi;
  float e = fmaf(x, chi, -p);          // x * chi = p + e exactly
  e = fmaf(x, clo, e);
  const float t = s.hi + p;            // two-sum s.hi + p = t + err
  const float bb = t - s.hi;
  const float err = (s.hi - (t - bb)) + (p - bb);
  s.hi = t;
  s.lo += err + e;
}

template <typename T>
struct Closure;

template <>
struct Closure<double> {
  double L = 0.0, R = 0.0;
  __device__ __forceinline__ void add(const double* c, int n, int j, double phiL, double phiR) {
    L = fma(__ldg(c + j), phiL, L);
    R = fma(__ldg(c + n + j), phiR, R);
  }
  // 3 phi_0 + h phi_L, 3 phi_N - h phi_R, and the ghost offsets 2 h phi_L, 2 h phi_R
  __device__ __forceinline__ double d0(double phi0, double h) const { return 3.0 * phi0 + h * L; }
  __device__ __forceinline__ double dN(double phiN, double h) const { return 3.0 * phiN - h * R; }
  __device__ __forceinline__ double gl(double eta1, double h) const { return eta1 - 2.0 * h * L; }
  __device__ __forceinline__ double gr(double etaNm1, double h) const { return etaNm1 + 2.0 * h * R; }
};

template <>
struct Closure<float> {
  DF L{0.f, 0.f}, R{0.f, 0.f};
  __device__ __forceinline__ void add(const float* c, int n, int j, float phiL, float phiR) {
    df_acc(L, phiL, __ldg(c + j), __ldg(c + n + j));
    df_acc(R, phiR, __ldg(c + 2 * n + j), __ldg(c + 3 * n + j));
  }
  __device__ __forceinline__ float d0(float phi0, float hf) const {
    return fmaf(hf, L.hi, fmaf(hf, L.lo, 3.0f * phi0));
  }
  __device__ __forceinline__ float dN(float phiN, float hf) const {
    return fmaf(-hf, R.hi, fmaf(-hf, R.lo, 3.0f * phiN));
  }
  __device__ __forceinline__ float gl(float eta1, float h2f) const {
    return fmaf(-h2f, L.hi, fmaf(-h2f, L.lo, eta1));
  }
  __device__ __forceinline__ float gr(float etaNm1, float h2f) const {
    return fmaf(h2f, R.hi, fmaf(h2f, R.lo, etaNm1));
  }
};

// Closure stencils and Thomas factors of the register kernel, passed by value in the kernel's
// parameter block: every index is a compile-time constant there, so each coefficient is a
// constant-bank operand of its FMA instead of a load per line.
constexpr int kRegMaxNx = 64;
template <typename T>
struct AdvTabs;
template <>
struct AdvTabs<float> {
  float c[4][kRegMaxNx];     // c+ hi, c+ lo, c- hi, c- lo (zero-padded)
  float lu[2][kRegMaxNx];    // c'_i, 1 / pivot_i
};
template <>
struct AdvTabs<double> {
  double c[2][kRegMaxNx];    // c+, c-
  double lu[2][kRegMaxNx];
};

// The closure stencils decay like |sqrt(3) - 2|^j (about 0.27^j): from tap kClosHead on the
// coefficients are below 1e-5 of the leading ones, so the FP32 rounding of each tail product
// (added to the low part) is below about 1e-12 of the data's scale over h; the leading taps are
// accumulated error-free.
constexpr int kClosHead = 10;
template <int NX>
__device__ __forceinline__ void closure_tab(Closure<float>& cl, const AdvTabs<float>& tb, int j,
                                            float phiL, float phiR) {
  if (j < kClosHead) {
    df_acc(cl.L, phiL, tb.c[0][j], tb.c[1][j]);
    df_acc(cl.R, phiR, tb.c[2][j], tb.c[3][j]);
  } else {
    cl.L.lo = fmaf(phiL, tb.c[0][j], cl.L.lo);
    cl.R.lo = fmaf(phiR, tb.c[2][j], cl.R.lo);
  }
}
template <int NX>
__device__ __forceinline__ void closure_tab(Closure<double>& cl, const AdvTabs<double>& tb, int j,
                                            double phiL, double phiR) {
  cl.L = fma(tb.c[0][j], phiL, cl.L);
  cl.R = fma(tb.c[1][j], phiR, cl.R);
}

// the h arguments of the closure terms in the storage precision
template <typename T>
__device__ __forceinline__ T hval(const AdvParams<T>& p);
template <>
__device__ __forceinline__ double hval<double>(const AdvParams<double>& p) { return p.h; }
template <>
__device__ __forceinline__ float hval<float>(const AdvParams<float>& p) { return p.hf; }
template <typename T>
__device__ __forceinline__ T h2val(const AdvParams<T>& p);
template <>
__device__ __forceinline__ double h2val<double>(const AdvParams<double>& p) { return p.h; }
template <>
__device__ __forceinline__ float h2val<float>(const AdvParams<float>& p) { return p.h2f; }

template <typename T>
__device__ __forceinline__ void line_setup(const AdvParams<T>& p, int64_t line, T*& src, int& kd) {
  const int64_t kidx = line % p.kvol;
  const int64_t outer = line / p.kvol;
  const int64_t ia = outer / p.n_b, ib = outer % p.n_b;
  src = p.f + ia * p.s_a + ib * p.s_b + kidx;
  kd = (int)((kidx / p.kdiv) % p.nk);
}

// ---- register kernel ----
// out_j = w0 eta_{j-S-2} + w1 eta_{j-S-1} + w2 eta_{j-S} + w3 eta_{j-S+1}; slot of eta_nu = nu+1.
// st(j, out_j) writes the result (global memory or a shared-memory tile).
template <typename T, int NX, int S, class St>
__device__ __forceinline__ void eval_line(const T (&v)[NX + 2], T w0, T w1, T w2, T w3, St&& st) {
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    T acc = (T)0;
    const int s0 = j - S - 1;   // slot of eta_{j-S-2}
    if (s0 >= 0 && s0 <= NX + 1) acc = w0 * v[s0];
    if (s0 + 1 >= 0 && s0 + 1 <= NX + 1) acc = fma(w1, v[s0 + 1], acc);
    if (s0 + 2 >= 0 && s0 + 2 <= NX + 1) acc = fma(w2, v[s0 + 2], acc);
    if (s0 + 3 >= 0 && s0 + 3 <= NX + 1) acc = fma(w3, v[s0 + 3], acc);
    st(j, acc);
  }
}

// One line in registers: closure, Thomas sweep and ghosts; v holds the spline coefficients
// eta_{-1..N+1} afterwards.  JC: the number of closure taps evaluated (the stencil is zero beyond
// the launch's J <= JC).
template <typename T, int NX, int JC>
__device__ __forceinline__ void solve_line(const AdvParams<T>& p, const AdvTabs<T>& tb, T (&v)[NX + 2]) {
  constexpr int N = NX - 1;
  Closure<T> cl;
#pragma unroll
  for (int j = 0; j < JC; ++j) closure_tab<NX>(cl, tb, j, v[j + 1], v[N - j + 1]);

  T dp = (T)cl.d0(v[1], hval(p)) * tb.lu[1][0];
  v[1] = dp;
#pragma unroll
  for (int i = 1; i < N; ++i) {
    dp = ((T)6 * v[i + 1] - dp) * tb.lu[1][i];
    v[i + 1] = dp;
  }
  dp = ((T)cl.dN(v[N + 1], hval(p)) - dp) * tb.lu[1][N];
  v[N + 1] = dp;
#pragma unroll
  for (int i = N - 1; i >= 0; --i) v[i + 1] = v[i + 1] - tb.lu[0][i] * v[i + 2];
  v[0] = (T)cl.gl(v[2], h2val(p));
  v[N + 2] = (T)cl.gr(v[N], h2val(p));
}

// The same for a line of n points, NX - kRag < n <= NX: everything keeps its compile-time slot,
// what depends on the line's end is selected among the last kRag slots.  The right stencil is
// stored by node (tb.c[..][i] multiplies phi_i); the factors are zero beyond N, so the slots there
// become zero and take no part.  The leading taps of the right stencil may start anywhere in that
// window, so kClosHead + kRag - 1 of them are accumulated error-free.  Classes of four: with
// classes of eight 25 points ran at 4.04 TB/s per pass (5.53), 17 points at 4.00 (5.04).
constexpr int kRag = 4;
__device__ __forceinline__ void closure_left(Closure<float>& cl, const AdvTabs<float>& tb, int j, float phi) {
  if (j < kClosHead) df_acc(cl.L, phi, tb.c[0][j], tb.c[1][j]);
  else cl.L.lo = fmaf(phi, tb.c[0][j], cl.L.lo);
}
template <int NX>
__device__ __forceinline__ void closure_right(Closure<float>& cl, const AdvTabs<float>& tb, int i, float phi) {
  if (i >= NX - kRag + 1 - kClosHead) df_acc(cl.R, phi, tb.c[2][i], tb.c[3][i]);
  else cl.R.lo = fmaf(phi, tb.c[2][i], cl.R.lo);
}
template <typename T, int NX, int JC>
__device__ __forceinline__ void solve_ragged(const AdvParams<T>& p, const AdvTabs<T>& tb, T (&v)[NX + 2]) {
  const int N = p.n - 1;
  constexpr int W0 = NX > kRag ? NX - kRag : 0;   // first slot the line may end at
  Closure<T> cl;
#pragma unroll
  for (int j = 0; j < JC; ++j) closure_left(cl, tb, j, v[j + 1]);
#pragma unroll
  for (int i = NX - 1; i >= 0; --i)
    if (i > W0 - JC) closure_right<NX>(cl, tb, i, v[i + 1]);
  T dp = (T)cl.d0(v[1], hval(p)) * tb.lu[1][0];
  v[1] = dp;
#pragma unroll
  for (int i = 1; i < NX; ++i) {
    T r = (T)6 * v[i + 1];
    if (i >= W0 && i == N) r = (T)cl.dN(v[i + 1], hval(p));
    dp = (r - dp) * tb.lu[1][i];
    v[i + 1] = dp;
  }
#pragma unroll
  for (int i = NX - 2; i >= 0; --i) v[i + 1] = v[i + 1] - tb.lu[0][i] * v[i + 2];
  v[0] = (T)cl.gl(v[2], h2val(p));
#pragma unroll
  for (int i = W0 > 1 ? W0 : 1; i < NX; ++i)
    if (i == N) v[i + 2] = (T)cl.gr(v[i], h2val(p));
}
template <typename T, int NX, int JC, bool RAG>
__device__ __forceinline__ void solve_any(const AdvParams<T>& p, const AdvTabs<T>& tb, T (&v)[NX + 2]) {
  static_assert(!RAG || sizeof(T) == 4, "ragged lengths: FP32");
  if constexpr (RAG) solve_ragged<T, NX, JC>(p, tb, v);
  else solve_line<T, NX, JC>(p, tb, v);
}

// the 4-tap evaluation of two lines with the same integer shift S (weights wa, wb), written
// together by st(j, out_a, out_b)
template <typename T, int NX, int S, class St>
__device__ __forceinline__ void eval_line2(const T (&va)[NX + 2], const T (&vb)[NX + 2], const T (&wa)[4],
                                           const T (&wb)[4], St&& st) {
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    T a = (T)0, b = (T)0;
    const int s0 = j - S - 1;
    if (s0 >= 0 && s0 <= NX + 1) {
      a = wa[0] * va[s0];
      b = wb[0] * vb[s0];
    }
    if (s0 + 1 >= 0 && s0 + 1 <= NX + 1) {
      a = fma(wa[1], va[s0 + 1], a);
      b = fma(wb[1], vb[s0 + 1], b);
    }
    if (s0 + 2 >= 0 && s0 + 2 <= NX + 1) {
      a = fma(wa[2], va[s0 + 2], a);
      b = fma(wb[2], vb[s0 + 2], b);
    }
    if (s0 + 3 >= 0 && s0 + 3 <= NX + 1) {
      a = fma(wa[3], va[s0 + 3], a);
      b = fma(wb[3], vb[s0 + 3], b);
    }
    st(j, a, b);
  }
}

// the solve, then the 4-tap evaluation at the feet of line k index kd, written by st
template <typename T, int NX, int JC, bool RAG, class St>
__device__ __forceinline__ void solve_eval_line(const AdvParams<T>& p, const AdvTabs<T>& tb,
                                                T (&v)[NX + 2], int kd, St&& st) {
  solve_any<T, NX, JC, RAG>(p, tb, v);
  const int sh = __ldg(p.ns + kd);
  const T w0 = __ldg(p.w + 4 * kd + 0), w1 = __ldg(p.w + 4 * kd + 1);
  const T w2 = __ldg(p.w + 4 * kd + 2), w3 = __ldg(p.w + 4 * kd + 3);
  switch (sh) {
    case -2: eval_line<T, NX, -2>(v, w0, w1, w2, w3, st); break;
    case -1: eval_line<T, NX, -1>(v, w0, w1, w2, w3, st); break;
    case 0: eval_line<T, NX, 0>(v, w0, w1, w2, w3, st); break;
    default: eval_line<T, NX, 1>(v, w0, w1, w2, w3, st); break;
  }
}

// FP64 form: one line per thread.  FP32-mixed form: two adjacent k (lines l and l + 1 share the
// x indices) per thread, loaded with 8-byte accesses so each thread keeps twice the bytes in
// flight, and stored with 8-byte accesses when both lines have the same integer shift (always
// for the x1 and x2 passes, whose shift depends on k1 or k2 only).
template <typename T, int NX, int JC, bool RAG>
__global__ void __launch_bounds__(kAdvectThreads) k_advect_reg(AdvParams<T> p, const AdvTabs<T> tb) {
  constexpr int LPT = sizeof(T) == 4 ? 2 : 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t * LPT >= p.n_lines) return;
  T* src;
  int kd;
  line_setup(p, t * LPT, src, kd);
  auto in_line = [&](int j) { return !RAG || j < NX - kRag || j < p.n; };   // n > NX - kRag
  if constexpr (LPT == 1) {
    T v[NX + 2];   // slot nu + 1 holds eta_nu (phi_j before the solve)
#pragma unroll
    for (int j = 0; j < NX; ++j) v[j + 1] = src[(int64_t)j * p.s_d];
    solve_eval_line<T, NX, JC, RAG>(p, tb, v, kd, [&](int j, T o) { src[(int64_t)j * p.s_d] = o; });
  } else {
    T v0[NX + 2], v1[NX + 2];
#pragma unroll
    for (int j = 0; j < NX; ++j) {
      const float2 q = in_line(j) ? *reinterpret_cast<const float2*>(src + (int64_t)j * p.s_d) : make_float2(0.f, 0.f);
      v0[j + 1] = q.x;
      v1[j + 1] = q.y;
    }
    if constexpr (RAG) v0[0] = v0[NX + 1] = v1[0] = v1[NX + 1] = (T)0;
    int kd1;
    T* src1;
    line_setup(p, t * LPT + 1, src1, kd1);
    const int sh0 = __ldg(p.ns + kd), sh1 = __ldg(p.ns + kd1);
    if (sh0 != sh1) {   // rare: the two k straddle an integer shift
      solve_eval_line<T, NX, JC, RAG>(p, tb, v0, kd, [&](int j, T o) {
        if (in_line(j)) src[(int64_t)j * p.s_d] = o;
      });
      solve_eval_line<T, NX, JC, RAG>(p, tb, v1, kd1, [&](int j, T o) {
        if (in_line(j)) src1[(int64_t)j * p.s_d] = o;
      });
      return;
    }
    solve_any<T, NX, JC, RAG>(p, tb, v0);
    solve_any<T, NX, JC, RAG>(p, tb, v1);
    T wa[4], wb[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      wa[c] = __ldg(p.w + 4 * kd + c);
      wb[c] = __ldg(p.w + 4 * kd1 + c);
    }
    auto st = [&](int j, T a, T b) {
      if (in_line(j)) *reinterpret_cast<float2*>(src + (int64_t)j * p.s_d) = make_float2(a, b);
    };
    switch (sh0) {
      case -2: eval_line2<T, NX, -2>(v0, v1, wa, wb, st); break;
      case -1: eval_line2<T, NX, -1>(v0, v1, wa, wb, st); break;
      case 0: eval_line2<T, NX, 0>(v0, v1, wa, wb, st); break;
      default: eval_line2<T, NX, 1>(v0, v1, wa, wb, st); break;
    }
  }
}

// ---- all three dimensions at once (FP32, the smallest grids) ----
// A block holds the x grid of kBoxK consecutive k in shared memory and runs the three passes there: f
// is read and written once, by one launch instead of three, whose latency bounds such a grid (what is
// left is the chain of load, three solves and store: no ragged lengths, they would lengthen it).
// Line lengths are compile-time constants; rows along x3 have an odd pitch, so that the lines of a
// warp lie in different banks in every pass.
constexpr int kBoxK = 4;
constexpr int kBoxThreads = 256;
constexpr int kBoxMaxNx = 16;
constexpr int kBoxMaxNxp = 768;
struct BoxArgs {
  AdvParams<float> p[3];
  AdvTabs<float> tb[3];
};
template <int NX>
__device__ __forceinline__ void box_line(const AdvParams<float>& p, const AdvTabs<float>& tb, float* src, int sd,
                                         int kd0, int kd1) {
  constexpr int JC = NX;
  float v0[NX + 2], v1[NX + 2];
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    const float2 q = *reinterpret_cast<const float2*>(src + j * sd);
    v0[j + 1] = q.x;
    v1[j + 1] = q.y;
  }
  solve_line<float, NX, JC>(p, tb, v0);
  solve_line<float, NX, JC>(p, tb, v1);
  const int sh0 = __ldg(p.ns + kd0), sh1 = __ldg(p.ns + kd1);
  float wa[4], wb[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    wa[c] = __ldg(p.w + 4 * kd0 + c);
    wb[c] = __ldg(p.w + 4 * kd1 + c);
  }
  auto eval = [&](int sh, auto&& st) {
    switch (sh) {
      case -2: eval_line2<float, NX, -2>(v0, v1, wa, wb, st); break;
      case -1: eval_line2<float, NX, -1>(v0, v1, wa, wb, st); break;
      case 0: eval_line2<float, NX, 0>(v0, v1, wa, wb, st); break;
      default: eval_line2<float, NX, 1>(v0, v1, wa, wb, st); break;
    }
  };
  // the two lines nearly always have one shift; where they straddle an integer, each its own
  const int both = sh0 == sh1 ? 1 : 2;
#pragma unroll 1
  for (int q = 0; q < both; ++q)
    eval(q ? sh1 : sh0, [&](int j, float a, float b) {
      if (both == 1) *reinterpret_cast<float2*>(src + j * sd) = make_float2(a, b);
      else src[j * sd + q] = q ? b : a;
    });
}
__global__ void __launch_bounds__(kBoxThreads) k_advect_box(const __grid_constant__ BoxArgs a) {
  extern __shared__ __align__(16) float box[];
  const int n0 = a.p[0].n, n1 = a.p[1].n, n2 = a.p[2].n, P2 = n2 | 1;
  const int64_t k0 = (int64_t)blockIdx.x * kBoxK;
  float* f = a.p[0].f + k0;
  const int64_t kvol = a.p[0].kvol;
  constexpr int H = kBoxK / 2;   // pairs of k
  const int nxp = n0 * n1 * n2;
  for (int i = threadIdx.x; i < nxp * H; i += kBoxThreads) {
    const int x = i / H, c = 2 * (i % H);
    *reinterpret_cast<float2*>(box + (x / n2 * P2 + x % n2) * kBoxK + c) = *reinterpret_cast<const float2*>(f + x * kvol + c);
  }
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    __syncthreads();
    const AdvParams<float>& p = a.p[d];
    const int lines = nxp / p.n;
    const int sd = (d == 0 ? n1 * P2 : d == 1 ? P2 : 1) * kBoxK;
    for (int i = threadIdx.x; i < lines * H; i += kBoxThreads) {
      const int line = i / H, c = 2 * (i % H);
      const int x = d == 2 ? line * P2 : line / n2 * (d == 0 ? P2 : n1 * P2) + line % n2;
      float* src = box + x * kBoxK + c;
      const int kd0 = (int)((k0 + c) / p.kdiv % p.nk), kd1 = (int)((k0 + c + 1) / p.kdiv % p.nk);
      switch (p.n) {
        case 4: box_line<4>(p, a.tb[d], src, sd, kd0, kd1); break;
        case 8: box_line<8>(p, a.tb[d], src, sd, kd0, kd1); break;
        case 12: box_line<12>(p, a.tb[d], src, sd, kd0, kd1); break;
        default: box_line<16>(p, a.tb[d], src, sd, kd0, kd1); break;
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nxp * H; i += kBoxThreads) {
    const int x = i / H, c = 2 * (i % H);
    *reinterpret_cast<float2*>(f + x * kvol + c) = *reinterpret_cast<const float2*>(box + (x / n2 * P2 + x % n2) * kBoxK + c);
  }
}

// ---- shared-memory kernel (any line length, any shift) ----
template <typename T>
__global__ void __launch_bounds__(kAdvectThreads) k_advect_smem(AdvParams<T> p) {
  extern __shared__ unsigned char smem_raw[];
  T* buf = reinterpret_cast<T*>(smem_raw) + threadIdx.x;
  const int B = blockDim.x;
  const int64_t line = (int64_t)blockIdx.x * B + threadIdx.x;
  if (line >= p.n_lines) return;
  T* src;
  int kd;
  line_setup(p, line, src, kd);
  const int n = p.n, N = p.n - 1;

#pragma unroll 8
  for (int j = 0; j < n; ++j) buf[(j + 1) * B] = src[(int64_t)j * p.s_d];

  Closure<T> cl;
  for (int j = 0; j < p.J; ++j) cl.add(p.clos, n, j, buf[(j + 1) * B], buf[(N - j + 1) * B]);

  T dp = (T)cl.d0(buf[B], hval(p)) * __ldg(p.mult);
  buf[B] = dp;
  for (int i = 1; i < N; ++i) {
    dp = ((T)6 * buf[(i + 1) * B] - dp) * __ldg(p.mult + i);
    buf[(i + 1) * B] = dp;
  }
  dp = ((T)cl.dN(buf[(N + 1) * B], hval(p)) - dp) * __ldg(p.mult + N);
  buf[(N + 1) * B] = dp;
  T e = dp;
  for (int i = N - 1; i >= 0; --i) {
    e = buf[(i + 1) * B] - __ldg(p.cprime + i) * e;
    buf[(i + 1) * B] = e;
  }
  buf[0] = (T)cl.gl(buf[2 * B], h2val(p));
  buf[(N + 2) * B] = (T)cl.gr(buf[N * B], h2val(p));

  const int sh = __ldg(p.ns + kd);
  const T w0 = __ldg(p.w + 4 * kd + 0), w1 = __ldg(p.w + 4 * kd + 1);
  const T w2 = __ldg(p.w + 4 * kd + 2), w3 = __ldg(p.w + 4 * kd + 3);
  for (int j = 0; j < n; ++j) {
    const int nu0 = j - sh - 2;   // first tap index
    T acc = (T)0;
    if (nu0 >= -1 && nu0 <= N + 1) acc = w0 * buf[(nu0 + 1) * B];
    if (nu0 + 1 >= -1 && nu0 + 1 <= N + 1) acc = fma(w1, buf[(nu0 + 2) * B], acc);
    if (nu0 + 2 >= -1 && nu0 + 2 <= N + 1) acc = fma(w2, buf[(nu0 + 3) * B], acc);
    if (nu0 + 3 >= -1 && nu0 + 3 <= N + 1) acc = fma(w3, buf[(nu0 + 4) * B], acc);
    src[(int64_t)j * p.s_d] = acc;
  }
}

// ---- very short FP64 lines: the whole pass as a dense matrix per k ----
// Closure, solve and evaluation of an n-point line cost about 7 + 2 J/n FP64 FMAs per point on a pipe
// of 1.7 per clock and SM, the n x n matrix that they amount to costs n: less up to kAdvDenseMax
// points (5 points: 1.75 -> 0.83 ms a pass at 121 x 5^2 x 32^3; 8 points run at 1175 GB/s, 9 points in
// shared memory at 940).  The matrices come from the host
// (dense_rows), entry (j, q) of every k side by side, so a warp reads one value or consecutive ones.
template <int NX>
__global__ void __launch_bounds__(kAdvectThreads) k_advect_dense(AdvParams<double> p, const double* __restrict__ mat) {
  const int64_t line = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (line >= p.n_lines) return;
  double* src;
  int kd;
  line_setup(p, line, src, kd);
  double v[NX];
#pragma unroll
  for (int j = 0; j < NX; ++j) v[j] = src[(int64_t)j * p.s_d];
  const double* m = mat + kd;
#pragma unroll
  for (int j = 0; j < NX; ++j) {
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < NX; ++q) acc = fma(__ldg(m + (j * NX + q) * p.nk), v[q], acc);
    src[(int64_t)j * p.s_d] = acc;
  }
}

// ---- patches (p > 1): Sec. 3.1.2 steps (1)-(5) and the interpolation with correction of
// Sec. 3.1.3, one line per thread in shared memory (column layout) ----
template <typename T>
struct PatchArgs {
  int P, M, nb, W;
  const T* win;   // closure windows: FP64 [(P+1)][W]; FP32 [(P+1)][2][W] (hi, lo)
  const T* lu;    // [c' (M+1) | 1/pivot (M+1)] of the (M+1)-node patch system
};

// closure value of boundary b = sum over its window of coefficient * phi, hi/lo parts; phi_j at
// buf[j B], taps outside [0, N] dropped
__device__ __forceinline__ void patch_closure(const PatchArgs<double>& q, const double* buf, int B, int N,
                                              int b, double& hi, double& lo) {
  const int first = b * q.M - q.nb, i0 = max(0, -first), i1 = min(q.W - 1, N - first);
  const double* w = q.win + (size_t)b * q.W;
  double acc = 0.0;
#pragma unroll 4
  for (int i = i0; i <= i1; ++i) acc = fma(__ldg(w + i), buf[(first + i) * B], acc);
  hi = acc;
  lo = 0.0;
}
__device__ __forceinline__ void patch_closure(const PatchArgs<float>& q, const float* buf, int B, int N,
                                              int b, float& hi, float& lo) {
  const int first = b * q.M - q.nb, i0 = max(0, -first), i1 = min(q.W - 1, N - first);
  const float* w = q.win + (size_t)b * 2 * q.W;
  DF acc{0.f, 0.f};
#pragma unroll 4
  for (int i = i0; i <= i1; ++i) df_acc(acc, buf[(first + i) * B], __ldg(w + i), __ldg(w + q.W + i));
  hi = acc.hi;
  lo = acc.lo;
}

// All closures are formed first; then each patch is solved in place over its nodes and evaluated
// before the next one starts, so a line needs n + 2 values and its closures: the left ghost takes
// the slot before the patch (done with), the right ghost borrows the slot behind it, and the node
// two patches share is handed on.  With every patch's coefficients kept, 121 points in 4 patches
// left room for 3 FP64 warps per SM, which cannot keep the four FP64 pipes busy: 4.15 -> 2.03 ms a pass
// at 121 x 5^2 x 32^3 (6 warps).
template <typename T>
__global__ void __launch_bounds__(kAdvectThreads) k_advect_patches(AdvParams<T> p, PatchArgs<T> q) {
  constexpr int kParts = sizeof(T) == 4 ? 2 : 1;            // hi and lo part of a closure
  extern __shared__ unsigned char smem_raw[];
  const int B = blockDim.x;
  const int n = p.n, N = n - 1, P = q.P, M = q.M;
  T* buf = reinterpret_cast<T*>(smem_raw) + threadIdx.x + B;   // phi_j at buf[j B], j = -1..n
  T* cv = buf + (n + 1) * B;                                    // closure b at cv[kParts b B] (and + B)
  const int64_t line = (int64_t)blockIdx.x * B + threadIdx.x;
  if (line >= p.n_lines) return;                                // whole warps: kvol is a multiple of 32
  T* src;
  int kd;
  line_setup(p, line, src, kd);
#pragma unroll 8
  for (int j = 0; j < n; ++j) buf[j * B] = src[(int64_t)j * p.s_d];
  for (int b = 0; b <= P; ++b) {
    T hi, lo;
    patch_closure(q, buf, B, N, b, hi, lo);
    cv[kParts * b * B] = hi;
    if constexpr (kParts == 2) cv[(2 * b + 1) * B] = lo;
  }
  const T* cprime = q.lu;
  const T* mult = q.lu + (M + 1);
  const int sh = __ldg(p.ns + kd);
  const T w[4] = {__ldg(p.w + 4 * kd + 0), __ldg(p.w + 4 * kd + 1), __ldg(p.w + 4 * kd + 2),
                  __ldg(p.w + 4 * kd + 3)};
  T shared = buf[0];   // phi at the patch's first node
  for (int l = 0; l < P; ++l) {
    T* e = buf + l * M * B;   // eta_nu of this patch at e[nu B], nu = -1..M+1
    Closure<T> cl;            // phi_L of patch l in cl.L, phi_R in cl.R
    if constexpr (kParts == 2) {
      cl.L = DF{cv[2 * l * B], cv[(2 * l + 1) * B]};
      cl.R = DF{cv[(2 * l + 2) * B], cv[(2 * l + 3) * B]};
    } else {
      cl.L = cv[l * B];
      cl.R = cv[(l + 1) * B];
    }
    const T behind = e[(M + 1) * B], last = e[M * B];
    T dp = (T)cl.d0(shared, hval(p)) * __ldg(mult);
    e[0] = dp;
#pragma unroll 4
    for (int i = 1; i < M; ++i) {
      dp = ((T)6 * e[i * B] - dp) * __ldg(mult + i);
      e[i * B] = dp;
    }
    dp = ((T)cl.dN(last, hval(p)) - dp) * __ldg(mult + M);
    e[M * B] = dp;
    T nx = dp;
#pragma unroll 4
    for (int i = M - 1; i >= 0; --i) {
      nx = e[i * B] - __ldg(cprime + i) * nx;
      e[i * B] = nx;
    }
    e[-B] = (T)cl.gl(e[B], h2val(p));
    e[(M + 1) * B] = (T)cl.gr(e[(M - 1) * B], h2val(p));
    // the nodes whose foot x_j - (sh + a) h lies in this patch (the left patch at a shared node, the
    // end patches beyond the ends): j - sh - 1 in [l M, (l + 1) M); one loop for the warp
    const int j0 = l == 0 ? 0 : max(0, l * M + sh + 1);
    const int j1 = l == P - 1 ? n - 1 : min(n - 1, l * M + M + sh);
    const int first = __reduce_min_sync(0xffffffffu, j0), final = __reduce_max_sync(0xffffffffu, j1);
#pragma unroll 4
    for (int j = first; j <= final; ++j) {
      const int nu0 = j - l * M - sh - 2;   // first tap, local index
      T acc = (T)0;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int nu = nu0 + c;
        if (nu >= -1 && nu <= M + 1) acc = fma(w[c], e[nu * B], acc);
      }
      if (j >= j0 && j <= j1) src[(int64_t)j * p.s_d] = acc;
    }
    e[(M + 1) * B] = behind;
    shared = last;
  }
}

template <typename T>
AdvParams<T> make_params(const Handle& H, void* f, int dim) {
  const GridDesc& g = H.g;
  AdvParams<T> p;
  p.f = static_cast<T*>(f);
  p.kvol = g.kvol;
  const int64_t s3 = g.kvol, s2 = (int64_t)g.nx[2] * g.kvol, s1 = (int64_t)g.nx[1] * s2;
  const int64_t strides[3] = {s1, s2, s3};
  const int other[3][2] = {{1, 2}, {0, 2}, {0, 1}};
  p.s_d = strides[dim];
  p.s_a = strides[other[dim][0]];
  p.s_b = strides[other[dim][1]];
  p.n_b = g.nx[other[dim][1]];
  p.n = g.nx[dim];
  p.n_lines = (int64_t)g.nx[other[dim][0]] * g.nx[other[dim][1]] * g.kvol;
  p.nk = g.nk;
  p.kdiv = dim == 0 ? g.nk * g.nk : (dim == 1 ? g.nk : 1);
  p.J = H.J[dim];
  p.h = g.h[dim];
  p.hf = (float)g.h[dim];
  p.h2f = (float)(2.0 * g.h[dim]);
  p.clos = static_cast<const T*>(H.d_clos[dim]);
  p.cprime = static_cast<const T*>(H.d_lu[dim]);
  p.mult = static_cast<const T*>(H.d_lu[dim]) + g.nx[dim];
  const T* wbase = static_cast<const T*>(H.adv.dev);
  p.w = wbase + (size_t)dim * g.nk * 4;
  p.ns = reinterpret_cast<const int*>(wbase + (size_t)3 * g.nk * 4) + dim * g.nk;
  return p;
}

// closure stencils and Thomas factors of dimension dim for the register kernels (ragged: the
// right stencil by node instead of by distance from the end)
template <typename T>
AdvTabs<T> make_tabs(const Handle& H, int dim, bool ragged) {
  const int n = H.g.nx[dim];
  AdvTabs<T> tb;
  std::memset(&tb, 0, sizeof(tb));
  const std::vector<double>& hc = H.h_clos[dim];
  const std::vector<double>& hl = H.h_lu[dim];
  for (int j = 0; j < n; ++j) {
    const int jr = ragged ? n - 1 - j : j;
    if constexpr (sizeof(T) == 4) {   // unevaluated float pairs hi + lo of the FP64 stencils
      tb.c[0][j] = (float)hc[j];
      tb.c[1][j] = (float)(hc[j] - (double)tb.c[0][j]);
      tb.c[2][j] = (float)hc[n + jr];
      tb.c[3][j] = (float)(hc[n + jr] - (double)tb.c[2][j]);
    } else {
      tb.c[0][j] = hc[j];
      tb.c[1][j] = hc[n + jr];
    }
    tb.lu[0][j] = (T)hl[j];
    tb.lu[1][j] = (T)hl[n + j];
  }
  return tb;
}

// The register kernels apply: integer shifts in [-2, 1], up to kRegMaxNx points and (in FP32, for
// the 8-byte accesses) an even address.
bool reg_applies(const Handle& H, const void* f, int dim) {
  return H.adv.ns_min[dim] >= -2 && H.adv.ns_max[dim] <= 1 && H.opt.patches[dim] <= 1 &&
         H.g.nx[dim] <= kRegMaxNx && (reinterpret_cast<uintptr_t>(f) & 7) == 0;
}

// Lines of n points with their length a compile-time constant (the workloads' lengths)
template <typename T, int NX>
void launch_exact(const AdvParams<T>& p, const AdvTabs<T>& tb, unsigned blocks, cudaStream_t s) {
  // closure taps: the launch's J rounded up to a compiled bucket (the stencil is zero beyond J)
  constexpr int JS = NX > 24 ? 24 : NX;
  if (p.J <= JS) k_advect_reg<T, NX, JS, false><<<blocks, kAdvectThreads, 0, s>>>(p, tb);
  else k_advect_reg<T, NX, NX, false><<<blocks, kAdvectThreads, 0, s>>>(p, tb);
}
// NX - kRag < n <= NX, J <= 24, FP32
template <int NX>
bool launch_ragged(const AdvParams<float>& p, const AdvTabs<float>& tb, unsigned blocks, cudaStream_t s) {
  if constexpr (NX < 4) {
    return false;
  } else {
    if (p.n <= NX - kRag) return launch_ragged<NX - kRag>(p, tb, blocks, s);
    constexpr int JS = NX > 24 ? 24 : NX;
    k_advect_reg<float, NX, JS, true><<<blocks, kAdvectThreads, 0, s>>>(p, tb);
    return true;
  }
}

template <typename T>
cudaError_t launch_t(const Handle& H, void* f, int dim, cudaStream_t s) {
  const GridDesc& g = H.g;
  AdvParams<T> p = make_params<T>(H, f, dim);
  const int B = kAdvectThreads;
  const int P = H.opt.patches[dim];
  if (P > 1) {
    PatchArgs<T> q;
    q.P = P;
    q.M = (p.n - 1) / P;
    q.nb = H.opt.n_nb;
    q.W = 2 * q.nb + 1;
    q.win = static_cast<const T*>(H.d_pclos[dim]);
    q.lu = static_cast<const T*>(H.d_plu[dim]);
    const size_t elems = (size_t)p.n + 2 + (size_t)(P + 1) * (sizeof(T) == 4 ? 2 : 1);
    // the block size that leaves the most threads on an SM
    int Bp = 0;
    size_t most = 0;
    for (int b = kAdvectThreads; b >= 32; b -= 32) {
      const size_t bytes = elems * b * sizeof(T);
      if (bytes > (size_t)kAdvectMaxSmem) continue;
      const size_t on = (size_t)(227 * 1024) / (bytes + 1024) * b;
      if (on > most) {
        most = on;
        Bp = b;
      }
    }
    if (Bp == 0) return cudaErrorInvalidValue;
    k_advect_patches<T><<<(unsigned)((p.n_lines + Bp - 1) / Bp), Bp, elems * Bp * sizeof(T), s>>>(p, q);
    return cudaGetLastError();
  }
  if constexpr (sizeof(T) == 8) {
    if (advect_dense(H, dim)) {
      const double* mat = reinterpret_cast<const double*>(static_cast<const char*>(H.adv.dev) + advect_dense_offset(H, dim));
      const unsigned nb = (unsigned)((p.n_lines + B - 1) / B);
      switch (p.n) {
        case 4: k_advect_dense<4><<<nb, B, 0, s>>>(p, mat); break;
        case 5: k_advect_dense<5><<<nb, B, 0, s>>>(p, mat); break;
        case 6: k_advect_dense<6><<<nb, B, 0, s>>>(p, mat); break;
        case 7: k_advect_dense<7><<<nb, B, 0, s>>>(p, mat); break;
        default: k_advect_dense<8><<<nb, B, 0, s>>>(p, mat); break;
      }
      return cudaGetLastError();
    }
  }
  if (reg_applies(H, f, dim)) {
    const int64_t lpt = sizeof(T) == 4 ? 2 : 1;   // kvol = nk^3 is even
    const unsigned rblocks = (unsigned)((p.n_lines / lpt + B - 1) / B);
    const bool exact = p.n == 16 || p.n == 24 || p.n == 32 || p.n == 48 || p.n == 64;
    if (exact || (sizeof(T) == 4 && p.J <= 24)) {
      const AdvTabs<T> tb = make_tabs<T>(H, dim, !exact);
      switch (p.n) {
        case 16: launch_exact<T, 16>(p, tb, rblocks, s); break;
        case 24: launch_exact<T, 24>(p, tb, rblocks, s); break;
        case 32: launch_exact<T, 32>(p, tb, rblocks, s); break;
        case 48: launch_exact<T, 48>(p, tb, rblocks, s); break;
        case 64: launch_exact<T, 64>(p, tb, rblocks, s); break;
        default:
          if constexpr (sizeof(T) == 4) launch_ragged<kRegMaxNx>(p, tb, rblocks, s);
      }
      return cudaGetLastError();
    }
  }
  const size_t elems = advect_smem_elems(g.nx[dim], 1);
  const int Bs = advect_smem_threads(elems, sizeof(T));
  if (Bs == 0) return cudaErrorInvalidValue;
  k_advect_smem<T><<<(unsigned)((p.n_lines + Bs - 1) / Bs), Bs, elems * Bs * sizeof(T), s>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t advect_prepare() {
  // up to kAdvectMaxSmem bytes of dynamic shared memory (fewer threads per block for long lines;
  // lines too long even for 32 threads are rejected at create time)
  cudaError_t e = cudaFuncSetAttribute(k_advect_smem<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kAdvectMaxSmem);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_advect_smem<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kAdvectMaxSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_advect_patches<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdvectMaxSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_advect_patches<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, kAdvectMaxSmem);
  return e;
}

// The three passes in one launch, where a pass is bounded by its launch: N_k = 8 (128 blocks, fewer than
// SMs; each has an x grid, so more k only add waves) and few x points.  FP32 Strang step, three
// passes -> one: 4^3 27.8 -> 21.3 us, 8^3 33.4 -> 29.0, 12 x 8 x 8 41.2 -> 35.4, but 12^3 57.8 -> 60.0;
// with N_k = 16 4^3 41.3 -> 49.7, 8^3 107.7 -> 118.7.
bool advect_box(const Handle& H, const void* f) {
  if (H.fp64 || H.g.nk != 8 || H.g.nxp > kBoxMaxNxp) return false;
  for (int d = 0; d < 3; ++d)
    if (!reg_applies(H, f, d) || H.g.nx[d] % 4 != 0 || H.g.nx[d] > kBoxMaxNx) return false;
  return true;
}

cudaError_t launch_advect_box(const Handle& H, void* f, cudaStream_t s) {
  BoxArgs a;
  for (int d = 0; d < 3; ++d) {
    a.p[d] = make_params<float>(H, f, d);
    a.tb[d] = make_tabs<float>(H, d, false);
  }
  const size_t smem = (size_t)H.g.nx[0] * H.g.nx[1] * (H.g.nx[2] | 1) * kBoxK * sizeof(float);
  static_assert(kBoxMaxNxp * 5 / 4 * kBoxK * sizeof(float) <= 48 * 1024, "without an opt-in");   // nx >= 4
  k_advect_box<<<(unsigned)(H.g.kvol / kBoxK), kBoxThreads, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_advect_dim(const Handle& H, void* f, int dim, cudaStream_t s) {
  return H.fp64 ? launch_t<double>(H, f, dim, s) : launch_t<float>(H, f, dim, s);
}

}  // namespace chasm
