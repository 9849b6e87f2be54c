// Phase-space diagnostics of Sec. 5, in FP64 with a fixed summation order (bitwise reproducible):
//
//   W_j(x, k)  = integral of f over the other two x and the other two k coordinates
//   P(x1, x2)  = integral of f over x3 and k
//   <x_d>, <k_d> = sum x_d f / sum f, sum k_d f / sum f   (averaged position and momentum)
//
// W_j and P: S_d[x][q] = sum of f[x] over the two k indices other than k_d = q (k_diag_kpart, f read
// once), then W_j sums S_j over the other two x indices (a block per x_j) and P sums S_0 over x3
// and q (a warp per (x1, x2)).  The averages read f once as well (k_diag_expect, the sums of
// xsums.cuh); a second kernel adds the block partials in a fixed tree.  The grid factors (cell
// volumes, x and k node positions) are applied in FP64.
#include "xsums.cuh"

namespace chasm {
namespace {

constexpr int kDiagThreads = 256;

// Double precision: the same assignment as below with one value per access (the FP64 pipe adds 1.7
// per clock and SM, which one 8-byte access per lane keeps up with): D = 0, 1 a warp per (x
// point, q), D = 2 a warp per x point with one k3 per lane.
template <int N, int D>
__global__ void __launch_bounds__(kDiagThreads) k_diag_kpart_d(const double* __restrict__ f, int64_t nxp,
                                                               double* __restrict__ S) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= (D < 2 ? nxp * N : nxp)) return;
  const int q = (int)(w % N);
  const double* base = f + (D < 2 ? w / N : w) * (N * N * N);
  constexpr int kEach = D < 2 ? N * N : N * N * N;
  double s = 0.0;
#pragma unroll 8
  for (int g = lane; g < kEach; g += 32)
    s += __ldcs(base + (D == 0 ? q * N * N + g : (D == 1 ? (g / N * N + q) * N + g % N : g)));
#pragma unroll
  for (int o = D < 2 ? 1 : N; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if constexpr (D < 2) {
    if (lane == 0) S[w] = s;
  } else {
    if (lane < N) S[w * N + lane] = s;
  }
}

// Single precision: one warp per (x point, q) for d = 0, 1 and one warp per x point for d = 2,
// every lane summing its 16-byte loads in compensated FP32 (two-sum; the FP64 pipe runs at 1/64
// of the FP32 rate here), then a compensated butterfly across the lanes and one rounding to FP64.
// The lanes of a warp read consecutive 16-byte pieces: d = 0, the k1 = q slab (N^2 contiguous
// values); d = 1, the rows (a, q) of N contiguous values, N/4 lanes per row; d = 2, the rows
// (a, b), one k3 quad per lane, so that each lane owns four bins.
__device__ __forceinline__ void warp_two_sum(float& hi, float& lo, unsigned mask, int o) {
  const float oh = __shfl_xor_sync(mask, hi, o), ol = __shfl_xor_sync(mask, lo, o);
  two_sum_f(hi, lo, oh);
  lo += ol;
}

template <int N, int D>
__global__ void __launch_bounds__(kDiagThreads) k_diag_kpart_w(const float* __restrict__ f, int64_t nxp,
                                                               double* __restrict__ S) {
  constexpr int Q = N / 4;   // float4 per row of N
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if constexpr (D < 2) {
    if (w >= nxp * N) return;
    const int64_t xp = w / N;
    const int q = (int)(w % N);
    const float4* base = reinterpret_cast<const float4*>(f + xp * (N * N * N));
    float hi = 0.f, lo = 0.f;
#pragma unroll 8
    for (int g = lane; g < N * Q; g += 32) {
      const int a = g / Q, b4 = g % Q;
      const float4 v = __ldcs(base + (D == 0 ? q * N * Q + g : (a * N + q) * Q + b4));
      two_sum_f(hi, lo, v.x);
      two_sum_f(hi, lo, v.y);
      two_sum_f(hi, lo, v.z);
      two_sum_f(hi, lo, v.w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) warp_two_sum(hi, lo, 0xffffffffu, o);
    if (lane == 0) S[w] = (double)hi + (double)lo;
  } else {
    if (w >= nxp) return;
    const float4* base = reinterpret_cast<const float4*>(f + w * (N * N * N));
    constexpr int RPI = 32 / Q;   // rows read per iteration by the warp
    const int p = lane % Q, r0 = lane / Q;
    float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
    for (int row = r0; row < N * N; row += RPI) {
      const float4 v = __ldcs(base + row * Q + p);
      two_sum_f(hi[0], lo[0], v.x);
      two_sum_f(hi[1], lo[1], v.y);
      two_sum_f(hi[2], lo[2], v.z);
      two_sum_f(hi[3], lo[3], v.w);
    }
#pragma unroll
    for (int o = Q; o < 32; o <<= 1)
#pragma unroll
      for (int c = 0; c < 4; ++c) warp_two_sum(hi[c], lo[c], 0xffffffffu, o);
    if (lane < Q)
#pragma unroll
      for (int c = 0; c < 4; ++c) S[w * N + 4 * p + c] = (double)hi[c] + (double)lo[c];
  }
}

// W_j[i][q] = vol * sum over the other two x indices of S_j[x][q]: one block per i, thread t adds
// q = t mod N over the (a, b) pairs t / N, t / N + G, ... (G = threads / N), then the G partials
// of each q in ascending order (a fixed order: bitwise reproducible)
constexpr int kWigThreads = 1024;   // one block per x_j: few blocks, so wide ones (256 threads: 43 us at 32^3)
__global__ void __launch_bounds__(kWigThreads) k_diag_wigner(const double* __restrict__ S, int j, int nx0,
                                                             int nx1, int nx2, int N, double vol,
                                                             double* __restrict__ W) {
  __shared__ double part[kWigThreads];
  const int nx[3] = {nx0, nx1, nx2};
  const int i = blockIdx.x, t = threadIdx.x;
  const int q = t % N, G = kWigThreads / N;
  const int oa = j == 0 ? 1 : 0, ob = j == 2 ? 1 : 2;
  double s = 0.0;
  for (int ab = t / N; ab < nx[oa] * nx[ob]; ab += G) {
    int ix[3];
    ix[j] = i;
    ix[oa] = ab / nx[ob];
    ix[ob] = ab % nx[ob];
    const int64_t xp = ((int64_t)ix[0] * nx1 + ix[1]) * nx2 + ix[2];
    s += S[xp * N + q];
  }
  part[t] = s;
  __syncthreads();
  if (t < N) {
    double r = 0.0;
    for (int g = 0; g < G; ++g) r += part[g * N + t];
    W[(int64_t)i * N + t] = r * vol;
  }
}

// P[i1][i2] = vol * sum over i3 and q of S_0[x][q]: one warp per (i1, i2) (a thread each: 161 us at
// 32^3 x 32^3)
__global__ void k_diag_marginal(const double* __restrict__ S0, int nx0, int nx1, int nx2, int N,
                                double vol, double* __restrict__ P) {
  const int t = (int)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (t >= nx0 * nx1) return;
  const int lane = threadIdx.x & 31;
  const double* r = S0 + (int64_t)t * nx2 * N;
  double s = 0.0;
#pragma unroll 8
  for (int e = lane; e < nx2 * N; e += 32) s += r[e];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) P[t] = s * vol;
}

// Averages: per block the sums of f, of i_d f (x index) and of k_d f (integer k) over its x points.  Three reads
// of f, one per k-dimension, took 1.75 ms at 32^3 x 32^3 FP32, this one 0.78.
// fixed: the order of the sums does not depend on the device; four blocks on each of 152 SMs
constexpr int kExpBlocks = 608;
template <typename T, int N>
__global__ void __launch_bounds__(XSums<T, N>::kThreads) k_diag_expect(const T* __restrict__ f, int64_t nxp,
                                                                       int nx1, int nx2, bool wide,
                                                                       double* __restrict__ part) {
  using X = XSums<T, N>;
  const X me;
  double acc[7] = {0, 0, 0, 0, 0, 0, 0};
  Run<T> run[7];
  int n = 0;
  for (int64_t xp = blockIdx.x; xp < nxp; xp += gridDim.x) {
    // an x point holds at least 2 KB, so their number fits 32 bits
    const unsigned x = (unsigned)xp, r = x / (unsigned)nx2;
    const int i3 = (int)(x % (unsigned)nx2), i2 = (int)(r % (unsigned)nx1), i1 = (int)(r / (unsigned)nx1);
    Run<T> m, u, v;
    me.template add<false>(f + xp * (N * N * N), wide, m, u, v);
    run[0].add(m);
    run[1].add(m, (float)i1);
    run[2].add(m, (float)i2);
    run[3].add(m, (float)i3);
    run[4].add(u);
    run[5].add(m, (float)me.k2);
    run[6].add(v);
    if (++n == kRunLength<T> || xp + gridDim.x >= nxp) {
#pragma unroll
      for (int c = 0; c < 7; ++c) acc[c] += run[c].take();
      n = 0;
    }
  }
  block_sum_store<7>(acc, part);
}

// the block partials in a fixed tree; out[d] = x_lo + h sum i_d f / sum f, out[3 + d] = dk sum k_d f /
// sum f
__global__ void __launch_bounds__(kDiagThreads) k_diag_expect_final(const double* __restrict__ part, int nb,
                                                                    double3 xlo, double3 h, double dk,
                                                                    double* __restrict__ out) {
  __shared__ double tot[7];
  double v[7] = {0, 0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nb; b += kDiagThreads)
#pragma unroll
    for (int c = 0; c < 7; ++c) v[c] += part[7 * b + c];
  block_sum_store<7>(v, tot);
  __syncthreads();
  const int c = threadIdx.x;
  if (c < 6) {
    const double lo = c == 0 ? xlo.x : (c == 1 ? xlo.y : (c == 2 ? xlo.z : 0.0));
    const double step = c == 0 ? h.x : (c == 1 ? h.y : (c == 2 ? h.z : dk));
    out[c] = fma(step, tot[1 + c] / tot[0], lo);
  }
}

inline unsigned nblk(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

template <typename T, int N>
cudaError_t kpart_tn(const Handle& H, const void* f, int d, double* S, cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    const float* ff = static_cast<const float*>(f);
    double* Sd = S + (size_t)d * H.g.nxp * N;
    const int64_t warps = d == 2 ? H.g.nxp : H.g.nxp * N;
    const unsigned nb = nblk(warps * 32, kDiagThreads);
    if (d == 0) k_diag_kpart_w<N, 0><<<nb, kDiagThreads, 0, s>>>(ff, H.g.nxp, Sd);
    else if (d == 1) k_diag_kpart_w<N, 1><<<nb, kDiagThreads, 0, s>>>(ff, H.g.nxp, Sd);
    else k_diag_kpart_w<N, 2><<<nb, kDiagThreads, 0, s>>>(ff, H.g.nxp, Sd);
  } else {
    const double* fd = static_cast<const double*>(f);
    double* Sd = S + (size_t)d * H.g.nxp * N;
    const unsigned nb = nblk((d == 2 ? H.g.nxp : H.g.nxp * N) * 32, kDiagThreads);
    if (d == 0) k_diag_kpart_d<N, 0><<<nb, kDiagThreads, 0, s>>>(fd, H.g.nxp, Sd);
    else if (d == 1) k_diag_kpart_d<N, 1><<<nb, kDiagThreads, 0, s>>>(fd, H.g.nxp, Sd);
    else k_diag_kpart_d<N, 2><<<nb, kDiagThreads, 0, s>>>(fd, H.g.nxp, Sd);
  }
  return cudaGetLastError();
}

template <typename T, int N>
cudaError_t expect_tn(const Handle& H, const void* f, double* part, double* out, cudaStream_t s) {
  const int nb = (int)std::min<int64_t>(kExpBlocks, H.g.nxp);
  k_diag_expect<T, N><<<nb, XSums<T, N>::kThreads, 0, s>>>(
      static_cast<const T*>(f), H.g.nxp, H.g.nx[1], H.g.nx[2], (reinterpret_cast<uintptr_t>(f) & 15) == 0, part);
  k_diag_expect_final<<<1, kDiagThreads, 0, s>>>(part, nb, make_double3(H.g.x_lo[0], H.g.x_lo[1], H.g.x_lo[2]),
                                                 make_double3(H.g.h[0], H.g.h[1], H.g.h[2]), H.g.dk, out);
  return cudaGetLastError();
}

cudaError_t kpart(const Handle& H, const void* f, int d, double* S, cudaStream_t s) {
  switch (H.g.nk) {
    case 8: return H.fp64 ? kpart_tn<double, 8>(H, f, d, S, s) : kpart_tn<float, 8>(H, f, d, S, s);
    case 16: return H.fp64 ? kpart_tn<double, 16>(H, f, d, S, s) : kpart_tn<float, 16>(H, f, d, S, s);
    case 32: return H.fp64 ? kpart_tn<double, 32>(H, f, d, S, s) : kpart_tn<float, 32>(H, f, d, S, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

size_t diag_bytes(const int nx[3], int nk) {
  const size_t nxp = (size_t)nx[0] * nx[1] * nx[2];
  const size_t outn = std::max<size_t>({(size_t)nx[0] * nk, (size_t)nx[1] * nk, (size_t)nx[2] * nk,
                                        (size_t)nx[0] * nx[1], 8});
  return (3 * nxp * nk + std::max<size_t>(outn, 8 + 7 * (size_t)kExpBlocks)) * sizeof(double);
}

cudaError_t launch_diag(const Handle& H, const void* f, int what, int j, double* buf, double* out_dev,
                        cudaStream_t s) {
  const int N = H.g.nk;
  const int* nx = H.g.nx;
  cudaError_t e = cudaSuccess;
  if (what == 0) {   // reduced Wigner function W_j
    e = kpart(H, f, j, buf, s);
    if (e != cudaSuccess) return e;
    const int oa = j == 0 ? 1 : 0, ob = j == 2 ? 1 : 2;
    const double vol = H.g.h[oa] * H.g.h[ob] * H.g.dk * H.g.dk;
    k_diag_wigner<<<nx[j], kWigThreads, 0, s>>>(buf + (size_t)j * H.g.nxp * N, j, nx[0], nx[1],
                                                 nx[2], N, vol, out_dev);
  } else if (what == 1) {   // marginal P(x1, x2)
    e = kpart(H, f, 0, buf, s);
    if (e != cudaSuccess) return e;
    const double vol = H.g.h[2] * H.g.dk * H.g.dk * H.g.dk;
    k_diag_marginal<<<nblk((int64_t)nx[0] * nx[1] * 32, kDiagThreads), kDiagThreads, 0, s>>>(
        buf, nx[0], nx[1], nx[2], N, vol, out_dev);
  } else {   // averages
    double* part = out_dev + 8;   // the block partials go behind the six results (diag_bytes reserves them)
    switch (N) {
      case 8: return H.fp64 ? expect_tn<double, 8>(H, f, part, out_dev, s) : expect_tn<float, 8>(H, f, part, out_dev, s);
      case 16: return H.fp64 ? expect_tn<double, 16>(H, f, part, out_dev, s) : expect_tn<float, 16>(H, f, part, out_dev, s);
      case 32: return H.fp64 ? expect_tn<double, 32>(H, f, part, out_dev, s) : expect_tn<float, 32>(H, f, part, out_dev, s);
    }
    return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace chasm
