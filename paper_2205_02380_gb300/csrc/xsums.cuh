// Sums of f over the k grid of one x point, the common part of mass and energy (k_misc.cu) and of
// the averaged position and momentum (k_diag.cu): every thread of a block sums the elements that
// are its own in every x point,
//   m = sum f and sums of w(k) f, w = k1, k2, k3 or |k|^2 (centred indices).
// A thread's k2 and its kV consecutive k3 never change (the block's threads cover whole k1 planes),
// so only the weight of k1 enters per element; those of k2 and k3 are applied once per x point, to
// the thread's sums over k1.
//
// Bound: reading f once.  FP32 accumulates in compensated pairs (Knuth's two-sum; the products with
// their exact FMA residual, about 2^-44 relative), because the FP64 pipe cannot add one value per
// element at that speed: 15 FP32 operations per element, 16-byte loads, eight in flight per thread.
// FP64 is bound by its two operations per element on the FP64 pipe.
#pragma once

#include "internal.hpp"

namespace chasm {
namespace {

// A running sum in the accumulation type of T: FP64, or for FP32 data an unevaluated pair hi + lo that
// goes to FP64 every few x points (a conversion and an addition in FP64 occupy the pipe for 19 clocks
// per warp each; with all of them per x point the averages took 0.88 ms at 32^3 x 32^3).
template <typename T>
struct Run;
template <>
struct Run<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(const Run& a) { s += a.s; }
  __device__ __forceinline__ void add(const Run& a, float w) { s = fma((double)w, a.s, s); }
  __device__ __forceinline__ double take() {
    const double r = s;
    s = 0.0;
    return r;
  }
};
template <>
struct Run<float> {
  float h = 0.f, l = 0.f;
  __device__ __forceinline__ void add(const Run& a) {
    two_sum_f(h, l, a.h);
    l += a.l;
  }
  __device__ __forceinline__ void add(const Run& a, float w) {
    const float p = a.h * w;
    l += fmaf(a.h, w, -p) + a.l * w;   // exact product residual
    two_sum_f(h, l, p);
  }
  __device__ __forceinline__ double take() {
    const double r = (double)h + (double)l;
    h = l = 0.f;
    return r;
  }
};
template <typename T>
constexpr int kRunLength = sizeof(T) == 4 ? 4 : 1;   // x points between conversions

template <typename T, int N>
struct XSums {
  static constexpr int kV = 16 / sizeof(T);                    // elements per 16-byte access
  static constexpr int kThreads = sizeof(T) == 4 ? 256 : 512;  // a multiple of a k1 plane's accesses, or of all of them
  static constexpr int kRow = N / kV;                          // accesses per k3 row
  static constexpr int kPlane = N * kRow;                      // and per k1 plane
  static constexpr int kStep = kThreads / kPlane;              // k1 planes per pass of the block
  static_assert(kThreads % kPlane == 0, "the threads cover whole k1 planes");
  int k1, k2, k3;   // centred indices: k1 of the first pass, k2, first k3
  bool on;          // has elements (N = 8: an x point is less than one pass)
  __device__ __forceinline__ XSums() {
    const int tid = threadIdx.x;
    k3 = (tid % kRow) * kV - N / 2;
    k2 = (tid / kRow) % N - N / 2;
    k1 = tid / kPlane - N / 2;
    on = tid < N * kPlane;
  }
  // this thread's sums over the x point at fx (wide: fx is 16-byte aligned): m; SQUARE: u of |k|^2 f;
  // else u of k1 f and v of k3 f
  template <bool SQUARE>
  __device__ __forceinline__ void add(const T* fx, bool wide, Run<T>& m, Run<T>& u, Run<T>& v) const {
    constexpr int kPasses = N >= kStep ? N / kStep : 1;
    if constexpr (sizeof(T) == 4) {
      const float4* p = reinterpret_cast<const float4*>(fx) + threadIdx.x;
      Run<float> t[4];
      u = Run<float>();
      if (on) {
#pragma unroll 8
        for (int i = 0; i < kPasses; ++i) {
          const float4 q = __ldcs(p + i * kThreads);
          const int k = k1 + i * kStep;
          const float w = (float)(SQUARE ? k * k : k);   // exact
          const float x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            two_sum_f(t[c].h, t[c].l, x[c]);
            const float pr = x[c] * w;
            u.l += fmaf(x[c], w, -pr);   // exact product residual
            two_sum_f(u.h, u.l, pr);
          }
        }
      }
      m = v = Run<float>();
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        m.add(t[c]);
        v.add(t[c], (float)(SQUARE ? k2 * k2 + (k3 + c) * (k3 + c) : k3 + c));
      }
      if (SQUARE) u.add(v);
    } else {
      const T* p = fx + 2 * threadIdx.x;
      double t0 = 0.0, t1 = 0.0, w = 0.0;
      if (on) {
#pragma unroll 8
        for (int i = 0; i < kPasses; ++i) {
          double2 q;
          if (wide) q = __ldcs(reinterpret_cast<const double2*>(p + 2 * i * kThreads));
          else q = make_double2(p[2 * i * kThreads], p[2 * i * kThreads + 1]);
          const int k = k1 + i * kStep;
          t0 += q.x;
          t1 += q.y;
          w = fma((double)(SQUARE ? k * k : k), q.x + q.y, w);
        }
      }
      m.s = t0 + t1;
      if (SQUARE) {
        w = fma((double)(k2 * k2 + k3 * k3), t0, w);
        w = fma((double)(k2 * k2 + (k3 + 1) * (k3 + 1)), t1, w);
      } else {
        v.s = fma((double)k3, m.s, t1);   // k3 t0 + (k3 + 1) t1
      }
      u.s = w;
    }
  }
};

// the sums over a block of NV values per thread, in a fixed order, to out[NV * block + c]
template <int NV>
__device__ __forceinline__ void block_sum_store(double (&v)[NV], double* __restrict__ out) {
  __shared__ double red[NV][32];
  const int tid = threadIdx.x;
#pragma unroll
  for (int c = 0; c < NV; ++c)
    for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_xor_sync(0xffffffffu, v[c], o);
  if ((tid & 31) == 0)
#pragma unroll
    for (int c = 0; c < NV; ++c) red[c][tid >> 5] = v[c];
  __syncthreads();
  if (tid == 0)
#pragma unroll
    for (int c = 0; c < NV; ++c) {
      double a = 0.0;
      for (int w = 0; w < (int)blockDim.x / 32; ++w) a += red[c][w];
      out[(int64_t)NV * blockIdx.x + c] = a;
    }
}

}  // namespace
}  // namespace chasm
