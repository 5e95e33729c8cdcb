// Complex FP32 arithmetic of the mixed form's plane kernels, typed views of an instance's plane
// buffers and twiddle tables, and the small DFT butterflies shared by the shared-memory
// Stockham plane kernels (pcf_kernels.cu) and the warp-register plane kernels
// (pcf_planes_warp.cu).
#pragma once
#include "pcf_kernels.cuh"

namespace pcf {

// ------------------------------------------------------------------ helpers

// x-storage index i (m = i for i <= Kx, m = i - Mx otherwise) -> FFT bin
__device__ __forceinline__ int xbin(int i, int Kx, int Mx, int nx) { return i <= Kx ? i : nx - (Mx - i); }

// ------------------------------------------------------------------ complex helpers
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

template <class T> struct Cx;
template <> struct Cx<float> {
  using c = float2;
  static __device__ __forceinline__ float2 mk(float a, float b) { return make_float2(a, b); }
};

// plane sums of q^2 are kept in FP64
__device__ __forceinline__ void acc_sq(double* s, float q) { *s = fma((double)q, (double)q, *s); }

// typed views of an instance's plane buffers and twiddles
template <class T> __device__ __forceinline__ T* phys_of(const Inst& I);
template <> __device__ __forceinline__ float* phys_of<float>(const Inst& I) { return I.physf; }
template <class T> __device__ __forceinline__ const typename Cx<T>::c* yv_of(const Inst& I);
template <> __device__ __forceinline__ const float2* yv_of<float>(const Inst& I) { return I.yvf; }
template <class T> __device__ __forceinline__ typename Cx<T>::c* xz_of(const Inst& I);
template <> __device__ __forceinline__ float2* xz_of<float>(const Inst& I) { return I.xzf; }
template <class T> __device__ __forceinline__ const typename Cx<T>::c* twx_of(const Inst& I);
template <> __device__ __forceinline__ const float2* twx_of<float>(const Inst& I) { return I.twxf; }
template <class T> __device__ __forceinline__ const typename Cx<T>::c* twz_of(const Inst& I);
template <> __device__ __forceinline__ const float2* twz_of<float>(const Inst& I) { return I.twzf; }

// ------------------------------------------------------------------ Stockham FFT in shared memory
template <int R, class C>
__device__ __forceinline__ void butterfly(C* v, bool inv);

template <>
__device__ __forceinline__ void butterfly<2, float2>(float2* v, bool) {
  const float2 a = v[0], b = v[1];
  v[0] = cadd(a, b);
  v[1] = csub(a, b);
}

template <int R, class C>
__device__ __forceinline__ void butterfly4(C* v, bool inv) {
  const C t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
  const C t2 = cadd(v[1], v[3]), d = csub(v[1], v[3]);
  // t3 = -i d (forward) or +i d (inverse)
  C t3;
  if (inv) { t3.x = -d.y; t3.y = d.x; } else { t3.x = d.y; t3.y = -d.x; }
  v[0] = cadd(t0, t2);
  v[2] = csub(t0, t2);
  v[1] = cadd(t1, t3);
  v[3] = csub(t1, t3);
}
template <>
__device__ __forceinline__ void butterfly<4, float2>(float2* v, bool inv) { butterfly4<4, float2>(v, inv); }

template <class C>
__device__ __forceinline__ void butterfly3(C* v, bool inv) {
  using R = decltype(v[0].x);
  const R h = (R)0.86602540378443864676;  // sin(2 pi/3)
  const C s = cadd(v[1], v[2]), d = csub(v[1], v[2]);
  const C y0 = cadd(v[0], s);
  C m, it;
  m.x = fma((R)-0.5, s.x, v[0].x);
  m.y = fma((R)-0.5, s.y, v[0].y);
  // forward: y1 = m - i t, y2 = m + i t with t = h d
  it.x = -h * d.y;
  it.y = h * d.x;
  v[0] = y0;
  v[1] = inv ? cadd(m, it) : csub(m, it);
  v[2] = inv ? csub(m, it) : cadd(m, it);
}
template <>
__device__ __forceinline__ void butterfly<3, float2>(float2* v, bool inv) { butterfly3(v, inv); }

// ------------------------------------------------------------------ twiddled butterflies
// A Stockham pass of radix R with Ns > 1 multiplies input r of butterfly k by w^(r q1),
// q1 = k * twstep, w = exp(-2 pi i/L) (its conjugate for the inverse transform; tw[q] = w^q),
// then applies the radix-R DFT.
template <class C>
struct TwStd {
  const C* tw;
};

// The twiddled radix-R butterfly of a pass (Ns > 1), input r of butterfly k at v[r].
template <int R, class C>
__device__ __forceinline__ void tw_butterfly(C* v, const TwStd<C>& T, int k, int twstep, int L, bool inv) {
#pragma unroll
  for (int r = 1; r < R; ++r) {
    C w = T.tw[r * k * twstep];
    if (inv) w.y = -w.y;
    v[r] = cmul(v[r], w);
  }
  butterfly<R, C>(v, inv);
}

}  // namespace pcf
