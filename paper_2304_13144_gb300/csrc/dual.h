// Scalars of the per-neighborhood kernels: float, double, and dual numbers over them (value and
// derivative along one direction), with the helpers that let one kernel serve all of them.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace mtp {
namespace {

template <class R>
struct alignas(2 * sizeof(R)) Dual {
  R v, d;
};
template <class R> __device__ __forceinline__ Dual<R> operator+(Dual<R> a, Dual<R> b) { return {a.v + b.v, a.d + b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(Dual<R> a, Dual<R> b) { return {a.v - b.v, a.d - b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator*(Dual<R> a, Dual<R> b) {
  return {a.v * b.v, a.d * b.v + a.v * b.d};
}
template <class R> __device__ __forceinline__ Dual<R> operator*(R s, Dual<R> b) { return {s * b.v, s * b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator*(Dual<R> b, R s) { return {s * b.v, s * b.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator+(Dual<R> a, R s) { return {a.v + s, a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(R s, Dual<R> a) { return {s - a.v, -a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator-(Dual<R> a, R s) { return {a.v - s, a.d}; }
template <class R> __device__ __forceinline__ Dual<R> operator/(Dual<R> a, Dual<R> b) {
  R inv = R(1) / b.v;
  return {a.v * inv, (a.d - a.v * inv * b.d) * inv};
}
template <class R> __device__ __forceinline__ Dual<R>& operator+=(Dual<R>& a, Dual<R> b) { a.v += b.v; a.d += b.d; return a; }

template <class S> struct Traits;
template <> struct Traits<float> { using R = float; };
template <> struct Traits<double> { using R = double; };
template <> struct Traits<Dual<float>> { using R = float; };
template <> struct Traits<Dual<double>> { using R = double; };

template <class S> __device__ __forceinline__ S mk(typename Traits<S>::R v) {
  if constexpr (std::is_same<S, typename Traits<S>::R>::value) return v;
  else return S{v, typename Traits<S>::R(0)};
}
template <class S> __device__ __forceinline__ S mk2(typename Traits<S>::R v, typename Traits<S>::R d) {
  if constexpr (std::is_same<S, typename Traits<S>::R>::value) return v;
  else return S{v, d};
}
template <class S> __device__ __forceinline__ typename Traits<S>::R vpart(S x) {
  if constexpr (std::is_same<S, typename Traits<S>::R>::value) return x;
  else return x.v;
}
template <class S> __device__ __forceinline__ typename Traits<S>::R dpart(S x) {
  if constexpr (std::is_same<S, typename Traits<S>::R>::value) return typename Traits<S>::R(0);
  else return x.d;
}
__device__ __forceinline__ float ssqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ double ssqrt(double x) { return sqrt(x); }
template <class R> __device__ __forceinline__ Dual<R> ssqrt(Dual<R> x) {
  R s = ssqrt(x.v);
  return {s, x.d / (R(2) * s)};
}
template <class S> __device__ __forceinline__ S shfl_xor(S x, int m) {
  if constexpr (std::is_same<S, typename Traits<S>::R>::value) return __shfl_xor_sync(0xffffffffu, x, m);
  else return S{__shfl_xor_sync(0xffffffffu, x.v, m), __shfl_xor_sync(0xffffffffu, x.d, m)};
}
template <class S> __device__ __forceinline__ S warp_sum(S x) {
  for (int m = 16; m; m >>= 1) x = x + shfl_xor(x, m);
  return x;
}

// a b + c with one rounding per component's last addition (3 FMAs for duals)
__device__ __forceinline__ float madd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double madd(double a, double b, double c) { return fma(a, b, c); }
template <class R> __device__ __forceinline__ Dual<R> madd(Dual<R> a, Dual<R> b, Dual<R> c) {
  return {madd(a.v, b.v, c.v), madd(a.d, b.v, madd(a.v, b.d, c.d))};
}
template <class R> __device__ __forceinline__ Dual<R> madd(R a, Dual<R> b, Dual<R> c) {
  return {madd(a, b.v, c.v), madd(a, b.d, c.d)};
}

}  // namespace
}  // namespace mtp
