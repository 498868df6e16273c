// Complex element types of the grid product and their traits.
//   float2  : complex64 ("mixed" precision)
//   dfc     : double-float complex, FP64-class accuracy on the FP32 pipe (default FP64 mode)
//   double2 : IEEE binary64 complex (native FP64 mode)
#pragma once

#include "dfloat.cuh"
#include "fft_reg.cuh"

namespace aim {

template <typename CT> struct GridT;
// W: column-tile width (W * sizeof(CT) = 32 bytes); VT: type of restricted grid values handed
// to the gather; MaxThreads: launch bound (16-byte types hold 32 x 16 bytes per thread).
// MaxThreads is the launch bound with one transform of 16 elements per thread (TPT = 1); with two
// transforms per thread (TPT = 2) a CTA of the same work has half the threads, with 8 elements
// per thread twice as many (at most 1024).
template <> struct GridT<float2> {
  using VT = float2;
  static constexpr int W = 4, MaxThreads = 1024;
};
template <> struct GridT<double2> {
  using VT = double2;
  static constexpr int W = 2, MaxThreads = 512;
};
template <> struct GridT<dfc> {
  using VT = double2;
  static constexpr int W = 2, MaxThreads = 512;
};
// a double-float complex product is ~40 FP32-pipe instructions: twiddles come whole from the table
template <> struct TwiddleFromTable<dfc> { static constexpr bool value = true; };

template <typename CT, int TPT, int LOGE> struct LaunchMax {
  // fewer elements per thread: the same registers per thread hold the work of fewer elements,
  // so the same register file holds more threads
  static constexpr int base = TPT == 1 ? GridT<CT>::MaxThreads : GridT<CT>::MaxThreads / 2;
  static constexpr int value = (base << (4 - LOGE)) > 1024 ? 1024 : (base << (4 - LOGE));
};

constexpr int kWideMax = 512;   // launch bound of the wide variants (wide_pass)

template <typename CT> __device__ __forceinline__ CT czero();
template <> __device__ __forceinline__ float2 czero<float2>() { return float2{0.f, 0.f}; }
template <> __device__ __forceinline__ double2 czero<double2>() { return double2{0.0, 0.0}; }
template <> __device__ __forceinline__ dfc czero<dfc>() { return dfc{0.f, 0.f, 0.f, 0.f}; }

template <typename CT> __device__ __forceinline__ CT cfrom(double re, double im);
template <> __device__ __forceinline__ float2 cfrom<float2>(double re, double im) {
  return float2{(float)re, (float)im};
}
template <> __device__ __forceinline__ double2 cfrom<double2>(double re, double im) { return double2{re, im}; }
template <> __device__ __forceinline__ dfc cfrom<dfc>(double re, double im) {
  dfc r;
  df_split(re, r.xh, r.xl);
  df_split(im, r.yh, r.yl);
  return r;
}

__device__ __forceinline__ double2 cto_d2(float2 v, double s) { return double2{(double)v.x * s, (double)v.y * s}; }
__device__ __forceinline__ double2 cto_d2(double2 v, double s) { return double2{v.x * s, v.y * s}; }
__device__ __forceinline__ double2 cto_d2(dfc v, double s) {
  return double2{((double)v.xh + (double)v.xl) * s, ((double)v.yh + (double)v.yl) * s};
}

// value handed to the gather (restricted grid value times the 1/P^2 of the inverse DFT)
__device__ __forceinline__ float2 cto_vt(float2 v, double s) { return float2{v.x * (float)s, v.y * (float)s}; }
__device__ __forceinline__ double2 cto_vt(double2 v, double s) { return cto_d2(v, s); }
__device__ __forceinline__ double2 cto_vt(dfc v, double s) { return cto_d2(v, s); }

// one part (0: real, 1: imaginary) of cto_vt
__device__ __forceinline__ float cto_vt_part(float2 v, int part, double s) { return (part ? v.y : v.x) * (float)s; }
__device__ __forceinline__ double cto_vt_part(double2 v, int part, double s) { return (part ? v.y : v.x) * s; }
__device__ __forceinline__ double cto_vt_part(dfc v, int part, double s) {
  const float h = part ? v.yh : v.xh, l = part ? v.yl : v.xl;
  return ((double)h + (double)l) * s;
}

// tables of double-float values are float4 (xh, yh, xl, yl), the order of dfc
__device__ __forceinline__ dfc ldro(const dfc* p) {
  const float4 v = __ldg(reinterpret_cast<const float4*>(p));
  return dfc{v.x, v.y, v.z, v.w};
}

// two neighbouring values as one vector access: 32 bytes for the 16-byte types (p 32-byte aligned),
// 16 bytes for complex64 (p 16-byte aligned)
__device__ __forceinline__ void store_pair(float2* p, float2 a, float2 b) {
  *reinterpret_cast<float4*>(p) = float4{a.x, a.y, b.x, b.y};
}
__device__ __forceinline__ void store_pair(double2* p, double2 a, double2 b) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}
__device__ __forceinline__ void store_pair(dfc* p, dfc a, dfc b) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.xh), "f"(a.yh), "f"(a.xl),
               "f"(a.yl), "f"(b.xh), "f"(b.yh), "f"(b.xl), "f"(b.yl)
               : "memory");
}
__device__ __forceinline__ void load_pair(const float2* p, float2& a, float2& b) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  a = float2{v.x, v.y};
  b = float2{v.z, v.w};
}
__device__ __forceinline__ void load_pair(const double2* p, double2& a, double2& b) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(a.x), "=d"(a.y), "=d"(b.x), "=d"(b.y) : "l"(p) : "memory");
}
__device__ __forceinline__ void load_pair(const dfc* p, dfc& a, dfc& b) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(a.xh), "=f"(a.yh), "=f"(a.xl), "=f"(a.yl), "=f"(b.xh), "=f"(b.yh), "=f"(b.xl), "=f"(b.yl)
               : "l"(p)
               : "memory");
}

// value held by the partner lane (lane ^ 1); all 32 lanes must call it together
__device__ __forceinline__ float2 shfl_pair(float2 v) {
  return float2{__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ double2 shfl_pair(double2 v) {
  return double2{__shfl_xor_sync(0xffffffffu, v.x, 1), __shfl_xor_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ dfc shfl_pair(dfc v) {
  dfc r;
  r.xh = __shfl_xor_sync(0xffffffffu, v.xh, 1);
  r.yh = __shfl_xor_sync(0xffffffffu, v.yh, 1);
  r.xl = __shfl_xor_sync(0xffffffffu, v.xl, 1);
  r.yl = __shfl_xor_sync(0xffffffffu, v.yl, 1);
  return r;
}

}  // namespace aim
