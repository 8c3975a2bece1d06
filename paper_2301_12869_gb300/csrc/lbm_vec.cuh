// Value types of the fused step's per-node arithmetic: float, double, and f2, a
// pair of FP32 values (two neighbouring nodes) held in one 64-bit register and
// processed by sm_100-family packed FP32 instructions (add/sub/mul/fma .rn.f32x2).
// The per-node physics in lbm_kernels.cu is written once over these types.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace lbm {

struct f2 {
  unsigned long long v;
};

__device__ __forceinline__ f2 make_f2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lo(f2 x) {
  float a;
  [[maybe_unused]] float b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
  return a;
}
__device__ __forceinline__ float hi(f2 x) {
  [[maybe_unused]] float a;
  float b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
  return b;
}
__device__ __forceinline__ f2 operator+(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator-(f2 a, f2 b) {
  f2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 operator*(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}

// a * b + c with one rounding
__device__ __forceinline__ float fmadd(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmadd(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ f2 fmadd(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// constants and conversions
template <typename V>
struct VecTraits;
template <>
struct VecTraits<float> {
  using scalar = float;
  static constexpr int width = 1;
  __device__ static float cst(double c) { return float(c); }
};
template <>
struct VecTraits<double> {
  using scalar = double;
  static constexpr int width = 1;
  __device__ static double cst(double c) { return c; }
};
template <>
struct VecTraits<f2> {
  using scalar = float;
  static constexpr int width = 2;
  __device__ static f2 cst(double c) { return make_f2(float(c), float(c)); }
};
template <typename V>
__device__ __forceinline__ V cst(double c) {
  return VecTraits<V>::cst(c);
}

// Division and square root: IEEE in FP64 (the FP64 path is checked to 1e-14); in FP32
// the fast intrinsics __fdividef (<= 2 ulp) and rsqrtf (<= 2 ulp), and for node pairs the
// approximate reciprocal and square root instructions (rcp.approx / sqrt.approx, a few
// ulp), add at most a few ulp, far inside the FP32 path's 1e-6 bound against the FP64
// oracle.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double fast_div(double a, double b) { return a / b; }
__device__ __forceinline__ float fast_div(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ f2 fast_div(f2 a, f2 b) { return a * make_f2(rcp_approx(lo(b)), rcp_approx(hi(b))); }

// sqrt of max(x, 0); sets `bad` when x < 0 or NaN (psi undefined)
__device__ __forceinline__ double sqrt_checked(double x, bool& bad) {
  if (!(x >= 0.0)) {
    bad = true;
    x = 0.0;
  }
  return sqrt(x);
}
__device__ __forceinline__ float sqrt_checked(float x, bool& bad) {
  if (!(x >= 0.f)) {
    bad = true;
    x = 0.f;
  }
  return x > 0.f ? x * rsqrtf(x) : 0.f;
}
__device__ __forceinline__ f2 sqrt_checked(f2 x, bool& bad) {
  const float s = lo(x), t = hi(x);
  if (!(s >= 0.f) || !(t >= 0.f)) bad = true;
  return make_f2(sqrt_approx(fmaxf(s, 0.f)), sqrt_approx(fmaxf(t, 0.f)));
}

// true if any component is <= 0 or NaN
__device__ __forceinline__ bool nonpositive(double x) {
  // a positive normal number is told by its high word: the FP64 pipe is left alone
  return unsigned(__double2hiint(x)) - 0x00100000u >= 0x7fe00000u && !(x > 0.0);
}
__device__ __forceinline__ bool nonpositive(float x) { return !(x > 0.f); }
__device__ __forceinline__ bool nonpositive(f2 x) { return !(lo(x) > 0.f) || !(hi(x) > 0.f); }

// a value of type V from a double (one component)
template <typename V>
__host__ __device__ V from_double(double x);
template <>
__host__ __device__ inline float from_double<float>(double x) {
  return float(x);
}
template <>
__host__ __device__ inline double from_double<double>(double x) {
  return x;
}

// sum of the components in FP64
__device__ __forceinline__ double hsum(double x) { return x; }
__device__ __forceinline__ double hsum(float x) { return double(x); }
__device__ __forceinline__ double hsum(f2 x) { return double(lo(x)) + double(hi(x)); }

// FP64 <-> FP32 conversions share the slow FP64 pipe with the additions (2 lanes a clock and SM), so
// for a whole state they cost more than its memory traffic. These form the same values with integer
// instructions; zero, infinities, NaN and what is denormal in FP32 take the conversion, out of line:
// inline it was issued for every value, if only predicated off (a 1024 x 4096 state in and out 65 us more).
static __device__ __noinline__ float narrow_slowly(double d) { return float(d); }
static __device__ __noinline__ double widen_slowly(float f) { return double(f); }
__device__ __forceinline__ float narrow(double d) {  // to the nearest FP32, ties to even
  const uint32_t h = uint32_t(__double2hiint(d)), l = uint32_t(__double2loint(d));
  const uint32_t e = (h >> 20) & 0x7ffu;
  if (e - 897u >= 253u) return narrow_slowly(d);  // 2^-126 <= |d| < 2^127 otherwise
  uint32_t m = ((h & 0x7fffffffu) - (896u << 20)) << 3 | l >> 29;  // exponent and 23 bits, truncated
  m += ((l & 0x1fffffffu) + 0x0fffffffu + (m & 1u)) >> 29;          // the 29 bits below round it
  return __uint_as_float(m | (h & 0x80000000u));
}
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t e = (b >> 23) & 0xffu;
  if (e - 1u >= 254u) return widen_slowly(f);
  return __hiloint2double(int((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), int(b << 29));
}
__device__ __forceinline__ double narrow_to(double d, double) { return d; }
__device__ __forceinline__ float narrow_to(double d, float) { return narrow(d); }
__device__ __forceinline__ double widen(double d) { return d; }

}  // namespace lbm
