// Host stand-ins for the CUDA qualifiers and round-to-nearest intrinsics used by the
// library's binary64 solid code, so that the CPU baseline compiles that same code for the
// host (plain C++ built with -ffp-contract=off: every + - * rounds once, to nearest, as the
// intrinsics do on the device; / and sqrt are IEEE on both).
#pragma once
#include <cmath>
#include <cstdint>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__ __attribute__((noinline))

static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dsqrt_rn(double a) { return std::sqrt(a); }
using std::copysign;
using std::fabs;
using std::nan;
using std::sqrt;

// Stand-ins for what the binary32 passes (solid_fp32.cuh) use.  Reciprocal, division and
// reciprocal square root are correctly rounded here; the device's approximate ones lie within
// the passes' error bounds.
#include <cstring>
using std::fmaf;
using std::isfinite;
using std::isinf;
struct uint2 { uint32_t x, y; };
static inline uint2 make_uint2(uint32_t x, uint32_t y) { return {x, y}; }
template <class T> static inline T __ldg(const T* p) { return *p; }
template <class To, class From> static inline To shim_bits(From v) {
  To r;
  std::memcpy(&r, &v, sizeof(r));
  return r;
}
static inline float __uint_as_float(uint32_t v) { return shim_bits<float>(v); }
static inline uint32_t __float_as_uint(float v) { return shim_bits<uint32_t>(v); }
static inline long long __double_as_longlong(double v) { return shim_bits<long long>(v); }
static inline float __frcp_rn(float v) { return 1.0f / v; }
static inline float __fdividef(float a, float b) { return a / b; }
static inline float rsqrtf(float v) { return 1.0f / std::sqrt(v); }
static inline int __ffs(uint32_t v) { return __builtin_ffs((int)v); }
