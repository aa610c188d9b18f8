// Exact conversions between FP32 and FP64 with integer operations, off the
// low-rate FP64 pipe.
//
// The file compiles as CUDA (device functions) and as plain C++ (for tests).
#pragma once

#ifdef __CUDACC__
#define RT_FN __device__ __forceinline__
#else
#include <cmath>
#include <cstdint>
#include <cstring>
#define RT_FN static inline
#endif

namespace rtk {

#ifdef __CUDACC__
RT_FN long long bits_of(double v) { return __double_as_longlong(v); }
RT_FN double double_of(long long b) { return __longlong_as_double(b); }
RT_FN unsigned bits_of(float v) { return __float_as_uint(v); }
RT_FN float float_of(unsigned b) { return __uint_as_float(b); }
#else
RT_FN long long bits_of(double v) { long long b; std::memcpy(&b, &v, 8); return b; }
RT_FN double double_of(long long b) { double v; std::memcpy(&v, &b, 8); return v; }
RT_FN unsigned bits_of(float v) { unsigned b; std::memcpy(&b, &v, 4); return b; }
RT_FN float float_of(unsigned b) { float v; std::memcpy(&v, &b, 4); return v; }
#endif

// Exact widening of an FP32 value to FP64 with integer operations (rebias the
// exponent by 1023 - 127 and shift the significand), off the FP64 pipe.
// Subnormal and non-finite inputs take the ordinary conversion.
RT_FN double widen(float f) {
  const unsigned u = bits_of(f);
  const unsigned e = u & 0x7f800000u;
  if (e == 0u || e == 0x7f800000u) {
    if ((u & 0x7fffffffu) != 0u) return (double)f;
    return double_of((long long)((unsigned long long)u << 32));  // a zero keeps its sign
  }
  const unsigned hi = (((u & 0x7fffffffu) >> 3) + 0x38000000u) | (u & 0x80000000u);
  return double_of((long long)(((unsigned long long)hi << 32) | (unsigned long long)(u << 29)));
}

// FP64 to FP32 by cutting the significand to 24 bits, with integer
// operations; values outside the normal FP32 range take the ordinary
// conversion (a zero stays one).
RT_FN float cut(double v) {
  const long long b = bits_of(v);
  const int be = (int)((b >> 52) & 0x7ff);
  const unsigned top = (unsigned)((unsigned long long)b >> 32);
  if (be < 1023 - 126 || be > 1023 + 127) return (b << 1) == 0 ? float_of(top & 0x80000000u) : (float)v;
  return float_of((top & 0x80000000u) | ((unsigned)(be - 896) << 23) | ((unsigned)(b >> 29) & 0x7fffffu));
}

}  // namespace rtk
