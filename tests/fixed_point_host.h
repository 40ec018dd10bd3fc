// Host stand-ins for the device functions that the fixed-point headers use, so that a host compiler
// can build and check them.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#define __host__
#define __device__
#define __global__
#define __forceinline__ inline
#define __noinline__
using std::fma;
using std::isfinite;
using std::max;
using std::min;
using std::scalbn;

template <typename To, typename From>
To host_bits(From v) {
  To t;
  std::memcpy(&t, &v, sizeof(To));
  return t;
}
inline int __double2hiint(double v) { return (int)(host_bits<uint64_t>(v) >> 32); }
inline int __double2loint(double v) { return (int)(uint32_t)host_bits<uint64_t>(v); }
inline double __hiloint2double(int h, int l) { return host_bits<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
inline double __longlong_as_double(long long x) { return host_bits<double>(x); }
inline long long __double_as_longlong(double x) { return host_bits<long long>(x); }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
inline int __mulhi(int a, int b) { return (int)(((long long)a * b) >> 32); }
inline int __float_as_int(float v) { return host_bits<int>(v); }
inline unsigned __float_as_uint(float v) { return host_bits<unsigned>(v); }
inline long long __double2ll_rn(double x) { return std::llrint(x); }
template <typename T>
T __shfl_xor_sync(unsigned, T v, int) { return v; }
