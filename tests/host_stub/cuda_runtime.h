// The few CUDA names that csrc/fx.cuh and csrc/device.cuh use, for a host compiler: their device
// functions are plain C++ but for the warp intrinsics, which no host test calls.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

#define __device__
#define __host__
#define __global__
#define __shared__
#define __forceinline__ inline
#define __noinline__
#define __restrict__

struct double2 {
  double x, y;
};
struct int4 {
  int x, y, z, w;
};
inline double2 make_double2(double x, double y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
template <typename T>
inline T __ldg(const T* p) {
  return *p;
}
inline long long __double_as_longlong(double d) {
  long long r;
  std::memcpy(&r, &d, 8);
  return r;
}
inline double __longlong_as_double(long long l) {
  double r;
  std::memcpy(&r, &l, 8);
  return r;
}
inline int __float_as_int(float f) {
  int r;
  std::memcpy(&r, &f, 4);
  return r;
}
inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
inline void __syncwarp(unsigned = 0) {}
template <typename T>
inline T __shfl_xor_sync(unsigned, T v, int) {
  return v;
}
inline int __any_sync(unsigned, int p) { return p; }
using std::abs;
using std::fma;
using std::max;
using std::min;
