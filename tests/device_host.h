// The device intrinsics that the integer arithmetic headers use, for a host
// build of those headers (tests/test_fixed_int_host.py).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>

using std::max;
using std::min;

template <typename To, typename From>
inline To bits_as(From v) {
  static_assert(sizeof(To) == sizeof(From), "");
  To t;
  std::memcpy(&t, &v, sizeof t);
  return t;
}
inline int __double2hiint(double x) { return (int)(bits_as<uint64_t>(x) >> 32); }
inline int __double2loint(double x) { return (int)(uint32_t)bits_as<uint64_t>(x); }
inline double __hiloint2double(int hi, int lo) { return bits_as<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); }
inline unsigned __float_as_uint(float f) { return bits_as<unsigned>(f); }
inline float __uint_as_float(unsigned u) { return bits_as<float>(u); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)(((((uint64_t)hi << 32) | lo) << (s & 31)) >> 32);
}
inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((uint64_t)hi << 32) | lo) >> (s & 31));
}
inline double __ll2double_rn(long long v) { return (double)v; }
inline long long __double2ll_rn(double x) { return std::llrint(x); }
inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
