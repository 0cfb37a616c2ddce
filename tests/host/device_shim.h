// CUDA intrinsics of the device headers as host functions, so that a plain C++
// compiler can run the per-cell device code (round to nearest, no contraction).
// Warp-wide sums return the calling lane's share.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>

using std::max;
using std::min;

template <class D, class S>
inline D bits_as(S s) {
    static_assert(sizeof(D) == sizeof(S), "same size");
    D d;
    std::memcpy(&d, &s, sizeof d);
    return d;
}
inline double __dmul_rn(double a, double b) { return a * b; }
inline double __dadd_rn(double a, double b) { return a + b; }
inline double __dsub_rn(double a, double b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline float2 __fadd2_rn(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
inline float2 __fmul2_rn(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
inline float2 __ffma2_rn(float2 a, float2 b, float2 c) {
    return make_float2(std::fma(a.x, b.x, c.x), std::fma(a.y, b.y, c.y));
}
inline int __double2hiint(double d) { return (int)(bits_as<uint64_t>(d) >> 32); }
inline int __double2loint(double d) { return (int)(uint32_t)bits_as<uint64_t>(d); }
inline double __hiloint2double(int h, int l) {
    return bits_as<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l);
}
inline long long __double_as_longlong(double d) { return bits_as<long long>(d); }
inline double __longlong_as_double(long long v) { return bits_as<double>(v); }
inline unsigned __float_as_uint(float f) { return bits_as<unsigned>(f); }
inline float __uint_as_float(unsigned u) { return bits_as<float>(u); }
inline double __ll2double_rn(long long v) { return (double)v; }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
    return (unsigned)((((uint64_t)hi << 32 | lo) << (s & 31)) >> 32);
}
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
template <class T>
inline T __ldg(const T* p) {
    return *p;
}
inline int __reduce_add_sync(unsigned, int v) { return v; }
inline double __shfl_down_sync(unsigned, double, int) { return 0.0; }
