// Stand-in for the CUDA runtime header: lets g++ compile the register-level headers of csrc/ (the
// transforms' arithmetic, one thread at a time) for the tests of their range and accuracy.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __restrict__
#define __align__(n) alignas(n)
using std::max;
using std::min;
struct float2 { float x, y; };
struct float4 { float x, y, z, w; };
struct double2 { double x, y; };
struct int4 { int x, y, z, w; };
struct host_dim { unsigned x, y, z; };
static host_dim threadIdx{0, 0, 0}, blockDim{1, 1, 1};
inline float2 make_float2(float x, float y) { return {x, y}; }
inline double2 make_double2(double x, double y) { return {x, y}; }
inline int4 make_int4(int x, int y, int z, int w) { return {x, y, z, w}; }
template <class To, class From> inline To host_bits(From v) {
    static_assert(sizeof(To) == sizeof(From), "same size");
    To r;
    std::memcpy(&r, &v, sizeof(r));
    return r;
}
inline unsigned __float_as_uint(float v) { return host_bits<unsigned>(v); }
inline float __uint_as_float(unsigned v) { return host_bits<float>(v); }
inline long long __double_as_longlong(double v) { return host_bits<long long>(v); }
inline double __longlong_as_double(long long v) { return host_bits<double>(v); }
inline int __double2hiint(double v) { return (int)(host_bits<long long>(v) >> 32); }
inline int __double2loint(double v) { return (int)host_bits<long long>(v); }
inline double __hiloint2double(int h, int l) { return host_bits<double>((unsigned long long)(unsigned)h << 32 | (unsigned)l); }
inline float __double2float_rn(double v) { return (float)v; }
inline float __int2float_rn(int v) { return (float)v; }
inline float __fadd_rn(float a, float b) { return a + b; }
inline float __fsub_rn(float a, float b) { return a - b; }
inline float __fmul_rn(float a, float b) { return a * b; }
inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)((unsigned long long)a * b >> 32); }
inline unsigned __funnelshift_l(unsigned lo, unsigned hi, int s) { return (unsigned)(((unsigned long long)hi << 32 | lo) << (s & 31) >> 32); }
template <class T> inline T __ldg(const T* p) { return *p; }
inline unsigned __cvta_generic_to_shared(const void*) { return 0; }
inline void __syncthreads() {}
template <class T> inline T atomicOr(T* p, T v) { T o = *p; *p |= v; return o; }
