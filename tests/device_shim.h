// What the device headers under csrc take from CUDA, for a host compiler: the
// intrinsics by their definitions, one thread, no runtime.  A test that compiles
// them includes this file in place of cuda_runtime.h.
#pragma once
#include <math.h>
#include <stddef.h>
#include <stdint.h>
#include <string.h>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__

enum cudaError_t { cudaSuccess = 0 };
typedef struct CUstream_st *cudaStream_t;
template <class T> static inline cudaError_t cudaMemcpyFromSymbol(void *, const T &, size_t) { return cudaSuccess; }
template <class T> static inline cudaError_t cudaMemcpyToSymbol(const T &, const void *, size_t) { return cudaSuccess; }
struct float2 {
    float x, y;
};
static inline float2 make_float2(float x, float y) { return float2{x, y}; }

template <class To, class From>
static inline To bits_as(From x)
{
    static_assert(sizeof(To) == sizeof(From), "");
    To y;
    memcpy(&y, &x, sizeof(y));
    return y;
}
static inline long long __double_as_longlong(double x) { return bits_as<long long>(x); }
static inline double __longlong_as_double(long long x) { return bits_as<double>(x); }
static inline float __uint_as_float(unsigned x) { return bits_as<float>(x); }
static inline int __double2hiint(double x) { return (int)(bits_as<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)(uint32_t)bits_as<uint64_t>(x); }
static inline double __hiloint2double(int h, int l) { return bits_as<double>((uint64_t)(uint32_t)h << 32 | (uint32_t)l); }
static inline uint32_t __funnelshift_l(uint32_t lo, uint32_t hi, int s) { return (uint32_t)((((uint64_t)hi << 32 | lo) << s) >> 32); }
static inline int __mulhi(int a, int b) { return (int)(((int64_t)a * b) >> 32); }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((uint64_t)a * b) >> 32); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b)
{
    return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline int __clz(int v) { return v ? __builtin_clz((unsigned)v) : 32; }
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }
static inline int __ffs(unsigned v) { return __builtin_ffs((int)v); }
static inline int __popc(unsigned v) { return __builtin_popcount(v); }
template <class T> static inline T __ldg(const T *p) { return *p; }
static inline float __frcp_rn(float x) { return 1.0f / x; }
static int g_skew;  // rsqrtf on the GPU is within 2 ulp: skewed either way here
static inline float rsqrtf(float x) { return (1.0f / sqrtf(x)) * (1.0f + 1.2e-7f * (float)(g_skew++ % 3 - 1)); }
static inline double rsqrt(double x) { return 1.0 / sqrt(x); }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __double2float_rn(double x) { return (float)x; }
static inline float __int2float_rn(int x) { return (float)x; }
static inline float __ll2float_rn(long long x) { return (float)x; }
static inline float __ull2float_rn(unsigned long long x) { return (float)x; }
#define __logf logf
#define __expf expf
// one thread
static const struct { unsigned x; } threadIdx = {0};
static inline unsigned __ballot_sync(unsigned, bool p) { return p ? 1u : 0u; }
template <class T> static inline T __shfl_sync(unsigned, T v, int) { return v; }
template <class T> static inline T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T, class U> static inline T atomicAdd(T *p, U v) { const T o = *p; *p += v; return o; }
template <class T, class U> static inline T atomicOr(T *p, U v) { const T o = *p; *p |= v; return o; }
