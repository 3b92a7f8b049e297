// The names of CUDA that the pairs of csrc/ use, on the host: lets a CPU test
// call the functions of the FP64 pairs.  A warp is 32 threads that meet in
// every shuffle and vote.
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <pthread.h>

#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __shared__ static
#define __constant__
#define __launch_bounds__(...)

typedef int cudaError_t;
typedef void *cudaStream_t;

struct uint4 {
    uint32_t x, y, z, w;
};
static inline uint4 make_uint4(uint32_t x, uint32_t y, uint32_t z, uint32_t w) { return uint4{x, y, z, w}; }
static const struct { unsigned x; } threadIdx = {0}, blockDim = {1};
static inline void __syncthreads() {}

static thread_local int host_lane = 0;
static pthread_barrier_t host_warp;             // of 32
static uint64_t host_words[32];
template <typename T, typename F> static inline T host_exchange(T v, F from)
{
    uint64_t w = 0;
    memcpy(&w, &v, sizeof v);
    host_words[host_lane] = w;
    pthread_barrier_wait(&host_warp);
    const int l = from(host_lane);
    w = host_words[l >= 0 && l < 32 ? l : host_lane];
    pthread_barrier_wait(&host_warp);
    memcpy(&v, &w, sizeof v);
    return v;
}
template <typename T> static inline T __shfl_sync(unsigned, T v, int l) { return host_exchange(v, [=](int) { return l & 31; }); }
template <typename T> static inline T __shfl_up_sync(unsigned, T v, int d) { return host_exchange(v, [=](int l) { return l - d; }); }
template <typename T> static inline T __shfl_down_sync(unsigned, T v, int d) { return host_exchange(v, [=](int l) { return l + d; }); }
template <typename T> static inline T __shfl_xor_sync(unsigned, T v, int d) { return host_exchange(v, [=](int l) { return l ^ d; }); }
static inline unsigned __ballot_sync(unsigned, bool p)
{
    host_words[host_lane] = p;
    pthread_barrier_wait(&host_warp);
    unsigned m = 0;
    for (int l = 0; l < 32; ++l) m |= (unsigned)host_words[l] << l;
    pthread_barrier_wait(&host_warp);
    return m;
}
static inline bool __all_sync(unsigned m, bool p) { return __ballot_sync(m, p) == 0xffffffffu; }
static inline int __popc(unsigned x) { return __builtin_popcount(x); }
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }

template <typename A, typename B> static inline A host_bits(B b)
{
    A a;
    memcpy(&a, &b, sizeof a);
    return a;
}
static inline uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)((uint64_t)a * b >> 32); }
static inline uint32_t __float_as_uint(float x) { return host_bits<uint32_t>(x); }
static inline float __uint_as_float(uint32_t x) { return host_bits<float>(x); }
static inline float __uint2float_rn(uint32_t x) { return (float)x; }
static inline int __float2int_rz(float x) { return x < 2147483648.0f ? (int)x : 2147483647; }
static inline float __int2float_rn(int x) { return (float)x; }
static inline int __double2hiint(double x) { return (int)(host_bits<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)host_bits<uint64_t>(x); }
static inline float __fdividef(float a, float b) { return a / b; }
#define __expf expf
static inline float __frcp_rn(float x) { return 1.0f / x; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float rsqrtf(float x) { return 1.0f / sqrtf(x); }
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline void sincospi(double x, double *s, double *c) { *s = sin(M_PI * x); *c = cos(M_PI * x); }
static inline void sincospif(float x, float *s, float *c) { *s = (float)sin(M_PI * x); *c = (float)cos(M_PI * x); }
static inline double sinpi(double x) { return sin(M_PI * x); }
static inline float sinpif(float x) { return (float)sin(M_PI * x); }
// 2^52 + floor(q) for 0 <= q < 2^31
static inline double __dadd_rd(double q, double) { return 4503599627370496.0 + floor(q); }
template <typename T> static inline T min(T a, T b) { return a < b ? a : b; }
template <typename T> static inline T max(T a, T b) { return a > b ? a : b; }
