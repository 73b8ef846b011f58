// What a host build of the one-kernel branch-and-bound (direct.cuh) needs of
// CUDA: one thread runs a whole team (T = G = 1, one CTA), so barriers do
// nothing and a warp has one lane.  Included by the file direct_host.py makes.
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>
using std::isfinite;
using std::max;
using std::min;
#define __device__
#define __host__
#define __global__
#define __forceinline__ inline
#define __noinline__
#define __launch_bounds__(...)
#define __restrict__
#define __shared__ static
#define __align__(x)
static long long host_count[2][8];   // calls and sums by what is counted
#define LMS_DIRECT_COUNT(what, n) (++host_count[0][what], host_count[1][what] += (n))
struct int2 { int x, y; };
struct int4 { int x, y, z, w; };
struct uint4 { unsigned x, y, z, w; };
struct float2 { float x, y; };
struct double2 { double x, y; };
struct longlong2 { long long x, y; };
static inline int2 make_int2(int a, int b) { return {a, b}; }
static inline int4 make_int4(int a, int b, int c, int d) { return {a, b, c, d}; }
static inline uint4 make_uint4(unsigned a, unsigned b, unsigned c, unsigned d) { return {a, b, c, d}; }
static struct { unsigned x, y, z; } threadIdx = {0, 0, 0}, blockIdx = {0, 0, 0}, blockDim = {1, 1, 1};
#define __syncthreads()
#define __syncwarp()
static inline int __syncthreads_or(int v) { return v; }
static inline int __any_sync(unsigned, bool p) { return p; }
static inline unsigned __ballot_sync(unsigned, bool p) { return p; }
template <class T> T __shfl_xor_sync(unsigned, T v, int) { return v; }
template <class T> T __shfl_up_sync(unsigned, T v, int) { return v; }
template <class T> T __shfl_sync(unsigned, T v, int) { return v; }
template <class T> T __reduce_min_sync(unsigned, T v) { return v; }
template <class T> T __reduce_max_sync(unsigned, T v) { return v; }
template <class T> T __reduce_add_sync(unsigned, T v) { return v; }
template <class T, class U> T atomicAdd(T *p, U v) { T o = *p; *p += v; return o; }
template <class T, class U> T atomicMin(T *p, U v) { T o = *p; if ((T)v < o) *p = v; return o; }
template <class T, class U> T atomicMax(T *p, U v) { T o = *p; if ((T)v > o) *p = v; return o; }
template <class T, class U> T atomicOr(T *p, U v) { T o = *p; *p |= v; return o; }
template <class T> T atomicCAS(T *p, T c, T v) { T o = *p; if (o == c) *p = v; return o; }
template <class T> T __ldcg(const T *p) { return *p; }
template <class T> T __ldg(const T *p) { return *p; }
static inline int __popc(unsigned v) { return __builtin_popcount(v); }
static inline int __clz(int v) { return v ? __builtin_clz(v) : 32; }
static inline int __clzll(long long v) { return v ? __builtin_clzll(v) : 64; }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
template <class A, class B> A bits_as(B b) { A a; static_assert(sizeof a == sizeof b); memcpy(&a, &b, sizeof a); return a; }
static inline float __int_as_float(int v) { return bits_as<float>(v); }
static inline int __float_as_int(float v) { return bits_as<int>(v); }
static inline long long __double_as_longlong(double v) { return bits_as<long long>(v); }
static inline double __longlong_as_double(long long v) { return bits_as<double>(v); }
static inline float __fmul_ru(float a, float b)
{
    const float r = a * b;
    return (double)r < (double)a * b ? nextafterf(r, INFINITY) : r;
}
static inline float __ll2float_ru(long long v)
{
    const float r = (float)v;
    return (long double)r < (long double)v ? nextafterf(r, INFINITY) : r;
}
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fdividef(float a, float b) { return a / b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline unsigned __float2uint_rz(float f) { return (unsigned)f; }
static inline int __double2int_rn(double v) { return (int)nearbyint(v); }
static inline double __ddiv_rn(double a, double b) { return a / b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dadd_rn(double a, double b) { return a + b; }
#define fminf std::min<float>
#define fmaxf std::max<float>
// the sorting helpers of common.cuh, by the standard library
template <class T, class F> bool cta_fill_merge_sort_any(T *s, T *s2, int P, F fill)
{
    for (int k = 0; k < P; ++k) s[k] = fill(k);
    std::sort(s, s + P);
    for (int k = 0; k < P; ++k) s2[k] = 0;   // scratch
    return true;
}
template <int Q, class T, class F> T *cta_sort_chunked(T *, T *A, T *B, int P, F key)
{
    cta_fill_merge_sort_any(A, B, P, key);
    return A;
}
