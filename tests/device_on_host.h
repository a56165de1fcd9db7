// The device arithmetic of paper_2107_12027_gb300/csrc built for the host: CUDA's qualifiers
// and the intrinsics those headers call, in IEEE arithmetic.  Contractions that the GPU's
// compiler makes are not made here.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <type_traits>

#include <cuda_runtime.h>
#undef __device__
#undef __forceinline__
#undef __noinline__
#undef __global__
#undef __host__
#undef __launch_bounds__
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __global__
#define __host__
#define __launch_bounds__(...)
#define __maxnreg__(x)

static inline double __drcp_rn(double x) { return 1.0 / x; }
static inline float __frcp_rn(float x) { return 1.0f / x; }
static inline double rsqrt(double x) { return 1.0 / std::sqrt(x); }
static inline float rsqrtf(float x) { return (float)(1.0 / std::sqrt((double)x)); }
static inline double __dadd_rn(double a, double b) { return a + b; }
static inline double __dsub_rn(double a, double b) { return a - b; }
static inline double __dmul_rn(double a, double b) { return a * b; }
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
struct HostIndex { unsigned x, y, z; };
static HostIndex host_index_;
#define blockIdx host_index_
#define threadIdx host_index_
#define blockDim host_index_
#define gridDim host_index_
template <typename T> static T atomicAdd(T *a, T b) { T o = *a; *a += b; return o; }
using std::max;
using std::min;
