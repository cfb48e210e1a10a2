// CUDA's qualifiers and device functions for device code compiled for the host
// (the approximate functions within their error).
#pragma once

#include <math.h>
#include <stdint.h>

#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
static inline float __fdividef(float a, float b) { return a / b; }
static inline float rsqrtf(float a) { return (float)(1.0 / sqrt((double)a)); }
#define __logf logf
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
