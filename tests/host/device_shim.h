// Host stand-ins of the device intrinsics that df64.cuh and closed_form.cuh
// use, so that a plain C++ compiler can run their arithmetic (compiled with
// -ffp-contract=off: every FP32 operation rounds once, as the _rn forms do).
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
#define __noinline__
struct float2 {
    float x, y;
};
using std::fmaf;
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __frcp_rn(float a) { return 1.0f / a; }
static inline float __int_as_float(int i) {
    float f;
    std::memcpy(&f, &i, sizeof f);
    return f;
}
template <class T>
static inline T __ldg(const T* p) {
    return *p;
}
