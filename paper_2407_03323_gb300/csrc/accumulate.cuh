// Sums of complex lag products.  FP64 plainly; FP32 with an error-free two-sum (Knuth), so that
// the accumulation over up to ell lags adds no error beyond one rounding of the compensated total.
#pragma once

#include <cuda_runtime.h>

template <typename R> struct Acc;

template <> struct Acc<double> {
    double2 s;
    __device__ void zero() { s = make_double2(0.0, 0.0); }
    __device__ void add(double2 v) { s.x += v.x; s.y += v.y; }
    __device__ double2 get() const { return s; }
    __device__ void merge(int o) {           // add lane ^ o's sum
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
    }
};

__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = a + b;
    const float bp = s - a;
    const float ap = s - bp;
    e = (a - ap) + (b - bp);
}

template <> struct Acc<float> {
    float2 s, c;
    __device__ void zero() { s = make_float2(0.f, 0.f); c = make_float2(0.f, 0.f); }
    __device__ void add(float2 v) {
        float e;
        two_sum(s.x, v.x, s.x, e); c.x += e;
        two_sum(s.y, v.y, s.y, e); c.y += e;
    }
    __device__ float2 get() const { return make_float2(s.x + c.x, s.y + c.y); }
    __device__ void merge(int o) {
        const float cx = __shfl_xor_sync(0xffffffffu, c.x, o), cy = __shfl_xor_sync(0xffffffffu, c.y, o);
        add(make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o)));
        c.x += cx;
        c.y += cy;
    }
};
