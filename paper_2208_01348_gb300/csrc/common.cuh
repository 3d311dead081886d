// Shared device helpers: complex arithmetic on float2/double2, precision
// traits and launch-error plumbing.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };
template <typename R> using cx = typename Cx<R>::T;

template <typename C> __host__ __device__ __forceinline__ C mk(double re, double im) {
    C c; c.x = (decltype(c.x))re; c.y = (decltype(c.y))im; return c;
}
// Packed FP32 pairs (add/sub/fma.rn.f32x2, sm_100 and later): a complex addition
// in one issue slot, each half rounded as the scalar one is.  The lanes add at
// the same rate either way (measured: 118 scalar or 2 x 58 packed per clock and
// SM), but the FP32 transforms are bound by issue and latency, not by the adders:
// 128^3 matvec of 25 systems 962 -> 901 us, 64^3 of 200 842 -> 810 us, 160^3 of 4
// 530 -> 470 us.
#ifdef __CUDA_ARCH__
__device__ __forceinline__ unsigned long long pk2(float2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ float2 upk2(unsigned long long v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
#endif
__host__ __device__ __forceinline__ float2 operator+(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)));
    return upk2(r);
#else
    return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ float2 operator-(float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(pk2(a)), "l"(pk2(b)));
    return upk2(r);
#else
    return make_float2(a.x - b.x, a.y - b.y);
#endif
}
// s a + b with a real s
__host__ __device__ __forceinline__ float2 fma_s(float s, float2 a, float2 b) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(pk2(make_float2(s, s))), "l"(pk2(a)), "l"(pk2(b)));
    return upk2(r);
#else
    return make_float2(s * a.x + b.x, s * a.y + b.y);
#endif
}
__host__ __device__ __forceinline__ double2 fma_s(double s, double2 a, double2 b) {
    return make_double2(s * a.x + b.x, s * a.y + b.y);
}
__host__ __device__ __forceinline__ float2 operator*(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__host__ __device__ __forceinline__ float2 operator*(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__host__ __device__ __forceinline__ float2 operator-(float2 a) { return make_float2(-a.x, -a.y); }
__host__ __device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ double2 operator*(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__host__ __device__ __forceinline__ double2 operator*(double s, double2 a) { return make_double2(s * a.x, s * a.y); }
__host__ __device__ __forceinline__ double2 operator-(double2 a) { return make_double2(-a.x, -a.y); }

template <typename C> __host__ __device__ __forceinline__ C conj_(C a) { a.y = -a.y; return a; }
template <typename C> __host__ __device__ __forceinline__ auto abs2_(C a) { return a.x * a.x + a.y * a.y; }
// multiply by +i (INV=false gives -i): used by radix butterflies
template <typename C> __host__ __device__ __forceinline__ C mul_i(C a) { C r; r.x = -a.y; r.y = a.x; return r; }
template <typename C> __host__ __device__ __forceinline__ C mul_mi(C a) { C r; r.x = a.y; r.y = -a.x; return r; }

__host__ __device__ __forceinline__ float2 to_f(double2 a) { return make_float2((float)a.x, (float)a.y); }
__host__ __device__ __forceinline__ double2 to_d(float2 a) { return make_double2(a.x, a.y); }
template <typename C> __host__ __device__ __forceinline__ C cvt(double2 a);
template <> __host__ __device__ __forceinline__ double2 cvt<double2>(double2 a) { return a; }
template <> __host__ __device__ __forceinline__ float2 cvt<float2>(double2 a) { return to_f(a); }
template <typename C> __host__ __device__ __forceinline__ double2 widen(C a) { return make_double2(a.x, a.y); }

__host__ __device__ __forceinline__ double2 cdiv(double2 a, double2 b) {
    // Smith's algorithm
    if (fabs(b.x) >= fabs(b.y)) {
        double r = b.y / b.x, den = b.x + b.y * r;
        return make_double2((a.x + a.y * r) / den, (a.y - a.x * r) / den);
    } else {
        double r = b.x / b.y, den = b.x * r + b.y;
        return make_double2((a.x * r + a.y) / den, (a.y * r - a.x) / den);
    }
}
__host__ __device__ __forceinline__ double cabs_(double2 a) { return hypot(a.x, a.y); }

#ifdef __CUDACC__
// Programmatic dependent launch (launch_dep): a kernel may start while the one
// before it drains, and waits, before it touches memory, until it has finished;
// then it lets the next one start.
__device__ __forceinline__ void dep_wait(int on) {
    if (on) asm volatile("griddepcontrol.wait;\n griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

// Fixed-size per-system scalars of the solve (device resident).
#define EELS_MAX_MAT 8
