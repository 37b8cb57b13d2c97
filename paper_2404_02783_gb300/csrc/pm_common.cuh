// Common device-side types and helpers for the sm_103a particle-mesh library.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pm.h"

namespace pm {

// ------------------------------------------------------------------ launches that overlap their ramps
// The kernels of a step are launched so that each may start while the one before it on the stream
// drains (programmatic dependent launch): launch_next lets the next one in, and wait_previous
// holds this one until the kernels before it are complete and their writes visible.  Every such
// kernel calls it before its first access to anything an earlier kernel writes (the constant
// tables, uploaded once, may be read before), so the order of the stream holds; kernels launched
// in the ordinary way see the whole of it as before.  A chained kernel is resident while its
// predecessor still writes what it will read, so it reads that by plain loads: the non-coherent
// ones (__ldg, const __restrict__ parameters) ask for data that is constant as long as the kernel
// runs, which holds for the tables alone.  On small meshes, where a
// step is six kernels of a few microseconds, the ramps are a good part of the time: a step took
// 33.4 us at 32^3 and takes 22.2, 77.5 and 71.0 at 128^3, 470 and 453 at 256^3, 3848 and 3834 at 512^3.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A plain load that keeps its place among the other asm statements: the compiler does not gather
// many of them ahead of their use, which costs registers (58 for 48 in k_adj_kick).
__device__ __forceinline__ float load_ordered(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// overlap = false: an ordinary launch.
template <typename... K, typename... A>
cudaError_t launch_chained(void (*fn)(K...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, bool overlap,
                           A... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, fn, K(args)...);
}

// ------------------------------------------------------------------ type traits
template <typename T> struct CT;
template <> struct CT<float> { typedef float2 type; };
template <> struct CT<double> { typedef double2 type; };

template <typename T> using cplx = typename CT<T>::type;

template <typename C> __host__ __device__ __forceinline__ C cmake(decltype(C().x) a, decltype(C().x) b) {
    C c; c.x = a; c.y = b; return c;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
    C c; c.x = a.x * b.x - a.y * b.y; c.y = a.x * b.y + a.y * b.x; return c;
}
// a conj(b)
template <typename C> __device__ __forceinline__ C cmulc(C a, C b) {
    C c; c.x = a.x * b.x + a.y * b.y; c.y = a.y * b.x - a.x * b.y; return c;
}
template <typename C> __device__ __forceinline__ C cconj(C a) { a.y = -a.y; return a; }
template <typename C, typename T> __device__ __forceinline__ C cscale(C a, T s) { a.x *= s; a.y *= s; return a; }
// both parts in one instruction (packed FP32 add of sm_100 and later; the same roundings)
template <> __device__ __forceinline__ float2 cadd<float2>(float2 a, float2 b) {
    unsigned long long r, x = *reinterpret_cast<unsigned long long*>(&a), y = *reinterpret_cast<unsigned long long*>(&b);
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return *reinterpret_cast<float2*>(&r);
}
template <> __device__ __forceinline__ float2 csub<float2>(float2 a, float2 b) {
    unsigned long long r, x = *reinterpret_cast<unsigned long long*>(&a), y = *reinterpret_cast<unsigned long long*>(&b);
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return *reinterpret_cast<float2*>(&r);
}
// s a, and s a + c
__device__ __forceinline__ float2 mul2(float s, float2 a) {
    const float2 s2 = make_float2(s, s);
    unsigned long long r, x = *reinterpret_cast<const unsigned long long*>(&s2), y = *reinterpret_cast<unsigned long long*>(&a);
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(x), "l"(y));
    return *reinterpret_cast<float2*>(&r);
}
__device__ __forceinline__ float2 fma2(float s, float2 a, float2 c) {
    const float2 s2 = make_float2(s, s);
    unsigned long long r, x = *reinterpret_cast<const unsigned long long*>(&s2), y = *reinterpret_cast<unsigned long long*>(&a),
                          z = *reinterpret_cast<unsigned long long*>(&c);
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(x), "l"(y), "l"(z));
    return *reinterpret_cast<float2*>(&r);
}
// s a + c, each part rounded once
__device__ __forceinline__ float2 cfma(float s, float2 a, float2 c) { return fma2(s, a, c); }
__device__ __forceinline__ double2 cfma(double s, double2 a, double2 c) {
    return make_double2(fma(s, a.x, c.x), fma(s, a.y, c.y));
}
// multiply by -i (forward) or +i (inverse)
template <bool INV, typename C> __device__ __forceinline__ C cmul_mi(C a) {
    C c;
    if (INV) { c.x = -a.y; c.y = a.x; } else { c.x = a.y; c.y = -a.x; }
    return c;
}

// ------------------------------------------------------------------ constants
constexpr int kMaxLogN = 10;  // meshes up to 1024^3 in index arithmetic

__host__ __device__ __forceinline__ int ilog2(int n) {
    int l = 0;
    while ((1 << l) < n) ++l;
    return l;
}

// Signed wavenumber of FFT index i on an n-point axis: 0..n/2-1, -n/2..-1.
__device__ __forceinline__ int signed_k(int i, int n) { return i < (n >> 1) ? i : i - n; }

}  // namespace pm
