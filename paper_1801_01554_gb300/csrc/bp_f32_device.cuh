// Device helpers shared by the float32 kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bp_internal.h"

namespace bp {
namespace {

// Logistic: CUDA's expf and the fast reciprocal divide (2 ulp, far inside the
// float32 bar; for 1 + e^-x beyond 2^126 the quotient is 0, the logistic's value).
__device__ __forceinline__ float sigmoid_f(float x) { return __fdividef(1.0f, 1.0f + expf(-x)); }

// Table-lookup logistic (Section 4.3, Figure 3): the logistic at 256 equally
// spaced points over [-15, 15], built in shared memory by each CTA that runs a
// forward pass with the table mode on.  Inputs outside the range take the end
// values; inside, x is remapped to [0, 255], the integer part picks the entry
// and the fractional part interpolates linearly to the next one.  NaN stays NaN.
constexpr int kSigPoints = 256;
__shared__ float s_sigtab[kSigPoints];

__device__ void sigmoid_table_init(const F32View& v) {
    if (v.sig_table)
        for (int k = threadIdx.x; k < kSigPoints; k += blockDim.x)
            s_sigtab[k] = sigmoid_f(-15.f + (30.f * (float)k) / (float)(kSigPoints - 1));
}

__device__ __forceinline__ float sigmoid_tab(float x) {
    if (x != x) return x;
    const float xc = fminf(fmaxf(x, -15.f), 15.f);
    const float x1 = (xc + 15.f) * ((float)(kSigPoints - 1) / 30.f);
    const int i = min((int)x1, kSigPoints - 2);   // x1 >= 0: truncation is the floor
    const float f = x1 - (float)i;
    const float t0 = s_sigtab[i];
    return fmaf(f, s_sigtab[i + 1] - t0, t0);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// Butterfly reduce-scatter of V per-lane values over aligned groups of V lanes:
// afterwards lane k of a group holds in v[0] the group's sum of value k mod V.
// A binary-tree sum (Section 10.3), V - 1 shuffles for V sums.
template <int V>
__device__ __forceinline__ void reduce_scatter(float (&v)[V], int lane) {
#pragma unroll
    for (int half = V / 2; half >= 1; half >>= 1) {
        const bool up = (lane & half) != 0;
#pragma unroll
        for (int k = 0; k < half; ++k) {
            const float send = up ? v[k] : v[k + half];
            const float keep = up ? v[k + half] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, send, half);
        }
    }
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// Pairs of floats in one 64-bit register: two multiply-adds (each rounded as fmaf)
// per issued instruction.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
    f32x2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 unpack2(f32x2 x) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(x));
    return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
// Four consecutive floats of shared memory as two pairs.
__device__ __forceinline__ ulonglong2 ld4x2(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

// The fault guard's test without an atomic per change: zeroes and counts into n_bad.
__device__ __forceinline__ float guard_count(float guard, float g, unsigned& n_bad) {
    const bool bad = guard > 0.f && !(fabsf(g) <= guard);
    n_bad += bad ? 1u : 0u;
    return bad ? 0.f : g;
}

}  // namespace
}  // namespace bp
