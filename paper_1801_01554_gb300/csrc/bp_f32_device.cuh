// Device helpers shared by the float32 kernels.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "bp_internal.h"

namespace bp {
namespace {

constexpr unsigned long long kWaitNs = 2000000000ull;   // 2 s per wait
constexpr unsigned kWaitIters = 1u << 26;

// Checked build (-DBP_CHECK): phases test that their shared-memory regions fit
// the launch's dynamic shared memory and that their rows and tile origins lie
// inside their buffers; a failed test latches kFlagBounds (bp_check reports it)
// and the phase skips its accesses.  Without BP_CHECK the tests compile away.
extern __shared__ __align__(128) float g_dyn_smem[];   // every kernel's dynamic shared memory
__device__ __forceinline__ const float* pattern_smem_base() { return g_dyn_smem; }
__device__ __forceinline__ unsigned dyn_smem_floats() {
    unsigned b;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(b));
    return b / 4;
}
__device__ __forceinline__ bool bounds_ok(bool ok, int* flags) {
#ifdef BP_CHECK
    if (!ok) {
        atomicOr(flags, kFlagBounds);
        return false;
    }
#else
    (void)ok;
    (void)flags;
#endif
    return true;
}

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

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// Grid barrier for a cooperative launch.  bar[1] counts arrivals over every
// launch on the net; bar[0] holds its value at the end of the previous launch.
// Barrier k of a launch completes when the count reaches bar[0] + k * grid:
// thread 0 of each CTA adds its arrival with a fire-and-forget release
// reduction and then polls the count (no CTA has to relay a release).  The
// wait is bounded; on a timeout the error word latches kFlagTimeout and the
// function returns false in every thread of the CTA (the caller must then
// return).  Counts compare modulo 2^32.
__device__ __forceinline__ bool count_reached(unsigned v, unsigned target) {
    return (int)(v - target) >= 0;
}
__device__ bool grid_barrier(unsigned* bar, unsigned target, int* flags, unsigned long long limit_ns) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        // the release is cumulative: with the CTA barrier above it also orders
        // every thread's earlier writes before the arrival (no separate fence)
        asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar + 1), "r"(1u) : "memory");
        const unsigned long long t0 = global_ns();
        unsigned it = 0;
        while (!count_reached(ld_acquire(bar + 1), target)) {
            ++it;
            if (it > kWaitIters || ((it & 63u) == 0 && global_ns() - t0 > limit_ns)) {
                atomicOr(flags, kFlagTimeout);
                ok = 0;
                break;
            }
        }
    }
    return __syncthreads_and(ok) != 0;
}

// Limit of the grid barrier's wait: 2 s, or in the checked build the limit a
// test set on the net (bp_debug_wait_test), so that a test can make a wait run
// out in about a millisecond.
__device__ __forceinline__ unsigned long long wait_limit_ns(const F32View& v) {
#ifdef BP_CHECK
    return v.wait_ns != 0 ? v.wait_ns : kWaitNs;
#else
    (void)v;
    return kWaitNs;
#endif
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Programmatic dependent launch: wait for the kernels this one depends on (their
// writes are then visible), and let the next kernel of the stream start its setup.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

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

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// Orders this CTA's shared-memory writes, remote ones included, before the
// peers' reads after it (release / acquire at cluster scope).
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
// Stores x at p in CTA `rank`'s shared memory and counts its 4 bytes on that CTA's bar.
__device__ __forceinline__ void st_remote(float* p, uint64_t* bar, unsigned rank, float x) {
    uint32_t a, b;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(smem_u32(bar)), "r"(rank));
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
                 "r"(__float_as_uint(x)), "r"(b)
                 : "memory");
}
__device__ __forceinline__ void arm(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// Bounded wait for the bytes of a phase; false (kFlagTimeout latched) if it ran out.
__device__ __forceinline__ bool wait_bytes(uint64_t* bar, unsigned parity, int* flags, unsigned long long limit_ns) {
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 255u) == 0) {
            unsigned long long t;
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (it == 0) t0 = t;
            else if (t - t0 > limit_ns) {
                atomicOr(flags, kFlagTimeout);
                return false;
            }
        }
    }
}

// Pairs of floats in one 64-bit register: two multiply-adds (each rounded as fmaf)
// per issued instruction.  The multiply-add rate per SM is the same, so what they
// save is issue slots: in the passes of 32 patterns and the weight phase, groups of
// 4,096 of 203-120-26 took 31.1 -> 29.3 us per update.  The lane-group forward of
// smaller passes keeps single ones: it gained nothing from pairs of columns, which
// add up in another order.
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
__device__ __forceinline__ float sum2(f32x2 x) {
    const float2 t = unpack2(x);
    return t.x + t.y;
}
// Four consecutive floats as two pairs.
__device__ __forceinline__ ulonglong2 ld4x2(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }

// The fault guard's test without an atomic per change: zeroes and counts into n_bad.
__device__ __forceinline__ float guard_count(float guard, float g, unsigned& n_bad) {
    const bool bad = guard > 0.f && !(fabsf(g) <= guard);
    n_bad += bad ? 1u : 0u;
    return bad ? 0.f : g;
}

}  // namespace
}  // namespace bp
