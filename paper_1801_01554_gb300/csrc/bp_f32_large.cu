// float32 training of one-hidden-layer nets in large groups.
//
// Every CTA trains its share of the group's patterns (Section 4.1's case
// parallelism), kP at a time, with all weights in shared memory and the sums of
// its changes on chip for the whole group: 256 threads, each with a block of
// TU x 12 changes of [W_1 | b_1], kept in tensor memory between its uses, and one of
// 4 x 4 of [W_2 | b_2] in registers.  Inputs, activations and deltas of a pass never
// leave shared memory (the hidden deltas replace the activations), so a group costs
// one read of its patterns and, at its end, one parameter vector of sums per CTA:
// after a grid barrier every CTA adds its share of the words over the CTAs in a fixed
// order, applies the momentum update of Section 6.2.1 and, after a second barrier,
// copies the new weights in.
//
// No sum runs in one chain: net inputs add up 16 columns at a time, changes 32
// patterns at a time (kCols, kChain), CTAs in four chains and a tree.  With one chain
// each, 431 patterns long at groups of 65,536, a change's error against float64 was up to
// half as large again as that of the tiled weight phase; now it is smaller (2-norm of W_1's
// change, tiled / one chain / this: 203-60-26 by 16,384 1.65e-7 / 2.4e-7 / 1.6e-7, by 65,536
// 1.3e-7 / 1.8e-7 / 1.0e-7; 64-50-10 by 65,536 8.6e-8 / 1.2e-7 / 6.5e-8).
//
// All five products are register-blocked: 4 patterns x 8 units in layer 1 (12
// float4 loads for 128 multiply-adds), 4 x 2 in layer 2, 4 x 8 in the hidden
// deltas, TU x 12 and 4 x 4 for the changes (5 loads for 96, 2 for 16, per
// pattern).  What bounds it is shared memory's way into the registers, 128 bytes a
// clock whatever the lanes share: a pass of 64 patterns of 203-120-26 takes 65,000
// clocks, 26,000 in layer 1 (20,000 of loads, 13,000 of multiply-adds), 15,000 in
// the changes of W_1 (12,300 of multiply-adds), 6,000 for the rows.  Tensor memory frees the
// registers that layer 1's two levels of sums need (kept in registers, W_1's sums made it
// spill and cost a fifth); adding to them there takes about 700 clocks for TU = 8.
// us per update, tiled weight phase (k_train) -> this kernel: 203-120-26 at groups of
// 8,192: 52.8 -> 45.1, 16,384: 103.5 -> 76.7, 65,536: 349 -> 242; 203-60-26 at 65,536:
// 391 -> 157; 64-50-10: 140 -> 88.  The changes run over the rows a pass has: 9,729 patterns, a
// second pass of one row, take 67 us (79 when it summed 64), 11,777 of 203-90-26 68 (75; tiled 71).
//
// Which nets: one block of each product per thread (plan_tu), for 203 inputs up to 120 hidden
// units, for 255 up to 88; wider ones keep the tiled weight phase.
#include <cuda_runtime.h>

#include "bp_f32_device.cuh"
#include "bp_internal.h"

namespace bp {
namespace {

constexpr int kT = 256;
constexpr int kChain = 32;   // patterns of one chain of a change's sum
constexpr int kCols = 16;    // columns of one chain of a net input

struct LargePlan {
    int w1, w2, x, h, d, t, red, total;   // shared-memory offsets (floats)
    int xp, hp, dp;   // pitches of the input and activation rows (an odd number of float4, so that
                      // consecutive rows' float4 reads spread over the banks) and of the output deltas
};

template <int TU>
struct LargeCfg {
    static constexpr int kP = TU == 8 ? 64 : 128;   // patterns of a pass
    static constexpr int kPG = kP / 4;              // pattern groups: patterns pg, pg + kPG, ..
    // patterns between additions to the sums of W_1 in tensor memory (at TU = 8 the registers
    // hold one level of sums only)
    static constexpr int kMerge = TU == 8 ? kChain : kP;
};

__device__ __forceinline__ float4 add4(float4 x, float4 y) { return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w); }

// A float4 of a row of changes whose bias is component `last` (or lies further on).
__device__ __forceinline__ float4 pads_cleared(float4 x, int last) {
    return make_float4(x.x, last >= 1 ? x.y : 0.f, last >= 2 ? x.z : 0.f, last >= 3 ? x.w : 0.f);
}

// A thread's TU x 12 sums of changes of W_1 in its lane of tensor memory, columns from
// taddr on, 16 at a time.
__device__ __forceinline__ void sums_st16(uint32_t taddr, const f32x2 (&x)[8]) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float2 t = unpack2(x[i]);
        r[2 * i] = __float_as_uint(t.x);
        r[2 * i + 1] = __float_as_uint(t.y);
    }
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]),
        "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]),
        "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void sums_ld16(uint32_t taddr, f32x2 (&x)[8]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = pack2(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1]));
}
__device__ __forceinline__ void sums_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
template <int TU>
__device__ __forceinline__ void clear_sums(uint32_t taddr) {
    const f32x2 z[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    for (int w = 0; w < TU * 12; w += 16) sums_st16(taddr + w, z);
    sums_wait_st();
}
template <int TU>
__device__ __forceinline__ void load_sums(uint32_t taddr, f32x2 (&g)[TU][6]) {
#pragma unroll
    for (int w = 0; w < TU * 12; w += 16) {
        f32x2 x[8];
        sums_ld16(taddr + w, x);
#pragma unroll
        for (int i = 0; i < 8; ++i) g[(w / 2 + i) / 6][(w / 2 + i) % 6] = x[i];
    }
}
template <int TU>
__device__ __forceinline__ void add_sums(uint32_t taddr, const f32x2 (&g)[TU][6]) {
#pragma unroll
    for (int w = 0; w < TU * 12; w += 16) {
        f32x2 x[8];
        sums_ld16(taddr + w, x);
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = add2(x[i], g[(w / 2 + i) / 6][(w / 2 + i) % 6]);
        sums_st16(taddr + w, x);
    }
    sums_wait_st();
}

template <int TU>
__global__ void __launch_bounds__(kT, 1)
    k_train_large(const __grid_constant__ F32View v, const __grid_constant__ LargePlan c, const float* X, const float* T,
                  int n_patterns, int minibatch, int n_steps, float* sse_out, int fold_g) {
    constexpr int P = LargeCfg<TU>::kP, PG = LargeCfg<TU>::kPG;
    constexpr int kMerge = LargeCfg<TU>::kMerge;
    constexpr int kTmem = 2 * 12 * TU <= 128 ? 128 : 256;   // columns of tensor memory
    extern __shared__ __align__(128) float sm[];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ float s_sse[kT / 32];
    __shared__ uint32_t s_tmem;
    if (!bounds_ok((unsigned)c.total <= dyn_smem_floats(), v.flags)) return;   // in every CTA alike
    // a latched timeout means an earlier launch left the barrier half-way
    if (__ldcg(v.flags) & kFlagTimeout) return;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = v.n[0], H = v.n[1], n2 = v.n[2], kp1 = v.kp[1], kp2 = v.kp[2], xp = c.xp, hp = c.hp, dp = c.dp;
    const bool table = v.sig_table != 0;
    const float lr = v.lr * v.grad_scale, mom = v.momentum;
    unsigned phase = 0;
    sigmoid_table_init(v);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s_bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "n"(kTmem) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    unsigned target = __ldcg(v.bar);
    // pads: the true unit's 1 after the inputs and the activations, zeros after it
    for (int e = tid; e < P * (kp1 - n0); e += kT) {
        const int r = e / (kp1 - n0), i = n0 + e - r * (kp1 - n0);
        sm[c.x + r * xp + i] = i == n0 ? 1.f : 0.f;
    }
    for (int e = tid; e < P * (kp2 - H); e += kT) {
        const int r = e / (kp2 - H), i = H + e - r * (kp2 - H);
        sm[c.h + r * hp + i] = i == H ? 1.f : 0.f;
    }
    for (int e = tid; e < P * dp; e += kT) sm[c.d + e] = 0.f;
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // this thread's sums of W_1 between the passes: two warps a lane quarter
    const uint32_t tmem = s_tmem, own = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)(warp >> 2) * (TU * 12);
    auto leave = [&] {   // every thread: the CTA's tensor memory is given back
        __syncthreads();
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(kTmem) : "memory");
    };

    // this thread's blocks
    const int pg = tid % PG, ug = tid / PG;            // layer 1: patterns pg + PG i, units ug + UG j
    const int UG = (H + 7) / 8;
    const bool l1 = ug < UG, hid = l1;                 // hidden deltas: units 8 ug .. 8 ug + 7
    const int C1 = (kp1 + 11) / 12;
    const int cg1 = tid % C1, ur1 = tid / C1;          // W_1 changes: rows TU ur1 .., columns 12 cg1 ..
    const bool w1c = ur1 * TU < H;
    const int C2 = kp2 / 4;
    const int cg2 = tid % C2, kr2 = tid / C2;          // W_2 changes: rows 4 kr2 .., columns 4 cg2 ..
    const bool w2c = 4 * kr2 < n2;
    const float* W1 = sm + c.w1;
    const float* W2 = sm + c.w2;

    for (int s = 0; s < n_steps; ++s) {
        const long long g0 = (long long)s * minibatch;
        const long long B = min((long long)minibatch, (long long)n_patterns - g0);
        const long long lo = g0 + B * blockIdx.x / gridDim.x, hi = g0 + B * (blockIdx.x + 1) / gridDim.x;
        // weights: one bulk copy each of W_1 and W_2 (both padded row blocks are whole 16-byte words)
        if (tid == 0) {
            asm volatile("fence.proxy.async.global;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            unsigned lost = 0;
#ifdef BP_CHECK
            lost = v.debug_stall != 0 ? 16u : 0u;   // test hook: the copy waits for bytes that never come
#endif
            arm(&s_bar, (unsigned)v.P * 4u + lost);
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             smem_u32(sm + c.w1)),
                         "l"(v.theta), "r"((unsigned)v.P * 4u), "r"(smem_u32(&s_bar))
                         : "memory");
        }
        float g2[4][4], sse = 0.f;
        clear_sums<TU>(own);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
            for (int q = 0; q < 4; ++q) g2[u][q] = 0.f;
        bool have_w = false, ok = true;
        for (long long p0 = lo; p0 < hi || !have_w; p0 += P) {
            const int np = (int)max(0LL, min((long long)P, hi - p0));
            const int np4 = (np + 3) & ~3;   // rows that the sums of changes run over
            // rows of this pass; those past the share are zero
            for (int r = warp; r < P; r += kT / 32) {
                float* dst = sm + c.x + r * xp;
                if (r < np) {
                    const float* src = X + (p0 + r) * n0;
#pragma unroll 8
                    for (int i = lane; i < n0; i += 32) cp_async4(dst + i, src + i);
                } else {
                    for (int i = lane; i < n0; i += 32) dst[i] = 0.f;
                }
            }
            for (int e = tid; e < np * n2; e += kT) cp_async4(sm + c.t + e, T + p0 * n2 + e);
            cp_async_commit();
            if (!have_w) {
                ok = wait_bytes(&s_bar, phase, v.flags, wait_limit_ns(v));
                if (!ok) wait_bytes(&s_bar, phase, v.flags, wait_limit_ns(v));   // let a late copy land
                phase ^= 1u;
                have_w = true;
            }
            cp_async_wait<0>();
            ok = __syncthreads_and(ok) != 0;
            if (!ok) return leave();   // the copy did not arrive: no update
            if (np == 0) break;
            // the next pass's rows on their way to L2
            {
                const long long pn = p0 + P;
                const int nn = (int)max(0LL, min((long long)P, hi - pn)) * n0;
                for (int e = tid * 32; e < nn; e += kT * 32)
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(X + pn * n0 + e));
            }
            // 1. layer 1
            if (l1) {
                float acc[4][8];
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
                const float* xr = sm + c.x + pg * xp;
                int wo[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) wo[j] = min(ug + UG * j, H - 1) * kp1;
                auto columns = [&](int k, float (&sum)[4][8]) {
                    float4 x[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) x[i] = ld4(xr + PG * i * xp + k);
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float4 w = ld4(W1 + wo[j] + k);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            sum[i][j] = fmaf(w.x, x[i].x, sum[i][j]);
                            sum[i][j] = fmaf(w.y, x[i].y, sum[i][j]);
                            sum[i][j] = fmaf(w.z, x[i].z, sum[i][j]);
                            sum[i][j] = fmaf(w.w, x[i].w, sum[i][j]);
                        }
                    }
                };
                int k = 0;
                for (; k + kCols <= kp1; k += kCols) {
                    float blk[4][8];
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j) blk[i][j] = 0.f;
#pragma unroll 2
                    for (int q = 0; q < kCols; q += 4) columns(k + q, blk);
#pragma unroll
                    for (int i = 0; i < 4; ++i)
#pragma unroll
                        for (int j = 0; j < 8; ++j) acc[i][j] += blk[i][j];
                }
                for (; k < kp1; k += 4) columns(k, acc);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const int u = ug + UG * j;
                    if (u < H)
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            sm[c.h + (pg + PG * i) * hp + u] = table ? sigmoid_tab(acc[i][j]) : sigmoid_f(acc[i][j]);
                }
            }
            __syncthreads();
            // 2. outputs, error sum, output deltas
            for (int t = tid; t < PG * ((n2 + 1) / 2); t += kT) {
                const int pp = t % PG, k0 = t / PG * 2, k1 = min(k0 + 1, n2 - 1);
                float acc[4][2];
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = 0.f;
                const float* hr = sm + c.h + pp * hp;
                auto columns = [&](int k, float (&sum)[4][2]) {
                    const float4 wa = ld4(W2 + k0 * kp2 + k), wb = ld4(W2 + k1 * kp2 + k);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float4 h = ld4(hr + PG * i * hp + k);
                        sum[i][0] = fmaf(wa.x, h.x, sum[i][0]);
                        sum[i][1] = fmaf(wb.x, h.x, sum[i][1]);
                        sum[i][0] = fmaf(wa.y, h.y, sum[i][0]);
                        sum[i][1] = fmaf(wb.y, h.y, sum[i][1]);
                        sum[i][0] = fmaf(wa.z, h.z, sum[i][0]);
                        sum[i][1] = fmaf(wb.z, h.z, sum[i][1]);
                        sum[i][0] = fmaf(wa.w, h.w, sum[i][0]);
                        sum[i][1] = fmaf(wb.w, h.w, sum[i][1]);
                    }
                };
                int k = 0;
                for (; k + kCols <= kp2; k += kCols) {
                    float blk[4][2];
#pragma unroll
                    for (int i = 0; i < 4; ++i) blk[i][0] = blk[i][1] = 0.f;
#pragma unroll
                    for (int q = 0; q < kCols; q += 4) columns(k + q, blk);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        acc[i][0] += blk[i][0];
                        acc[i][1] += blk[i][1];
                    }
                }
                for (; k < kp2; k += 4) columns(k, acc);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int p = pp + PG * i;
#pragma unroll
                    for (int j = 0; j < 2; ++j) {
                        if (k0 + j >= n2) continue;
                        const float o = table ? sigmoid_tab(acc[i][j]) : sigmoid_f(acc[i][j]);
                        const float err = p < np ? sm[c.t + p * n2 + k0 + j] - o : 0.f;
                        sse = fmaf(err, err, sse);
                        sm[c.d + p * dp + k0 + j] = err * o * (1.f - o);
                    }
                }
            }
            __syncthreads();
            // 3. hidden sums (kept in registers) and the changes of W_2
            float hd[4][8];
            if (hid) {
#pragma unroll
                for (int i = 0; i < 4; ++i)
#pragma unroll
                    for (int j = 0; j < 8; ++j) hd[i][j] = 0.f;
                const float* wr = W2 + 8 * ug;   // past the last unit: the bias column and pads, or the next row; not used
                const float* dr = sm + c.d + pg * dp;
                for (int k = 0; k < n2; k += 4) {
                    float4 d[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) d[i] = ld4(dr + PG * i * dp + k);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int kk = min(k + q, n2 - 1);   // deltas past the last output are zero
                        const float4 wa = ld4(wr + kk * kp2), wb = ld4(wr + kk * kp2 + 4);
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float dq = q == 0 ? d[i].x : q == 1 ? d[i].y : q == 2 ? d[i].z : d[i].w;
                            hd[i][0] = fmaf(dq, wa.x, hd[i][0]);
                            hd[i][1] = fmaf(dq, wa.y, hd[i][1]);
                            hd[i][2] = fmaf(dq, wa.z, hd[i][2]);
                            hd[i][3] = fmaf(dq, wa.w, hd[i][3]);
                            hd[i][4] = fmaf(dq, wb.x, hd[i][4]);
                            hd[i][5] = fmaf(dq, wb.y, hd[i][5]);
                            hd[i][6] = fmaf(dq, wb.z, hd[i][6]);
                            hd[i][7] = fmaf(dq, wb.w, hd[i][7]);
                        }
                    }
                }
            }
            if (w2c) {
                const float* dr = sm + c.d + 4 * kr2;
                const float* hr = sm + c.h + 4 * cg2;
                for (int pc = 0; pc < np4; pc += kChain) {
                    float l2[4][4];
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int q = 0; q < 4; ++q) l2[u][q] = 0.f;
#pragma unroll 4
                    for (int p = pc; p < min(pc + kChain, np4); ++p) {
                        const float4 d = ld4(dr + p * dp), h = ld4(hr + p * hp);
                        const float dv[4] = {d.x, d.y, d.z, d.w}, hx[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
                        for (int u = 0; u < 4; ++u)
#pragma unroll
                            for (int q = 0; q < 4; ++q) l2[u][q] = fmaf(dv[u], hx[q], l2[u][q]);
                    }
#pragma unroll
                    for (int u = 0; u < 4; ++u)
#pragma unroll
                        for (int q = 0; q < 4; ++q) g2[u][q] += l2[u][q];
                }
            }
            __syncthreads();
            // hidden deltas replace the activations
            if (hid) {
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    float* hr = sm + c.h + (pg + PG * i) * hp + 8 * ug;
#pragma unroll
                    for (int j = 0; j < 8; ++j)
                        if (8 * ug + j < H) {
                            const float a = hr[j];
                            hr[j] = hd[i][j] * a * (1.f - a);
                        }
                }
            }
            __syncthreads();
            // 4. the changes of W_1
            {
                const float* dr = sm + c.h + TU * ur1;
                const float* xr = sm + c.x + 12 * cg1;
                for (int pm = 0; pm < np4; pm += kMerge) {
                    f32x2 g1[TU][6];   // sums of kMerge patterns, pairs of columns
#pragma unroll
                    for (int u = 0; u < TU; ++u)
#pragma unroll
                        for (int q = 0; q < 6; ++q) g1[u][q] = 0;
                    if (w1c)
                        for (int pc = pm; pc < min(pm + kMerge, np4); pc += kChain) {
                            f32x2 l1[TU][6];   // of one chain
#pragma unroll
                            for (int u = 0; u < TU; ++u)
#pragma unroll
                                for (int q = 0; q < 6; ++q) l1[u][q] = 0;
#pragma unroll 2
                            for (int p = pc; p < min(pc + kChain, np4); ++p) {
                                f32x2 xv[6];
#pragma unroll
                                for (int q = 0; q < 3; ++q) {
                                    const ulonglong2 x = ld4x2(xr + p * xp + 4 * q);
                                    xv[2 * q] = x.x;
                                    xv[2 * q + 1] = x.y;
                                }
#pragma unroll
                                for (int u = 0; u < TU; u += 4) {
                                    const float4 d = ld4(dr + p * hp + u);
                                    const f32x2 dd[4] = {pack2(d.x, d.x), pack2(d.y, d.y), pack2(d.z, d.z), pack2(d.w, d.w)};
#pragma unroll
                                    for (int t = 0; t < 4; ++t)
#pragma unroll
                                        for (int q = 0; q < 6; ++q) l1[u + t][q] = fma2(dd[t], xv[q], l1[u + t][q]);
                                }
                            }
#pragma unroll
                            for (int u = 0; u < TU; ++u)
#pragma unroll
                                for (int q = 0; q < 6; ++q)
                                    g1[u][q] = kMerge > kChain ? add2(g1[u][q], l1[u][q]) : l1[u][q];
                        }
                    __syncwarp();
                    add_sums<TU>(own, g1);
                }
            }
            __syncthreads();   // the rows may be overwritten
        }
        // this CTA's sums; those of a row's padding columns are 0 (their inputs are 0, but 0
        // times a NaN or an infinite delta is NaN)
        float* gp = v.gpart + (long long)blockIdx.x * v.P;
        f32x2 g1[TU][6];
        load_sums<TU>(own, g1);
        if (w1c) {
#pragma unroll
            for (int u = 0; u < TU; ++u)
#pragma unroll
                for (int q = 0; q < 12; q += 4)
                    if (TU * ur1 + u < H && 12 * cg1 + q < kp1) {
                        const float2 a = unpack2(g1[u][q / 2]), b = unpack2(g1[u][q / 2 + 1]);
                        __stcg(reinterpret_cast<float4*>(gp + v.woff[1] + (long long)(TU * ur1 + u) * kp1 + 12 * cg1 + q),
                               pads_cleared(make_float4(a.x, a.y, b.x, b.y), n0 - 12 * cg1 - q));
                    }
        }
        if (w2c) {
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (4 * kr2 + u < n2)
                    __stcg(reinterpret_cast<float4*>(gp + v.woff[2] + (long long)(4 * kr2 + u) * kp2 + 4 * cg2),
                           pads_cleared(make_float4(g2[u][0], g2[u][1], g2[u][2], g2[u][3]), H - 4 * cg2));
        }
        sse = warp_sum(sse);
        if (lane == 0) s_sse[warp] = sse;
        __syncthreads();
        if (tid == 0) {
            float e = 0.f;
            for (int k = 0; k < kT / 32; ++k) e += s_sse[k];
            __stcg(v.sse_part + blockIdx.x, e);
        }
        if (!grid_barrier(v.bar, target += gridDim.x, v.flags, wait_limit_ns(v))) return leave();
        if (blockIdx.x == gridDim.x - 1 && warp == 0) {
            float e = 0.f;
            for (int k = lane; k < (int)gridDim.x; k += 32) e += __ldcg(v.sse_part + k);
            e = warp_sum(e);
            if (lane == 0) {
                if (sse_out != nullptr) sse_out[s] = e;
                if (!isfinite(e)) atomicOr(v.flags, kFlagNonfinite);
            }
        }
        // this CTA's share of the words: nj float4 from j0 on, SL threads each adding
        // every SL-th CTA's sums, then the SL sums in order
        const long long P4 = v.P >> 2;
        const int j0 = (int)(P4 * blockIdx.x / gridDim.x), nj = (int)(P4 * (blockIdx.x + 1) / gridDim.x) - j0;
        const int njp = min(nj, kT), SL = njp > 0 ? min(kT / njp, 16) : 0;
        float4* red = reinterpret_cast<float4*>(sm + c.red);
        for (int jb = 0; jb < nj; jb += njp) {
            const int sl = tid / njp, j = jb + tid - sl * njp;
            const bool mine = sl < SL && j < nj, owner = mine && sl == 0;
            const long long word = j0 + j;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), vo = a, th = a, go = a;
            if (owner) {
                vo = __ldcg(reinterpret_cast<const float4*>(v.V) + word);
                th = __ldcg(reinterpret_cast<const float4*>(v.theta) + word);
                if (fold_g && s == 0) go = __ldcg(reinterpret_cast<const float4*>(v.G) + word);
            }
            if (mine) {
                const float4* src = reinterpret_cast<const float4*>(v.gpart) + word;
                float4 f[4] = {a, a, a, a};   // four chains, then their tree
                const int n_cta = (int)gridDim.x;
                int k = sl;
                for (; k + 7 * SL < n_cta; k += 8 * SL) {
                    float4 t[8];
#pragma unroll
                    for (int q = 0; q < 8; ++q) t[q] = __ldcg(src + (long long)(k + q * SL) * P4);
#pragma unroll
                    for (int q = 0; q < 8; ++q) f[q & 3] = add4(f[q & 3], t[q]);
                }
#pragma unroll
                for (int q = 0; q < 7; ++q)
                    if (k + q * SL < n_cta) f[q & 3] = add4(f[q & 3], __ldcg(src + (long long)(k + q * SL) * P4));
                a = add4(add4(f[0], f[1]), add4(f[2], f[3]));
                red[sl * njp + (j - jb)] = a;
            }
            __syncthreads();
            if (owner) {
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                float4 f[4] = {z, z, z, z};
                for (int k = 0; k < SL; k += 4)
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (k + q < SL) f[q] = add4(f[q], red[(k + q) * njp + (j - jb)]);
                a = add4(add4(f[0], f[1]), add4(f[2], f[3]));
                float g[4] = {a.x + go.x, a.y + go.y, a.z + go.z, a.w + go.w};
                float* vv = &vo.x;
                float* tt = &th.x;
                unsigned n_bad = 0;
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    g[q] = guard_count(v.guard, g[q], n_bad);
                    vv[q] = lr * g[q] + mom * vv[q];
                    tt[q] += vv[q];
                }
                if (n_bad != 0) atomicAdd(v.faults, n_bad);
                __stcg(reinterpret_cast<float4*>(v.V) + word, vo);
                __stcg(reinterpret_cast<float4*>(v.theta) + word, th);
                if (fold_g && s == 0) __stcg(reinterpret_cast<float4*>(v.G) + word, make_float4(0.f, 0.f, 0.f, 0.f));
            }
            __syncthreads();
        }
        // the next group's bulk copy reads theta through the async proxy
        asm volatile("fence.proxy.async.global;" ::: "memory");
        if (s + 1 < n_steps && !grid_barrier(v.bar, target += gridDim.x, v.flags, wait_limit_ns(v))) return leave();
    }
    // every CTA has passed a barrier, so every CTA has read bar[0]: publish the
    // count for the next launch
    if (blockIdx.x == 0 && tid == 0) v.bar[0] = target;
    leave();
}

template <int TU>
bool plan_tu(const F32View& v, LargePlan& c) {
    constexpr int P = LargeCfg<TU>::kP, PG = LargeCfg<TU>::kPG;
    const int H = v.n[1], n2 = v.n[2], kp1 = v.kp[1], kp2 = v.kp[2];
    // one block of each product per thread
    if (PG * ((H + 7) / 8) > kT || (kp1 + 11) / 12 * ((H + TU - 1) / TU) > kT || (n2 + 3) / 4 * (kp2 / 4) > kT) return false;
    c.xp = kp1 / 4 % 2 ? kp1 : kp1 + 4;
    c.hp = kp2 / 4 % 2 ? kp2 : kp2 + 4;
    c.dp = (n2 + 3) & ~3;
    int off = 0;
    auto take = [&](long long n) { const int o = off; off += (int)((n + 3) & ~3LL); return o; };
    c.w1 = take(v.woff[2]);
    c.w2 = take(v.P - v.woff[2]);
    c.x = take((long long)P * c.xp + 12);   // (the last column block of the last row may read past it)
    c.h = take((long long)P * c.hp + 8);
    c.d = take((long long)P * c.dp);
    c.t = take((long long)P * n2);
    c.red = take(4 * kT);
    c.total = off;
    return (size_t)off * sizeof(float) <= kF32SmemLimit;
}

}  // namespace

cudaError_t f32_large_setup() {
    for (const void* f : {(const void*)k_train_large<8>, (const void*)k_train_large<4>}) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32SmemLimit);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static int large_tu(const F32View& v, LargePlan& c) {
    if (v.L != 2) return 0;
    return plan_tu<4>(v, c) ? 4 : plan_tu<8>(v, c) ? 8 : 0;
}

bool f32_large_shape_ok(const F32View& v) {
    LargePlan c;
    return large_tu(v, c) != 0;
}

cudaError_t f32_train_large(const F32View& v, const float* X, const float* T, int n_patterns, int minibatch,
                            int n_steps, float* sse_out, bool fold_g, int num_sms, cudaStream_t s) {
    LargePlan c;
    const int tu = large_tu(v, c);
    if (tu == 0) return cudaErrorInvalidValue;
    F32View vv = v;
    int fold = fold_g ? 1 : 0;
    void* args[] = {(void*)&vv, (void*)&c, (void*)&X, (void*)&T, (void*)&n_patterns, (void*)&minibatch, (void*)&n_steps,
                    (void*)&sse_out, (void*)&fold};
    const void* fn = tu == 8 ? (const void*)k_train_large<8> : (const void*)k_train_large<4>;
    return cudaLaunchCooperativeKernel(fn, dim3(num_sms), dim3(kT), args, (size_t)c.total * sizeof(float), s);
}

}  // namespace bp
