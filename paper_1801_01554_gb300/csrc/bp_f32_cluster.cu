// float32 training of one-hidden-layer nets in small groups on one cluster.
//
// A group of a few patterns leaves no time for a grid barrier (1.3 us each way)
// and too little work for 152 SMs.  Here a cluster of up to 8 CTAs keeps the whole
// net on chip for the launch: CTA r owns U hidden units, that is U rows of
// [W_1 | b_1] and U columns of W_2.  S lanes share a unit's row, 4 kc4 columns
// each, whose weights and weight changes stay in registers as pairs (no pass over
// them touches shared memory, and a packed multiply-add does two); the W_2 columns
// stay in shared memory.  A group of at most PG patterns is one pass:
//   1. layer 1: every lane's products, a butterfly over its S lanes, logistic;
//   2. the CTA's share of the output sums, stored into every CTA of the cluster
//      (st.async to distributed shared memory, counted on the receiver's mbarrier);
//   3. outputs, error sums and output deltas, in every CTA alike;
//   4. hidden deltas of the CTA's own units and, lane by lane, the update of
//      W_2 and W_1.
// Three waits a pass, no global memory but the patterns, whose rows other warps
// copy three passes ahead.  All sums have a fixed order.  The pass is a chain of
// latencies (about 4,500 clocks for one pattern, 6,000 for four): shuffles, two
// logistics, shared memory, the exchange.
#include <cuda_runtime.h>

#include <algorithm>

#include "bp_f32_device.cuh"
#include "bp_internal.h"

namespace bp {
namespace {

constexpr int kCThreads = 512;   // most threads of a CTA
constexpr int kStagesX = 4;      // pattern rows in flight (passes)
constexpr int kLoaders = 3;      // warps that copy pattern rows
constexpr int kHelpers = 32 * (kLoaders + 1);   // and one for output biases and error sums

// Shared-memory offsets in floats, and the split of the net over the cluster.
struct ClusterPlan {
    int C, U, S, kc4;       // CTAs, units per CTA, lanes per unit, float4 columns per lane (4 or 7)
    int S2, p2;             // lanes per output; pitch of the W_2 rows
    int xp;                 // pitch of an input row, S * 4 * kc4
    int threads, uthr, outs, pg;   // threads; those of the units and of the output sums, whole warps
    int xb, tb, h, d1, d2, w2, v2, b2, vb2, part, e2, total;
};

// Sums of PG values over aligned groups of S lanes (PG <= S, powers of two):
// afterwards lane k of a group holds the sum of value k mod PG.
template <int PG>
__device__ __forceinline__ float lanes_sum(float (&acc)[PG], int S, int lane) {
    reduce_scatter<PG>(acc, lane);
    float r = acc[0];
#pragma unroll
    for (int o = PG; o < 32; o <<= 1)
        if (o < S) r += __shfl_xor_sync(0xffffffffu, r, o);
    return r;
}

// PG consecutive floats of shared memory (aligned to PG floats up to 4).
template <int PG>
__device__ __forceinline__ void ld_pg(float (&x)[PG], const float* p) {
    if constexpr (PG == 1) {
        x[0] = p[0];
    } else if constexpr (PG == 2) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        x[0] = t.x;
        x[1] = t.y;
    } else {
        const float4 t = ld4(p);
        x[0] = t.x;
        x[1] = t.y;
        x[2] = t.z;
        x[3] = t.w;
    }
}

// One weight's change g into its weight change v and the weight w.
template <bool GUARD>
__device__ __forceinline__ void momentum(float& w, float& v, float g, float lr, float mom, float guard, unsigned& n_bad) {
    if (GUARD) g = guard_count(guard, g, n_bad);
    v = lr * g + mom * v;
    w += v;
}

// KC4: float4 columns of a lane: s, s + S, ..., s + (KC4 - 1) S.
// GUARD: the fault guard is on (a separate instantiation: 1,000 unguarded updates of
// 203-120-26 by one pattern take 1,807 us; with the guard a branch, 1,939, and 1,983 once the
// branch tells weights from padding).
template <int PG, int KC4, bool GUARD>
__global__ void __launch_bounds__(kCThreads, 1)
    k_train_cluster(const __grid_constant__ F32View v, const __grid_constant__ ClusterPlan c, const float* X,
                    const float* T, int n_patterns, int minibatch, int n_steps, float* sse_out) {
    extern __shared__ __align__(128) float sm[];
    __shared__ __align__(8) uint64_t s_bar[2];   // bytes of the output sums, one barrier per buffer
    if (!bounds_ok((unsigned)c.total <= dyn_smem_floats() && minibatch <= PG, v.flags)) return;   // in every CTA alike
    const int tid = threadIdx.x, lane = tid & 31, nthr = blockDim.x;
    const int rank = (int)cluster_rank();
    const int n0 = v.n[0], H = v.n[1], n2 = v.n[2];
    const int S = c.S, S2 = c.S2, p2 = c.p2, xp = c.xp, C = c.C;
    const int u0 = rank * c.U, nu = max(0, min(c.U, H - u0));
    const int ul = tid / S, s = tid - ul * S;   // this lane's unit and its part of the row
    const bool unit = ul < nu;
    const int ko = tid / S2, t2 = tid - ko * S2;   // this lane's output
    const bool output = ko < n2;
    const bool loader = tid >= nthr - 32 * kLoaders, biaser = !loader && tid >= nthr - kHelpers;
    const int lw = (tid - (nthr - 32 * kLoaders)) >> 5;   // this loader warp
    const float lr = v.lr * v.grad_scale, mom = v.momentum, guard = v.guard;
    const bool table = v.sig_table != 0;
    unsigned n_bad = 0;
    const int latched = __ldcg(v.flags);   // nothing in this launch latches a timeout before the cluster's barrier
    sigmoid_table_init(v);

    unsigned pads = 0;   // this lane's columns past the bias
    if (GUARD)
        for (int i = 0; i < KC4; ++i) pads += (unsigned)min(max(4 * (s + S * i) + 3 - n0, 0), 4);

    // weights: W_1 rows to registers, W_2 columns and b_2 to shared memory
    const long long row1 = v.woff[1] + (long long)(u0 + ul) * v.kp[1];
    f32x2 w[2 * KC4], vel[2 * KC4];   // pairs of columns
#pragma unroll
    for (int j = 0; j < 2 * KC4; ++j) {
        const int col = 4 * (s + S * (j >> 1)) + 2 * (j & 1);
        const bool in0 = unit && col <= n0, in1 = unit && col + 1 <= n0;   // column n0: the bias
        w[j] = pack2(in0 ? v.theta[row1 + col] : 0.f, in1 ? v.theta[row1 + col + 1] : 0.f);
        vel[j] = pack2(in0 ? v.V[row1 + col] : 0.f, in1 ? v.V[row1 + col + 1] : 0.f);
    }
    for (int e = tid; e < n2 * nu; e += nthr) {
        const int k = e / nu, u = e - k * nu;
        const long long g = v.woff[2] + (long long)k * v.kp[2] + u0 + u;
        sm[c.w2 + k * p2 + u] = v.theta[g];
        sm[c.v2 + k * p2 + u] = v.V[g];
    }
    for (int k = tid; k < n2; k += nthr) {
        const long long g = v.woff[2] + (long long)k * v.kp[2] + H;
        sm[c.b2 + k] = v.theta[g];
        sm[c.vb2 + k] = v.V[g];
    }
    // the true unit's 1 and the zero pads of every input row
    for (int r = tid; r < kStagesX * PG; r += nthr)
        for (int i = n0; i < xp; ++i) sm[c.xb + r * xp + i] = i == n0 ? 1.f : 0.f;

    if (tid < 2) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(s_bar + tid)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // The loader warps copy the rows of one pass after another (every kLoaders-th
    // row each), one cp.async group a pass: patterns from lp on, at most PG, the
    // group of patterns ends at lend.
    const float *lx = X, *lt = T;
    int lp = 0, lend = min(minibatch, n_patterns), lstage = 0;
    auto load_next = [&]() {
        const int np = min(PG, lend - lp);   // 0 past the last pattern
        float* xb = sm + c.xb + lstage * PG * xp;
        for (int r = lw; r < PG; r += kLoaders) {
            if (r < np) {
                const float* src = lx + (size_t)r * n0;
#pragma unroll 8
                for (int i = lane; i < n0; i += 32) cp_async4(xb + r * xp + i, src + i);
            } else {
                for (int i = lane; i < n0; i += 32) xb[r * xp + i] = 0.f;
            }
        }
        float* tb = sm + c.tb + lstage * PG * n2;
        for (int e = lane + 32 * (kLoaders - 1 - lw); e < np * n2; e += 32 * kLoaders) cp_async4(tb + e, lt + e);
        cp_async_commit();
        lx += (size_t)np * n0;
        lt += np * n2;
        lp += np;
        if (lp == lend) lend = (int)min((long long)lend + minibatch, (long long)n_patterns);
        lstage = (lstage + 1) & (kStagesX - 1);
    };
    if (loader) {
        for (int k = 0; k < kStagesX - 1; ++k) load_next();
        cp_async_wait<kStagesX - 2>();
    }
    // a latched timeout: nothing is trained until bp_check has cleared it (every CTA returns)
    if (latched & kFlagTimeout) {
        cp_async_wait<0>();
        return;
    }
    cluster_barrier();   // every CTA of the cluster has started; its shared memory is set up

    if (tid == 0) {
        unsigned lost = 0;
#ifdef BP_CHECK
        lost = v.debug_stall != 0 ? 16u : 0u;   // test hook: the first exchange waits for bytes that never come
#endif
        arm(s_bar, C * n2 * PG * 4 + lost);
        arm(s_bar + 1, C * n2 * PG * 4);
    }
    int stage = 0, buf = 0;
    unsigned parity = 0;
    bool ok = true;
    const float* const w2o = sm + c.w2 + ko * p2;        // this lane's output row
    float* const w2u = sm + c.w2 + ul;                   // this lane's unit column
    const int v2off = c.v2 - c.w2;
    float* const hu = sm + c.h + ul * PG;
    for (int step = 0; step < n_steps && ok; ++step) {
        const int np = (int)min((long long)minibatch, (long long)n_patterns - (long long)step * minibatch);
        const float* xr = sm + c.xb + stage * PG * xp + 4 * s;
        // 1. layer 1
        if (tid < c.uthr) {
            f32x2 a2[PG][PG <= 2 ? 2 : 1];   // one or two chains of column pairs
#pragma unroll
            for (int p = 0; p < PG; ++p) a2[p][0] = a2[p][PG <= 2 ? 1 : 0] = 0;
#pragma unroll
            for (int i = 0; i < KC4; ++i) {
#pragma unroll
                for (int p = 0; p < PG; ++p) {
                    const ulonglong2 x = ld4x2(xr + p * xp + 4 * S * i);
                    a2[p][0] = fma2(w[2 * i], x.x, a2[p][0]);
                    a2[p][PG <= 2 ? 1 : 0] = fma2(w[2 * i + 1], x.y, a2[p][PG <= 2 ? 1 : 0]);
                }
            }
            float acc[PG];
#pragma unroll
            for (int p = 0; p < PG; ++p) {
                if (PG <= 2) a2[p][0] = add2(a2[p][0], a2[p][1]);
                const float2 t = unpack2(a2[p][0]);
                acc[p] = t.x + t.y;
            }
            const float net = lanes_sum<PG>(acc, S, lane);
            if (unit && s < PG) hu[s] = table ? sigmoid_tab(net) : sigmoid_f(net);
        }
        __syncthreads();
        // 2. this CTA's share of the output sums, to every CTA
        if (tid < c.outs) {
            float o[PG];
#pragma unroll
            for (int p = 0; p < PG; ++p) o[p] = 0.f;
            if (output) {
#pragma unroll 2
                for (int u = t2; u < nu; u += S2) {
                    const float wk = w2o[u];
                    float hv[PG];
                    ld_pg<PG>(hv, sm + c.h + u * PG);
#pragma unroll
                    for (int p = 0; p < PG; ++p) o[p] = fmaf(wk, hv[p], o[p]);
                }
            }
            const float r = lanes_sum<PG>(o, S2, lane);
            if (output) {
                // lanes t2 = p (mod PG) all hold pattern p's sum: they share the ranks
                float* dst = sm + c.part + (buf * C + rank) * n2 * PG + ko * PG + (t2 & (PG - 1));
                for (int q = t2 / PG; q < C; q += S2 / PG) st_remote(dst, s_bar + buf, q, r);
            }
        }
        // Bytes of buffer `buf` from all CTAs.  A peer writes this buffer again two
        // passes on, after it has this CTA's sums of the next pass, which are sent
        // after the reads below.
        ok = wait_bytes(s_bar + buf, parity, v.flags, wait_limit_ns(v));
        if (ok && tid == 0) arm(s_bar + buf, C * n2 * PG * 4);
        // 3. outputs and output deltas
        for (int e = tid; e < n2 * PG; e += nthr) {
            const int k = e / PG, p = e & (PG - 1);
            const float* pp = sm + c.part + buf * C * n2 * PG + e;
            float q[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) q[r] = r < C ? pp[r * n2 * PG] : 0.f;
            const float net = sm[c.b2 + k] + (((q[0] + q[1]) + (q[2] + q[3])) + ((q[4] + q[5]) + (q[6] + q[7])));
            const float o = table ? sigmoid_tab(net) : sigmoid_f(net);
            float err = 0.f;
            if (p < np) err = sm[c.tb + (stage * PG + p) * n2 + k] - o;
            sm[c.d2 + e] = err * o * (1.f - o);
            sm[c.e2 + e] = err * err;
        }
        if (loader) cp_async_wait<kStagesX - 3>();   // the next pass's rows
        ok = __syncthreads_and(ok) != 0;
        if (!ok) break;   // a peer's sums did not arrive
        // 4. hidden deltas and the changes of this lane's weights
        if (tid < c.uthr) {
            float hv[PG], a[PG];
#pragma unroll
            for (int p = 0; p < PG; ++p) a[p] = hv[p] = 0.f;
            if (unit) {
                ld_pg<PG>(hv, hu);
                float* we = w2u + s * p2;
#pragma unroll 2
                for (int k = s; k < n2; k += S, we += S * p2) {
                    float dk[PG];
                    ld_pg<PG>(dk, sm + c.d2 + k * PG);
                    float wk = *we;
                    float g = 0.f;
#pragma unroll
                    for (int p = 0; p < PG; ++p) {
                        a[p] = fmaf(wk, dk[p], a[p]);
                        g = fmaf(dk[p], hv[p], g);
                    }
                    float ve = we[v2off];
                    momentum<GUARD>(wk, ve, g, lr, mom, guard, n_bad);
                    we[v2off] = ve;
                    *we = wk;
                }
            }
            float d1[PG];
            {
                const float r = lanes_sum<PG>(a, S, lane);
                if constexpr (PG == 1) {
                    d1[0] = r * hv[0] * (1.f - hv[0]);
                } else {
                    float* du = sm + c.d1 + ul * PG;
                    if (unit && s < PG) {
                        const float hs = hu[s];
                        du[s] = r * hs * (1.f - hs);
                    }
                    __syncwarp();
                    ld_pg<PG>(d1, du);   // (dead units: not used)
                }
            }
            if (unit) {
                f32x2 g[2 * KC4];
#pragma unroll
                for (int j = 0; j < 2 * KC4; ++j) g[j] = 0;
#pragma unroll
                for (int i = 0; i < KC4; ++i) {
#pragma unroll
                    for (int p = 0; p < PG; ++p) {
                        const ulonglong2 x = ld4x2(xr + p * xp + 4 * S * i);
                        const f32x2 d = pack2(d1[p], d1[p]);
                        g[2 * i] = fma2(d, x.x, g[2 * i]);
                        g[2 * i + 1] = fma2(d, x.y, g[2 * i + 1]);
                    }
                }
                if (GUARD) {
#pragma unroll
                    for (int j = 0; j < 2 * KC4; ++j) {
                        const float2 t = unpack2(g[j]);
                        g[j] = pack2(guard_count(guard, t.x, n_bad), guard_count(guard, t.y, n_bad));
                    }
                    // Columns past the bias are no weights: their inputs are 0, but 0 times a NaN
                    // or an infinite delta is NaN, zeroed and counted above; not to be counted.
                    // (masking each column instead cost 10-20%)
                    float z = 0.f;
#pragma unroll
                    for (int p = 0; p < PG; ++p) z = fmaf(0.f, d1[p], z);
                    if (z != 0.f) n_bad -= pads;
                }
                const f32x2 lr2 = pack2(lr, lr), mom2 = pack2(mom, mom);
#pragma unroll
                for (int j = 0; j < 2 * KC4; ++j) {
                    vel[j] = fma2(mom2, vel[j], mul2(lr2, g[j]));
                    w[j] = add2(w[j], vel[j]);
                }
            }
        } else if (loader) {
            load_next();   // three passes ahead, into the rows that the last pass is done with
        } else if (biaser) {
            // output biases (every CTA keeps the same copy) and the group's error sum
            for (int k = lane; k < n2; k += 32) {
                float g = 0.f;
#pragma unroll
                for (int p = 0; p < PG; ++p) g += sm[c.d2 + k * PG + p];
                unsigned bad = 0;
                float ve = sm[c.vb2 + k], wk = sm[c.b2 + k];
                momentum<GUARD>(wk, ve, g, lr, mom, guard, bad);
                if (rank == 0) n_bad += bad;
                sm[c.vb2 + k] = ve;
                sm[c.b2 + k] = wk;
            }
            if (rank == 0) {
                float e = 0.f;
                for (int k = lane; k < n2 * PG; k += 32) e += sm[c.e2 + k];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
                if (lane == 0) {
                    if (sse_out != nullptr) sse_out[step] = e;
                    if (!isfinite(e)) atomicOr(v.flags, kFlagNonfinite);
                }
            }
        }
        stage = (stage + 1) & (kStagesX - 1);
        buf ^= 1;
        parity ^= buf == 0 ? 1u : 0u;
    }
    cp_async_wait<0>();
    // No CTA sends anything after this barrier, so that a CTA whose sums all came may leave; one
    // whose wait ran out gives the missing ones as long again to land in its shared memory.
    cluster_barrier();
    if (!ok) wait_bytes(s_bar + buf, parity, v.flags, wait_limit_ns(v));
    // A wait that ran out in one CTA leaves the others an update ahead: then none writes
    // back, and the weights are those before the launch.
    if (__ldcg(v.flags) & kFlagTimeout) return;
    if (n_bad != 0) atomicAdd(v.faults, n_bad);
    // weights and weight changes back to global memory
#pragma unroll
    for (int j = 0; j < 2 * KC4; ++j) {
        const int col = 4 * (s + S * (j >> 1)) + 2 * (j & 1);
        const float2 wj = unpack2(w[j]), vj = unpack2(vel[j]);
        if (unit && col <= n0) {
            v.theta[row1 + col] = wj.x;
            v.V[row1 + col] = vj.x;
        }
        if (unit && col + 1 <= n0) {
            v.theta[row1 + col + 1] = wj.y;
            v.V[row1 + col + 1] = vj.y;
        }
    }
    for (int e = tid; e < n2 * nu; e += nthr) {
        const int k = e / nu, u = e - k * nu;
        const long long g = v.woff[2] + (long long)k * v.kp[2] + u0 + u;
        v.theta[g] = sm[c.w2 + k * p2 + u];
        v.V[g] = sm[c.v2 + k * p2 + u];
    }
    if (rank == 0)
        for (int k = tid; k < n2; k += nthr) {
            const long long g = v.woff[2] + (long long)k * v.kp[2] + H;
            v.theta[g] = sm[c.b2 + k];
            v.V[g] = sm[c.vb2 + k];
        }
}

// Largest group.  us per update of 203-120-26, one-CTA kernel -> this one: 6.76 -> 2.2
// (1 pattern), 7.4 -> 2.4 (2), 9.4 -> 2.9 (4); 203-300-26, on the grid-wide kernel: 18.4
// -> 2.7 (1).  Groups of 5 to 16 would gain too (8: 9.8 -> 3.6), but sum in another
// order than the grid-wide kernel, and at that size a few hundred updates of a net that
// memorises its patterns amplify the last bit of a sum a hundred thousand times.
constexpr int kClusterMaxB = 4;

// Splits the net: as many CTAs as leave each four units (8 CTAs against 4 at 203-120-26:
// 2.22 / 2.36 us with 1 pattern), and the fewest lanes per unit whose 4 float4 columns
// each cover a row (7 columns halve the lanes and cost 5-20% more; they are for nets of
// so many units that 4 do not fit 512 threads).
bool make_plan(const F32View& v, int minibatch, ClusterPlan& c) {
    if (v.L != 2 || minibatch > kClusterMaxB) return false;
    const int cols4 = (v.n[0] + 1 + 3) / 4, H = v.n[1], n2 = v.n[2];
    if (H > 8 * kCThreads || n2 > 128) return false;
    c.pg = minibatch >= 3 ? 4 : minibatch;
    c.C = H >= 32 ? 8 : H >= 16 ? 4 : H >= 8 ? 2 : 1;
    c.U = (H + c.C - 1) / c.C;
    for (int kc4 : {4, 7}) {
        c.kc4 = kc4;
        c.S = c.pg;
        while (c.S < 32 && c.S * kc4 < cols4) c.S *= 2;
        c.uthr = (c.U * c.S + 31) / 32 * 32;
        c.threads = c.uthr + kHelpers;
        if (c.S * kc4 < cols4 || c.threads > kCThreads) continue;
        c.S2 = 32;
        while (c.S2 > 1 && n2 * c.S2 > c.threads) c.S2 /= 2;
        if (c.S2 < c.pg) continue;
        c.outs = (n2 * c.S2 + 31) / 32 * 32;
        c.p2 = (c.U + 27) / 32 * 32 + 4;
        c.xp = c.S * 4 * c.kc4;
        int off = 0;
        auto take = [&](int n) { const int o = off; off += (n + 3) & ~3; return o; };
        c.xb = take(kStagesX * c.pg * c.xp);
        c.tb = take(kStagesX * c.pg * n2);
        c.h = take(c.U * c.pg);
        c.d1 = take((c.U + 32) * c.pg);   // lanes past the last unit read, but do not use, a row
        c.d2 = take(n2 * c.pg);
        c.w2 = take(n2 * c.p2);
        c.v2 = take(n2 * c.p2);
        c.b2 = take(n2);
        c.vb2 = take(n2);
        c.part = take(2 * c.C * n2 * c.pg);
        c.e2 = take(n2 * c.pg);
        c.total = off;
        if ((size_t)off * sizeof(float) <= kF32SmemLimit) return true;
    }
    return false;
}

template <int PG, int KC4, bool GUARD>
cudaError_t launch(const F32View& v, const ClusterPlan& c, const float* X, const float* T, int n_patterns,
                   int minibatch, int n_steps, float* sse_out, cudaStream_t s) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c.C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(c.C);
    cfg.blockDim = dim3(c.threads);
    cfg.dynamicSmemBytes = (size_t)c.total * sizeof(float);
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_train_cluster<PG, KC4, GUARD>, v, c, X, T, n_patterns, minibatch, n_steps, sse_out);
}

template <int KC4, bool GUARD>
cudaError_t launch_kc(const F32View& v, const ClusterPlan& c, const float* X, const float* T, int n_patterns,
                      int minibatch, int n_steps, float* sse_out, cudaStream_t s) {
#define BP_ARGS v, c, X, T, n_patterns, minibatch, n_steps, sse_out, s
    switch (c.pg) {
        case 1: return launch<1, KC4, GUARD>(BP_ARGS);
        case 2: return launch<2, KC4, GUARD>(BP_ARGS);
        default: return launch<4, KC4, GUARD>(BP_ARGS);
    }
#undef BP_ARGS
}

template <int KC4>
cudaError_t setup_kc() {
    const void* fns[] = {(const void*)k_train_cluster<1, KC4, false>, (const void*)k_train_cluster<2, KC4, false>,
                         (const void*)k_train_cluster<4, KC4, false>, (const void*)k_train_cluster<1, KC4, true>,
                         (const void*)k_train_cluster<2, KC4, true>, (const void*)k_train_cluster<4, KC4, true>};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kF32SmemLimit);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t f32_cluster_setup() {
    const cudaError_t e = setup_kc<4>();
    return e != cudaSuccess ? e : setup_kc<7>();
}

bool f32_cluster_ok(const F32View& v, int minibatch) {
    ClusterPlan c;
    return make_plan(v, minibatch, c);
}

cudaError_t f32_train_cluster(const F32View& v, const float* X, const float* T, int n_patterns, int minibatch,
                              int n_steps, float* sse_out, cudaStream_t s) {
    ClusterPlan c;
    if (!make_plan(v, minibatch, c)) return cudaErrorInvalidValue;
    const auto f = v.guard > 0.f ? (c.kc4 == 4 ? launch_kc<4, true> : launch_kc<7, true>)
                                 : (c.kc4 == 4 ? launch_kc<4, false> : launch_kc<7, false>);
    return f(v, c, X, T, n_patterns, minibatch, n_steps, sse_out, s);
}

}  // namespace bp
