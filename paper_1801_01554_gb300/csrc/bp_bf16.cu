// bfloat16 back-propagation step on the sm_103a tensor cores.
//
// Every contraction of the step is a GEMM C[M,N] = A[M,K] * B[N,K]^T fed by TMA
// (128-byte swizzle) into a multi-stage shared-memory ring, multiplied by
// tcgen05.mma (kind::f16, bf16 in, fp32 accumulate) into a double-buffered TMEM
// accumulator, and finished by an epilogue that reads TMEM with tcgen05.ld:
//
//   forward  (Section 3)      A_l  = sigma(A_{l-1} W_l^T + b_l)
//                               epilogue: bias, logistic, bf16 stores of A_l
//   output   (Sections 3, 8)  o = sigma(...); delta_L = (t - o) o (1 - o);
//                               error sum; bias-gradient column sums
//   hidden delta (Section 3)  delta_{l-1} = (delta_l W_l) * a (1 - a), for
//                               l = L..2 only: no delta for the input units
//                               (Section 6.1)
//   pooled change (Sec. 4.1)  G_l = delta_l^T A_{l-1}, K = the batch, summed
//                               in fp32 chains of bounded length and, where tiles
//                               are few, split over CTAs into partial sums; the
//                               layers share one launch
//
// Activations, deltas and weights are stored once, row-major.  An operand whose
// rows run along K is staged as it lies; one whose rows run along M or N (W_l in
// the hidden delta, delta_l and A_{l-1} in the pooled change) is staged as 64 x
// 64 blocks and handed to the tensor cores as an MN-major operand, so that no
// transposed copy is ever written.  The update applies the momentum rule of Section
// 6.2.1 to the fp32 master weights and rewrites the bf16 weight copy: in the epilogue
// of the pooled change where K is not split, else in a kernel that also sums the
// partial changes.  The kernels of a step are launched with
// programmatic stream serialisation: each sets up its barriers and TMEM while
// its predecessor drains, and waits (griddepcontrol.wait) before it touches
// global memory.  All device-side waits are bounded and latch kFlagTimeout.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

#include "bp_bf16.h"
#include "bp_internal.h"

namespace bp {
namespace {

using bf16 = __nv_bfloat16;

constexpr int BM = 128;   // rows of a tile (TMEM lanes)
constexpr int BK = 64;    // K per stage: 64 bf16 = one 128-byte swizzle row
constexpr int UMMA_K = 16;
constexpr int kEpiWarps = 8;         // two per TMEM lane quarter, each on half of the columns
constexpr int kEpiThreads = 32 * kEpiWarps;
constexpr int kGemmThreads = 64 + kEpiThreads;   // warp 0 TMA, warp 1 MMA, warps 2.. epilogue

constexpr unsigned long long kWaitNs = 2000000000ull;
constexpr unsigned kWaitIters = 1u << 28;

enum Mode : int { MODE_FWD = 0, MODE_FWD_OUT = 1, MODE_DX = 2, MODE_DW = 3, MODE_DWU = 4 };

struct GemmArgs {
    int M, N, K;
    int num_m, num_n;       // tiles along M and N
    int kb_total;           // K blocks
    const float* bias;      // [N]                          FWD, FWD_OUT
    bf16* out;              // [M, ldo] row-major            FWD: A_l; FWD_OUT: A_L; DX: delta
    int ldo;
    bf16* out2;             // [M, ld2] row-major            FWD_OUT: delta_L (with T), else a second copy of A_L
    int ld2;
    const bf16* aux;        // FWD_OUT: T [M, ld_aux]; DX: A_{l-1} [M, ld_aux]
    int ld_aux;
    float* bias_part;       // [num_m, N]                    FWD_OUT (with T), DX
    float* sse_part;        // [num_m * num_n]               FWD_OUT (with T)
    int* flags;
};

// The pooled-change GEMMs of all layers, one launch: layer l's tiles are
// [tile0[l], tile0[l + 1]), times `splits` runs of kb_per_split K blocks.  A run is
// accumulated in TMEM `chain` K blocks at a time; the epilogue adds these sums.
struct DwLayer {
    int M, N;               // n_l, n_{l-1}
    int num_m, num_n;
    int tile0;              // first tile of the layer
    int chain;              // K blocks of one sum in TMEM (sum_chain)
    float* gpart;           // [splits, M, N]
};
struct DwArgs {
    int L, tiles, splits, kb_per_split, kb_total;
    DwLayer ly[kMaxL];
    int* flags;
};
struct DwMaps {
    CUtensorMap a[kMaxL], b[kMaxL];   // delta_l, A_{l-1}
};

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Whether the phase is complete, without waiting.
__device__ __forceinline__ bool mbar_test(uint64_t* bar, unsigned parity) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0;
}
// Bounded wait.  Returns false if it ran out or another role aborted.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, unsigned parity, volatile int* abort_flag,
                                          int* flags) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned it = 1; it < kWaitIters; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 0) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > kWaitNs) break;
        }
    }
    *abort_flag = 1;
    atomicOr(flags, kFlagTimeout);
    return false;
}

__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, int c0, int c1,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes "
        "[%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(smem_dst)),
        "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

// True in one lane of the (converged) warp.  Unlike a test of the lane number it tells
// the compiler that a single thread follows, so that the operands of the TMA and MMA
// instructions can stay in uniform registers.
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}

// Programmatic dependent launch: wait for the kernels this one depends on (their
// writes are then visible), and let the next kernel of the stream start its setup.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle (tcgen05 descriptor version 1).
//   K-major:  the operand's rows are 128 bytes (64 of K); 8-row groups 1024 bytes
//             apart (stride offset); the leading offset is unused.
//   MN-major: blocks of 64 K rows x 64 of M or N (128 bytes); 8 K rows are 1024
//             bytes apart (stride offset), the next 64 of M or N one block, 8 KB
//             (leading offset).
// The upper word is constant; the lower one holds the address (in 16-byte units, below
// 2^14) and the leading offset, so that stages and K steps are plain additions to it.
constexpr uint32_t kMnBlockBytes = BK * 64 * 2;
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);   // stride offset, version 1, 128-byte swizzle
template <bool MN>
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) {
    return (addr >> 4) | (((MN ? kMnBlockBytes : 16u) >> 4) << 16);
}
// From one K step of UMMA_K to the next inside a stage, in 16-byte units.
template <bool MN>
__device__ __forceinline__ constexpr uint32_t k_step_units() { return (MN ? UMMA_K * 128 : UMMA_K * 2) >> 4; }

// Instruction descriptor of tcgen05.mma kind::f16: bf16 A and B, fp32 D, M x N
// tile, each operand K-major or MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn, bool b_mn) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// One tcgen05.mma: operands by the lower words of their descriptors; the first one of
// a tile overwrites the accumulator.
template <uint32_t IDESC>
__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint32_t a_lo, uint32_t b_lo, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(tmem_d),
        "r"(a_lo), "r"(b_lo), "n"(kDescHi), "n"(IDESC), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// 32 lanes x 32 consecutive fp32 columns from TMEM.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Logistic for bf16 outputs: hardware exp2 and reciprocal (1 ulp each; an IEEE divide
// here cost a quarter of a training step in the epilogues).  For 1 + e^-x beyond the
// largest float the quotient is 0, the logistic's value there.
__device__ __forceinline__ float sigmoid_fast(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + __expf(-x)));
    return r;
}

__device__ __forceinline__ float bf16_round(float x) {
    return __bfloat162float(__float2bfloat16_rn(x));
}

__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, %0;" ::"n"(kEpiThreads) : "memory"); }

// The same barrier; true in every epilogue thread if x is true in any.
__device__ __forceinline__ bool epi_any(bool x) {
    unsigned r;
    __syncwarp();
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 q, %1, 0;\n\t"
        "bar.red.or.pred p, 1, %2, q;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r)
        : "r"(x ? 1u : 0u), "n"(kEpiThreads)
        : "memory");
    return r != 0;
}

// ------------------------------------------------------------ epilogue
// A warp's 32 x 32 block of bf16 as 16-byte pieces (8 columns).  Global memory is read
// and written with lane (row 8 j + lane / 4, piece lane % 4), four lanes to a 64-byte
// row segment; the arithmetic wants lane = row.  The warp's 2 KB of shared memory turns
// one into the other (pieces permuted by row so that both sides spread over the banks).
// Loading a row per lane instead costs 32 cache-line lookups an instruction (the output
// layer's epilogue took 17,200 clocks a 128 x 256 tile, 14,600 with whole segments; a
// 1024-2048-2048-512 step of 1,001 patterns 81.8 us, 79.8), but no turn through shared
// memory: it is kept for 64-column tiles, one chunk per warp, where the latency of that
// counts for more (208-1024-32 at 512 patterns: 20.6 us against 20.9).
struct Row32 {
    uint4 u[4];
};
__device__ __forceinline__ uint4* piece_at(uint4* sS4, int row, int piece) {
    return sS4 + row * 4 + (piece ^ ((row >> 1) & 3));
}
// rows past `rows` and pieces past `pieces` are zero
__device__ __forceinline__ void load_block(Row32& r, const bf16* p, int ld, int rows, int pieces) {
    const int lane = threadIdx.x & 31, piece = lane & 3;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int row = 8 * j + (lane >> 2);
        r.u[j] = (row < rows && piece < pieces) ? *reinterpret_cast<const uint4*>(p + (size_t)row * ld + piece * 8)
                                                : make_uint4(0u, 0u, 0u, 0u);
    }
}
__device__ __forceinline__ void load_own_row(Row32& r, const bf16* p, int ld, int rows, int pieces) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        r.u[k] = (lane < rows && k < pieces) ? reinterpret_cast<const uint4*>(p + (size_t)lane * ld)[k]
                                             : make_uint4(0u, 0u, 0u, 0u);
}
__device__ __forceinline__ void block_to_rows(Row32& r, uint4* sS4) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < 4; ++j) *piece_at(sS4, 8 * j + (lane >> 2), lane & 3) = r.u[j];
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) r.u[k] = *piece_at(sS4, lane, k);
    __syncwarp();   // the block is rewritten
}
__device__ __forceinline__ float row_value(const Row32& r, int c) {   // c is a compile-time constant
    const uint4& u = r.u[c >> 3];
    const uint32_t w = ((c >> 1) & 3) == 0 ? u.x : ((c >> 1) & 3) == 1 ? u.y : ((c >> 1) & 3) == 2 ? u.z : u.w;
    return __uint_as_float((c & 1) ? (w & 0xffff0000u) : (w << 16));
}

// One 32-column chunk of a pooled-change tile: this lane's row m of the partial sums.
__device__ __forceinline__ void store_partial(float* gpart, int M, int N, int m, int n0, int split, const float (&v)[32]) {
    if (m >= M) return;
    float* dst = gpart + ((size_t)split * M + m) * N + n0;   // N is a multiple of 8
#pragma unroll
    for (int c = 0; c < 32; c += 4)
        if (n0 + c < N) *reinterpret_cast<float4*>(dst + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
}

// 32 lanes x 16 consecutive fp32 columns from TMEM.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// And back.
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float (&v)[16]) {
    uint32_t r[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]),
        "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]),
        "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// One 32-column chunk of the tile for the 32 rows of one epilogue warp (this
// lane's row m).  Values are rounded to bf16 and staged by rows in the warp's
// 2 KB shared-memory block (16-byte pieces permuted by row so that the lanes'
// writes hit distinct banks); the warp then writes every 64-byte row segment
// with four lanes' 16-byte stores, eight segments per instruction.  The column
// sums of a delta block (bias change) are taken from the pieces on their way
// out: each lane adds its four rows of 8 columns, then the eight lanes of a
// piece reduce-scatter them (7 shuffles).
template <int BN, int MODE>
__device__ __forceinline__ void epilogue_chunk(const GemmArgs& g, int m0, int n0, float (&v)[32], float& sse,
                                               bool row_ok, bf16* sS, const float* sbias, Row32& aux,
                                               float* colsum_slot) {
    const int N = g.N;
    const int lane = threadIdx.x & 31;
    const int valid = min(32, N - n0);
    const bool with_t = (MODE == MODE_FWD_OUT) && (g.aux != nullptr);
    uint4* sS4 = reinterpret_cast<uint4*>(sS);
    if (BN > 64 && (with_t || MODE == MODE_DX)) block_to_rows(aux, sS4);
    // values in place; they are rounded when they are packed below
    if (MODE == MODE_FWD || MODE == MODE_FWD_OUT) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {   // the tile's biases, staged in shared memory (0 past N)
            const float4 f = reinterpret_cast<const float4*>(sbias)[k];
            v[4 * k] = sigmoid_fast(v[4 * k] + f.x);
            v[4 * k + 1] = sigmoid_fast(v[4 * k + 1] + f.y);
            v[4 * k + 2] = sigmoid_fast(v[4 * k + 2] + f.z);
            v[4 * k + 3] = sigmoid_fast(v[4 * k + 3] + f.w);
        }
        if (with_t) {
#pragma unroll
            for (int c = 0; c < 32; ++c) {
                const float o = bf16_round(v[c]);
                const float err = (row_ok && c < valid) ? row_value(aux, c) - o : 0.f;
                sse = fmaf(err, err, sse);
                v[c] = err * o * (1.f - o);
            }
        }
    } else {   // MODE_DX: delta_{l-1} = (delta_l W_l) a (1 - a); rows and columns past the edges have a = 0
#pragma unroll
        for (int c = 0; c < 32; ++c) {
            const float a = row_value(aux, c);
            v[c] = v[c] * a * (1.f - a);
        }
    }
    // rows: A_l, A_L (and the caller's copy) or delta_L (training output layer), or delta_{l-1}
    bf16* const rows = with_t ? g.out2 : g.out;
    const int ldr = with_t ? g.ld2 : g.ldo;
    bf16* const copy = (MODE == MODE_FWD_OUT && !with_t) ? g.out2 : nullptr;
    const int piece = lane & 3;   // 16-byte piece of a 64-byte segment
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        __align__(16) __nv_bfloat162 h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) h[q] = __floats2bfloat162_rn(v[8 * k + 2 * q], v[8 * k + 2 * q + 1]);
        *piece_at(sS4, lane, k) = *reinterpret_cast<const uint4*>(h);
    }
    __syncwarp();
    const int pieces = valid >> 3;   // N is a multiple of 8
    float cs[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) cs[q] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = j * 8 + (lane >> 2);
        const uint4 u = *piece_at(sS4, r, piece);
        if (m0 + r < g.M && piece < pieces) {
            *reinterpret_cast<uint4*>(rows + (size_t)(m0 + r) * ldr + n0 + piece * 8) = u;
            if (copy != nullptr) *reinterpret_cast<uint4*>(copy + (size_t)(m0 + r) * g.ld2 + n0 + piece * 8) = u;
        }
        if (colsum_slot != nullptr) {   // rows past the batch and columns past N hold zeros
            const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float2 f = __bfloat1622float2(h[q]);
                cs[2 * q] += f.x;
                cs[2 * q + 1] += f.y;
            }
        }
    }
    if (colsum_slot != nullptr) {
#pragma unroll
        for (int half = 4; half >= 1; half >>= 1) {
            const bool up = (lane & (4 * half)) != 0;
#pragma unroll
            for (int k = 0; k < half; ++k) {
                const float send = up ? cs[k] : cs[k + half];
                const float keep = up ? cs[k + half] : cs[k];
                cs[k] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * half);
            }
        }
        colsum_slot[piece * 8 + (lane >> 2)] = cs[0];
    }
    __syncwarp();   // the staging block may be rewritten
}

// ------------------------------------------------------------ update arguments
constexpr int kUpdThreads = 256;
constexpr int kUpdPieces = 2;                                    // float4 pieces per thread of a weight block
constexpr int kUpdFloats = kUpdThreads * kUpdPieces * 4;         // weights per block
constexpr int kUpdBiases = 32, kUpdSlices = kUpdThreads / kUpdBiases;   // biases per block, threads per bias

struct LayerUpd {
    long long nw;               // n_out * n_in, a multiple of 64
    int n_out;
    long long woff, boff;       // offsets in theta / V / G
    const float* gpart;         // [splits, n_out, n_in]
    const float* bias_part;     // [mtiles, n_out]
    bf16* wb;                   // [n_out, n_in]
    int block0, bias0;          // first weight block of the layer; first bias block (counted apart)
};
struct UpdArgs {
    int L;
    LayerUpd ly[kMaxL];
    int blocks, bias_blocks;    // weight blocks and bias blocks of all layers
    int splits, mtiles;         // pending partial changes (0: none)
    float* theta;
    float* V;
    float* G;
    float lr_gs, momentum;
    int mode;                   // 0: apply update; 1: accumulate into G; 2: refresh the bf16 copy
    int fold_g;
    const float* sse_part;
    int n_sse;
    float* sse_out;
    int* flags;
    float guard;          // > 0: fault guard of Section 8
    unsigned* faults;     // changes the guard zeroed
};

// Fault guard of Section 8: a total weight change outside (-guard, guard), or
// not a number, is set to zero and counted (off while guard <= 0).
__device__ __forceinline__ float guard_change(const UpdArgs& a, float g) {
    if (a.guard > 0.f && !(fabsf(g) <= a.guard)) {
        atomicAdd(a.faults, 1u);
        return 0.f;
    }
    return g;
}
__device__ __forceinline__ float4 add4(float4 x, float4 y) { return make_float4(x.x + y.x, x.y + y.y, x.z + y.z, x.w + y.w); }

// One bias or error-sum block of an update, by 256 threads (t = 0 .. 255) with
// 1 KB of shared memory; `sync` is their barrier.  Block b: bias blocks
// [0, a.bias_blocks) layer by layer, then, if the group's error sum is wanted, one more.
// (the slices of a sum, then the slices in order: the same order on every run)
// The bias blocks' and the error sum's reduction: slice k of `rows` partials,
// then the slices in order (the same order on every run).
__device__ __forceinline__ float slice_sum(const float* p, int rows, size_t pitch, int k, int slices) {
    const int per = (rows + slices - 1) / slices;
    const int lo = k * per, hi = min(rows, lo + per);
    float s = 0.f;
#pragma unroll 8
    for (int r = lo; r < hi; ++r) s += p[(size_t)r * pitch];
    return s;
}

template <class Sync>
__device__ __forceinline__ void update_bias_block(const UpdArgs& a, int b, int t, float* red, Sync sync) {
    if (b == a.bias_blocks) {   // the group's error sum
        float s = slice_sum(a.sse_part, a.n_sse, 1, t, kUpdThreads);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 31) == 0) red[t >> 5] = s;
        sync();
        if (t == 0) {
            s = 0.f;
            for (int w = 0; w < kUpdThreads / 32; ++w) s += red[w];
            *a.sse_out = s;
            if (!isfinite(s)) atomicOr(a.flags, kFlagNonfinite);
        }
        sync();
        return;
    }
    int l = 0;
    while (l + 1 < a.L && b >= a.ly[l + 1].bias0) ++l;
    const LayerUpd& u = a.ly[l];
    // kUpdSlices threads share each bias's row-block partials
    const int i = t & (kUpdBiases - 1), k = t / kUpdBiases;
    const int j = (b - u.bias0) * kUpdBiases + i;
    red[k * kUpdBiases + i] = j < u.n_out ? slice_sum(u.bias_part + j, a.mtiles, u.n_out, k, kUpdSlices) : 0.f;
    sync();
    if (t < kUpdBiases && j < u.n_out) {
        float g = 0.f;
#pragma unroll
        for (int q = 0; q < kUpdSlices; ++q) g += red[q * kUpdBiases + t];
        const long long idx = u.boff + j;
        if (a.mode == 1) {
            a.G[idx] += g;
        } else if (a.mode == 0) {
            if (a.fold_g) {
                g += a.G[idx];
                a.G[idx] = 0.f;
            }
            const float vel = a.lr_gs * guard_change(a, g) + a.momentum * a.V[idx];
            a.V[idx] = vel;
            a.theta[idx] += vel;
        }
    }
    sync();
}

// ------------------------------------------------------------ GEMM kernel
// Tile order: groups of GROUP row blocks, each group swept over all column blocks (row
// block fastest), so that the tiles in flight on the 152 SMs share a few row blocks of A
// and column blocks of B, which stay in L2, instead of reading every row block of A at
// once (that was 10% slower for 4096^5).  16 row blocks in the backward: 152 tiles of
// 128 x 256 are then about a square, 16 x 10, and read least (with 4, 12 x 16 tiles, the
// pooled changes of 4096^5 read 4.0 GB from DRAM for 1.6 GB of operands and weights).  ms
// per step of 4096^5, 4 / 8 / 12 / 16 / 32 in the pooled changes: 3.93 / 3.93 / 3.91 /
// 3.90 / 3.90.  The forward keeps 4: 16 gains it nothing at that size, and costs 0.9% where
// all tiles run at once (1,001 of 1024-2048-2048-512).  A choice at run time costs the
// small launches 1-3%.
template <int GROUP>
__device__ __forceinline__ void tile_coords(int tile, int num_m, int num_n, int& mb, int& nb) {
    const int per_group = GROUP * num_n;
    const int grp = tile / per_group;
    const int first = grp * GROUP;
    const int gm = min(num_m - first, GROUP);
    const int local = tile - grp * per_group;
    mb = first + local % gm;
    nb = local / gm;
}

template <int BN>
struct GemmCfg {
    static constexpr int kStages = BN == 256 ? 4 : BN == 128 ? 6 : 8;
    static constexpr int kABytes = BM * BK * 2;
    static constexpr int kBBytes = BN * BK * 2;
    static constexpr int kStageBytes = kABytes + kBBytes;
    // tile ring, then barriers and scratch
    static constexpr int kRingBytes = kStages * kStageBytes;
    static constexpr int kColsumBytes = 4 * BN * 4;
    static constexpr int kStageOutBytes = kEpiWarps * 32 * 32 * 2;   // one 32 x 32 bf16 block per epilogue warp
    static constexpr int kBiasBytes = 2 * BN * 4;   // the tile's biases, one block per accumulator
    static constexpr int kSmemBytes =
        1024 + kRingBytes + kColsumBytes + kStageOutBytes + kBiasBytes + 512;
};

__device__ __forceinline__ void prefetch_map(const CUtensorMap* m) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)m) : "memory");
}

// A work item of a GEMM launch: a tile and its run of K blocks.
struct Item {
    int mb, nb, kb0, kb1;
    int chain;               // K blocks per sum in TMEM
    int l, split;            // pooled change only
};
// Work of the forward and hidden-delta launches: one problem, whole K.
template <int MODE>
struct OneGemm {
    static constexpr int kMode = MODE;
    static constexpr bool kAMn = false, kBMn = MODE == MODE_DX;
    const GemmArgs& g;
    const CUtensorMap *ma, *mb_;
    __device__ int items() const { return g.num_m * g.num_n; }
    __device__ Item item(int it) const {
        Item w{0, 0, 0, g.kb_total, g.kb_total, 0, 0};
        tile_coords<MODE == MODE_DX ? 16 : 4>(it, g.num_m, g.num_n, w.mb, w.nb);
        return w;
    }
    // The launch's parameters are read here once, while the previous kernel drains: their
    // first read misses the constant cache.
    __device__ void touch() const {
        asm volatile("" ::"r"(g.N), "r"(g.kb_total), "l"(g.bias), "l"(g.out), "r"(g.ldo), "l"(g.out2), "r"(g.ld2),
                     "l"(g.aux), "r"(g.ld_aux), "l"(g.bias_part), "l"(g.sse_part), "l"(g.flags));
    }
    __device__ void prefetch_maps() const {
        prefetch_map(ma);
        prefetch_map(mb_);
    }
    __device__ const CUtensorMap* map_a(const Item&) const { return ma; }
    __device__ const CUtensorMap* map_b(const Item&) const { return mb_; }
};
// Work of the pooled-change launch: every layer's tiles, `splits` times over.
struct DwGemm {
    static constexpr int kMode = MODE_DW;
    static constexpr bool kAMn = true, kBMn = true;
    const DwArgs& g;
    const DwMaps& maps;
    __device__ int items() const { return g.tiles * g.splits; }
    __device__ Item item(int it) const {
        Item w;
        w.split = it / g.tiles;
        const int tile = it - w.split * g.tiles;
        w.l = 0;
        while (w.l + 1 < g.L && tile >= g.ly[w.l + 1].tile0) ++w.l;
        const DwLayer& y = g.ly[w.l];
        tile_coords<16>(tile - y.tile0, y.num_m, y.num_n, w.mb, w.nb);
        w.kb0 = w.split * g.kb_per_split;
        w.kb1 = min(g.kb_total, w.kb0 + g.kb_per_split);
        w.chain = y.chain;
        return w;
    }
    __device__ void touch() const {
        asm volatile("" ::"r"(g.splits), "r"(g.kb_per_split), "r"(g.kb_total), "l"(g.flags));
        for (int l = 0; l < g.L; ++l) asm volatile("" ::"r"(g.ly[l].N), "r"(g.ly[l].chain), "l"(g.ly[l].gpart));
    }
    __device__ void prefetch_maps() const {
        for (int l = 0; l < g.L; ++l) {
            prefetch_map(&maps.a[l]);
            prefetch_map(&maps.b[l]);
        }
    }
    __device__ const CUtensorMap* map_a(const Item& w) const { return &maps.a[w.l]; }
    __device__ const CUtensorMap* map_b(const Item& w) const { return &maps.b[w.l]; }
};

// The same with the update in the epilogue (one K split).
struct DwuGemm : DwGemm {
    static constexpr int kMode = MODE_DWU;
    const UpdArgs& u;
    __device__ DwuGemm(const DwArgs& g_, const DwMaps& m_, const UpdArgs& u_) : DwGemm{g_, m_}, u(u_) {}
    __device__ void touch() const {
        DwGemm::touch();
        asm volatile("" ::"r"(u.bias_blocks), "l"(u.theta), "l"(u.V), "f"(u.lr_gs), "r"(u.fold_g), "f"(u.guard));
        for (int l = 0; l < g.L; ++l) asm volatile("" ::"l"(u.ly[l].woff), "l"(u.ly[l].wb), "l"(u.ly[l].bias_part));
    }
};

// Copies one operand's stage: ROWS of M or N by BK of K from K block kb.
template <int ROWS, bool MN>
__device__ __forceinline__ void load_operand(uint8_t* dst, const CUtensorMap* map, int row0, int kb, uint64_t* bar) {
    if (MN) {
#pragma unroll
        for (int i = 0; i < ROWS / 64; ++i) tma_load_2d(dst + i * kMnBlockBytes, map, row0 + 64 * i, kb * BK, bar);
    } else {
        tma_load_2d(dst, map, kb * BK, row0, bar);
    }
}

// Momentum update (as k_update_bf16) of 32 rows x 16 columns of a pooled-change
// tile, from the warp's TMEM lanes: the sums pass through the warp's 2 KB of shared
// memory (16-byte pieces permuted by row), after which lane (row lane / 4 + 8 j,
// piece lane % 4) owns 4 consecutive columns, so that theta, V and the bf16 copy
// move in whole 32-byte sectors.  w4 and v4 hold the block's theta and V, loaded ahead.
struct UpdBlock {
    float4 w4[4], v4[4];
};
__device__ __forceinline__ void update_block_load(const UpdArgs& a, const LayerUpd& u, int M, int N, int m0, int n0,
                                                  UpdBlock& x) {
    const int lane = threadIdx.x & 31, n = n0 + 4 * (lane & 3);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int m = m0 + 8 * j + (lane >> 2);
        x.w4[j] = x.v4[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m < M && n < N) {   // N is a multiple of 8
            const long long e = u.woff + (long long)m * N + n;
            x.w4[j] = __ldcs(reinterpret_cast<const float4*>(a.theta + e));
            x.v4[j] = __ldcs(reinterpret_cast<const float4*>(a.V + e));
        }
    }
}
__device__ __forceinline__ void update_block_apply(const UpdArgs& a, const LayerUpd& u, int M, int N, int m0, int n0,
                                                   const float (&r)[16], UpdBlock& x, float4* sF) {
    const int lane = threadIdx.x & 31, piece = lane & 3, n = n0 + 4 * piece;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        sF[lane * 4 + (k ^ ((lane >> 1) & 3))] = make_float4(r[4 * k], r[4 * k + 1], r[4 * k + 2], r[4 * k + 3]);
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int row = 8 * j + (lane >> 2), m = m0 + row;
        float4 g = sF[row * 4 + (piece ^ ((row >> 1) & 3))];
        if (m >= M || n >= N) continue;
        const long long i = (long long)m * N + n, e = u.woff + i;
        if (a.fold_g) {
            g = add4(g, *reinterpret_cast<const float4*>(a.G + e));
            *reinterpret_cast<float4*>(a.G + e) = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        const float* gc = &g.x;
        float* wc = &x.w4[j].x;
        float* vc = &x.v4[j].x;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float vel = a.lr_gs * guard_change(a, gc[c]) + a.momentum * vc[c];
            vc[c] = vel;
            wc[c] += vel;
        }
        __stcs(reinterpret_cast<float4*>(a.V + e), x.v4[j]);
        __stcs(reinterpret_cast<float4*>(a.theta + e), x.w4[j]);
        __align__(8) __nv_bfloat162 h[2];
        h[0] = __floats2bfloat162_rn(x.w4[j].x, x.w4[j].y);
        h[1] = __floats2bfloat162_rn(x.w4[j].z, x.w4[j].w);
        *reinterpret_cast<uint2*>(u.wb + i) = *reinterpret_cast<const uint2*>(h);
    }
    __syncwarp();   // the block may be rewritten
}

template <int BN, class Work>
__device__ __forceinline__ void gemm_body(const Work work) {
    using Cfg = GemmCfg<BN>;
    constexpr int MODE = Work::kMode;
    constexpr int S = Cfg::kStages;
    const auto& g = work.g;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t* ring = smem;
    float* colsum = reinterpret_cast<float*>(smem + Cfg::kRingBytes);   // [4][BN]
    bf16* stage_out = reinterpret_cast<bf16*>(smem + Cfg::kRingBytes + Cfg::kColsumBytes);
    float* bias_s = reinterpret_cast<float*>(smem + Cfg::kRingBytes + Cfg::kColsumBytes +
                                             Cfg::kStageOutBytes);   // [2][BN]
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + Cfg::kRingBytes + Cfg::kColsumBytes +
                                                 Cfg::kStageOutBytes + Cfg::kBiasBytes);
    uint64_t* full = bars;              // [S]
    uint64_t* empty = bars + S;         // [S]
    // Accumulators: two, so that the epilogue of a tile overlaps the next one's MMAs; as many as
    // fit in the pooled changes, whose chains are short where tiles are narrow (208-128-32 by
    // 512, eight chains of one K block: 19.2 us per update with two, 17.7 with eight).
    constexpr bool kDw = MODE == MODE_DW || MODE == MODE_DWU;
    constexpr int kAcc = kDw ? 512 / BN : 2;
    constexpr int kTmemCols = kAcc * BN;
    static_assert((2 * S + 2 * kAcc + 2) * sizeof(uint64_t) <= 512, "room for the barriers");
    uint64_t* tfull = bars + 2 * S;            // [kAcc]
    uint64_t* tempty = tfull + kAcc;           // [kAcc]
    uint64_t* drain = tempty + kAcc;           // [1] used only when a wait ran out
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int items = work.items();
    const Item first = work.item(blockIdx.x);   // (the grid has at most one CTA per item)

    pdl_launch();
    if (threadIdx.x == 32 * 2) work.prefetch_maps();
    work.touch();
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < kAcc; ++a) {
            mbar_init(&tfull[a], 1);
            mbar_init(&tempty[a], kEpiThreads);
        }
        mbar_init(drain, 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(tmem_slot)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    pdl_wait();   // every thread, before its first access to what earlier kernels wrote or still read

    if (warp == 0) {
        // ---------------- TMA producer
        if (elect_one()) {
            int stage = 0, issued = 0;   // copies issued so far
            unsigned phase = 0;
            bool ok = true, free_ = true;   // the stage's buffer is known to be free (all are at first)
            Item w = first;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
                if (it != (int)blockIdx.x) w = work.item(it);
                const CUtensorMap *ma = work.map_a(w), *mb = work.map_b(w);
                for (int kb = w.kb0; kb < w.kb1; ++kb) {
                    if (!free_ && !mbar_wait(&empty[stage], phase ^ 1u, abort_flag, g.flags)) { ok = false; break; }
                    uint8_t* sa = ring + stage * Cfg::kStageBytes;
                    mbar_expect_tx(&full[stage], Cfg::kStageBytes);
                    load_operand<BM, Work::kAMn>(sa, ma, w.mb * BM, kb, &full[stage]);
                    load_operand<BN, Work::kBMn>(sa + Cfg::kABytes, mb, w.nb * BN, kb, &full[stage]);
                    ++issued;
                    if (++stage == S) { stage = 0; phase ^= 1u; }
                    free_ = issued < S || mbar_test(&empty[stage], phase ^ 1u);
                }
            }
            if (!ok) {
                // let every copy already issued land before the CTA can exit
                for (int n = issued - 1; n >= 0 && n >= issued - S; --n) {   // each stage's last copy
                    const unsigned long long t0 = global_ns();
                    while (!mbar_try_wait(&full[n % S], (unsigned)(n / S) & 1u) && global_ns() - t0 < kWaitNs) {
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer
        if (elect_one()) {
            constexpr uint32_t idesc = idesc_bf16(BM, BN, Work::kAMn, Work::kBMn);
            const uint32_t a0 = desc_lo<Work::kAMn>(smem_u32(ring)), b0 = desc_lo<Work::kBMn>(smem_u32(ring) + Cfg::kABytes);
            int stage = 0;
            unsigned phase = 0;
            int acc = 0;
            unsigned acc_phase = 0;
            bool ok = true, ready = false;   // the stage's operands are known to be there
            bool issued_any = false;
            Item w = first;
            for (int it = blockIdx.x; it < items && ok; it += gridDim.x) {
                if (it != (int)blockIdx.x) w = work.item(it);
                for (int c0 = w.kb0; c0 < w.kb1; c0 += w.chain) {
                    const int c1 = min(w.kb1, c0 + w.chain);
                    if (!mbar_wait(&tempty[acc], acc_phase ^ 1u, abort_flag, g.flags)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t tmem_d = tmem_base + (uint32_t)(acc * BN);
                    uint32_t accumulate = 0;
                    for (int kb = c0; kb < c1; ++kb) {
                        if (!ready && !mbar_wait(&full[stage], phase, abort_flag, g.flags)) { ok = false; break; }
                        tc_fence_after();
                        const uint32_t al = a0 + stage * (Cfg::kStageBytes >> 4), bl = b0 + stage * (Cfg::kStageBytes >> 4);
                        umma_bf16<idesc>(tmem_d, al, bl, accumulate);
#pragma unroll
                        for (int kk = 1; kk < BK / UMMA_K; ++kk)
                            umma_bf16<idesc>(tmem_d, al + kk * k_step_units<Work::kAMn>(), bl + kk * k_step_units<Work::kBMn>(), 1u);
                        accumulate = 1u;
                        issued_any = true;
                        umma_commit(&empty[stage]);
                        if (++stage == S) { stage = 0; phase ^= 1u; }
                        ready = mbar_test(&full[stage], phase);
                    }
                    if (!ok) break;
                    umma_commit(&tfull[acc]);
                    if (++acc == kAcc) { acc = 0; acc_phase ^= 1u; }
                }
            }
            if (!ok && issued_any) {
                // let every MMA already issued finish before TMEM is released
                umma_commit(drain);
                const unsigned long long t0 = global_ns();
                while (!mbar_try_wait(drain, 0) && global_ns() - t0 < kWaitNs) {
                }
            }
        }
    } else {
        // ---------------- epilogue warps 2..9
        const int q = warp & 3;                  // TMEM lane quarter this warp may access
        const int ew = warp - 2;                 // 0..7
        const int slot = ew & 3;                 // row quarter's slot in the column-sum scratch
        const int cbeg = (ew >> 2) * (BN / 2);   // this warp's half of the columns
        int acc = 0;
        unsigned acc_phase = 0;
        if constexpr (MODE == MODE_DWU) {
            // this CTA's share of the biases and the error sum, while the first tile accumulates
            const int nb = work.u.bias_blocks + (work.u.sse_out != nullptr ? 1 : 0);
            for (int b = blockIdx.x; b < nb; b += gridDim.x)
                update_bias_block(work.u, b, threadIdx.x - 64, colsum, [] { epi_bar(); });
        }
        Item w = first;
        for (int it = blockIdx.x; it < items; it += gridDim.x) {
            if (it != (int)blockIdx.x) w = work.item(it);
            float* sbias = bias_s + acc * BN;
            if constexpr (MODE == MODE_FWD || MODE == MODE_FWD_OUT) {
                // block acc was last read two tiles ago, before the barrier of the previous tile
                for (int c = threadIdx.x - 64; c < BN; c += kEpiThreads) {
                    const int n = w.nb * BN + c;
                    sbias[c] = n < g.N ? g.bias[n] : 0.f;
                }
            }
            const int m0 = w.mb * BM + q * 32, m = m0 + lane;
            Row32 aux[2];   // the targets' or activations' block of this chunk and of the next one
            auto load_aux = [&](int c0, Row32& r) {
                if constexpr (MODE == MODE_FWD_OUT || MODE == MODE_DX) {
                    const int n0 = w.nb * BN + c0;
                    const bf16* p = g.aux + (size_t)m0 * g.ld_aux + n0;
                    if (g.aux == nullptr) return;
                    if (BN > 64) load_block(r, p, g.ld_aux, g.M - m0, (g.N - n0) >> 3);
                    else load_own_row(r, p, g.ld_aux, g.M - m0, (g.N - n0) >> 3);
                }
            };
            load_aux(cbeg, aux[0]);
            // Waits for the accumulator; false if that ran out.  With barriers between the epilogue
            // warps below, they leave together: the abort flag may rise between two warps' reads
            // of it, and a warp that stayed would wait for those that left.
            auto wait_acc = [&] {
                const bool got = mbar_wait(&tfull[acc], acc_phase, abort_flag, g.flags);
                const bool leave = kDw ? __any_sync(0xffffffffu, !got) : epi_any(!got || *abort_flag != 0);
                tc_fence_after();
                return !leave;
            };
            // This warp's lanes of an accumulator; that accumulator is free for the next sum.
            const uint32_t trow = tmem_base + ((uint32_t)(q * 32) << 16);
            auto release = [&](int a) {
                tc_fence_before();
                mbar_arrive(&tempty[a]);
            };
            auto next_acc = [&] {
                if (++acc == kAcc) { acc = 0; acc_phase ^= 1u; }
            };
            if constexpr (kDw) {
                const DwLayer& y = g.ly[w.l];
                const int ncol = y.N - w.nb * BN;   // columns of the layer from this tile on
                // The sums of the chains before the last one: in registers up to 128 columns, as
                // many as a thread holds beside the update's loads.  At 256 the two accumulators
                // take turns: each chain's sum has the one before added in place, which then is
                // free for the chain after it (its MMAs wait for that, about 1,000 clocks, which
                // a chain of 128 K blocks, 68,000, does not feel; through global memory, 128 KB
                // a CTA and tile, 50 steps of 4096^5 took 210.0 ms).
                constexpr bool kRegs = BN <= 128;
                float part[kRegs ? BN / 2 : 1];
                if constexpr (kRegs) {
#pragma unroll
                    for (int c = 0; c < BN / 2; ++c) part[c] = 0.f;
                }
                auto add_previous = [&] {   // 256 columns: accumulator 1 - acc into acc
                    for (int c = cbeg; c < cbeg + BN / 2; c += 16) {
                        float x[16], v[16];
                        tmem_ld16(trow + (uint32_t)((1 - acc) * BN + c), x);
                        tmem_ld16(trow + (uint32_t)(acc * BN + c), v);
#pragma unroll
                        for (int k = 0; k < 16; ++k) v[k] += x[k];
                        tmem_st16(trow + (uint32_t)(acc * BN + c), v);
                    }
                    tmem_wait_st();
                    release(1 - acc);
                };
                UpdBlock cur, nxt;
                auto load = [&](int c, UpdBlock& b) {
                    if constexpr (MODE == MODE_DWU)
                        update_block_load(work.u, work.u.ly[w.l], y.M, y.N, m0, w.nb * BN + cbeg + c, b);
                };
                load(0, cur);   // arrives while the chains accumulate (after them: 17.7 us, not 17.2)
                bool stay = true;
                for (int c0 = w.kb0; c0 + w.chain < w.kb1; c0 += w.chain) {
                    stay = wait_acc();
                    if (!stay) break;
                    if constexpr (kRegs) {
#pragma unroll
                        for (int i = 0; i < BN / 64; ++i) {
                            float v[32];
                            tmem_ld32(trow + (uint32_t)(acc * BN + cbeg + 32 * i), v);
#pragma unroll
                            for (int c = 0; c < 32; ++c) part[32 * i + c] += v[c];
                        }
                        release(acc);
                    } else if (c0 > w.kb0) {
                        add_previous();
                    }
                    next_acc();
                }
                if (!stay) break;
                const bool several = w.kb1 - w.kb0 > w.chain;
                if constexpr (MODE == MODE_DWU) {
                    const LayerUpd& u = work.u.ly[w.l];
                    float4* sF = reinterpret_cast<float4*>(stage_out + ew * 1024);
                    auto apply = [&](int c, UpdBlock& b) {
                        float r[16];
                        tmem_ld16(trow + (uint32_t)(acc * BN + cbeg + c), r);
                        if constexpr (kRegs) {
#pragma unroll
                            for (int k = 0; k < 16; ++k) r[k] += part[c + k];
                        }
                        update_block_apply(work.u, u, y.M, y.N, m0, w.nb * BN + cbeg + c, r, b, sF);
                    };
                    if (!wait_acc()) break;
                    if (!kRegs && several) add_previous();
#pragma unroll(kRegs ? BN / 64 : 1)
                    for (int i = 0; i < BN / 64; ++i) {
                        if (cbeg + 32 * i >= ncol) break;
                        load(32 * i + 16, nxt);
                        apply(32 * i, cur);
                        if (i + 1 < BN / 64) load(32 * i + 32, cur);
                        apply(32 * i + 16, nxt);
                    }
                } else {
                    if (!wait_acc()) break;
                    if (!kRegs && several) add_previous();
#pragma unroll(kRegs ? BN / 64 : 1)
                    for (int i = 0; i < BN / 64; ++i) {
                        if (cbeg + 32 * i >= ncol) break;
                        float v[32];
                        tmem_ld32(trow + (uint32_t)(acc * BN + cbeg + 32 * i), v);
                        if constexpr (kRegs) {
#pragma unroll
                            for (int c = 0; c < 32; ++c) v[c] += part[32 * i + c];
                        }
                        store_partial(y.gpart, y.M, y.N, m, w.nb * BN + cbeg + 32 * i, w.split, v);
                    }
                }
                release(acc);
                next_acc();
            } else {
                if (!wait_acc()) break;
                const bool row_ok = m < g.M;
                float sse = 0.f;
                bf16* sS = stage_out + ew * 1024;
                const bool want_colsum = (MODE == MODE_DX) || (MODE == MODE_FWD_OUT && g.aux != nullptr);
#pragma unroll 2
                for (int i = 0; i < BN / 64; ++i) {
                    const int c0 = cbeg + 32 * i, n0 = w.nb * BN + c0;
                    if (n0 >= g.N) break;   // (column sums past N are not read)
                    if (i + 1 < BN / 64) load_aux(c0 + 32, aux[(i + 1) & 1]);
                    float v[32];
                    tmem_ld32(trow + (uint32_t)(acc * BN + c0), v);
                    epilogue_chunk<BN, MODE>(g, m0, n0, v, sse, row_ok, sS, sbias + c0, aux[i & 1],
                                         want_colsum ? colsum + slot * BN + c0 : nullptr);
                }
                release(acc);   // TMEM is free for the next accumulation into this buffer
                next_acc();
                if (want_colsum) {
                    epi_bar();
                    const int t = threadIdx.x - 64;   // 0 .. kEpiThreads - 1
                    for (int c = t; c < BN; c += kEpiThreads) {
                        const int n = w.nb * BN + c;
                        if (n < g.N) {
                            const float s = (colsum[c] + colsum[BN + c]) + (colsum[2 * BN + c] + colsum[3 * BN + c]);
                            g.bias_part[(size_t)w.mb * g.N + n] = s;
                        }
                    }
                    if (MODE == MODE_FWD_OUT) {
                        // tile error sum: warp sums, then the eight warps in a fixed order
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) sse += __shfl_xor_sync(0xffffffffu, sse, o);
                        epi_bar();
                        if (lane == 0) colsum[ew] = sse;
                        epi_bar();
                        if (t == 0)
                            g.sse_part[it] = ((colsum[0] + colsum[1]) + (colsum[2] + colsum[3])) +
                                             ((colsum[4] + colsum[5]) + (colsum[6] + colsum[7]));
                    }
                    epi_bar();
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base),
                     "r"(kTmemCols)
                     : "memory");
    }
}

template <int BN, int MODE>
__global__ void __launch_bounds__(kGemmThreads, 1)
    k_gemm(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
           const __grid_constant__ GemmArgs g) {
    gemm_body<BN>(OneGemm<MODE>{g, &map_a, &map_b});
}

template <int BN>
__global__ void __launch_bounds__(kGemmThreads, 1)
    k_gemm_dw(const __grid_constant__ DwMaps maps, const __grid_constant__ DwArgs g) {
    gemm_body<BN>(DwGemm{g, maps});
}

template <int BN>
__global__ void __launch_bounds__(kGemmThreads, 1)
    k_gemm_dwu(const __grid_constant__ DwMaps maps, const __grid_constant__ DwArgs g, const __grid_constant__ UpdArgs u) {
    gemm_body<BN>(DwuGemm(g, maps, u));
}

// ------------------------------------------------------------ SIMT kernels
// Output deltas from stored outputs (bp_backward): delta = (t - o) o (1 - o),
// delta rows, per-128-row column sums and error sums.  One block of 256 threads
// per 128 rows x 64 columns; a thread moves 8 columns of 4 rows in 16-byte pieces.
__global__ void __launch_bounds__(256) k_output_delta(const bf16* O, const bf16* T, int M, int N, bf16* D,
                                                      float* bias_part, float* sse_part) {
    __shared__ float cs[8][64];
    __shared__ float ss[8];
    const int mb = blockIdx.y, nc = blockIdx.x;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int piece = threadIdx.x & 7;
    const int n = nc * 64 + piece * 8;   // N is a multiple of 8: a piece is whole or outside
    pdl_launch();
    pdl_wait();
    float sums[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) sums[q] = 0.f;
    float sse = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int m = mb * 128 + j * 32 + (threadIdx.x >> 3);
        if (m >= M || n >= N) continue;
        const size_t e = (size_t)m * N + n;
        const uint4 uo = *reinterpret_cast<const uint4*>(O + e);
        const uint4 ut = *reinterpret_cast<const uint4*>(T + e);
        const __nv_bfloat162* ho = reinterpret_cast<const __nv_bfloat162*>(&uo);
        const __nv_bfloat162* ht = reinterpret_cast<const __nv_bfloat162*>(&ut);
        __align__(16) __nv_bfloat162 hd[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 o = __bfloat1622float2(ho[q]), t = __bfloat1622float2(ht[q]);
            const float e0 = t.x - o.x, e1 = t.y - o.y;
            sse = fmaf(e0, e0, sse);
            sse = fmaf(e1, e1, sse);
            hd[q] = __floats2bfloat162_rn(e0 * o.x * (1.f - o.x), e1 * o.y * (1.f - o.y));
            const float2 d = __bfloat1622float2(hd[q]);
            sums[2 * q] += d.x;
            sums[2 * q + 1] += d.y;
        }
        *reinterpret_cast<uint4*>(D + e) = *reinterpret_cast<const uint4*>(hd);
    }
    // the four rows of a warp's lanes per piece (lane bits 3, 4), then the eight warps
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        sums[q] += __shfl_xor_sync(0xffffffffu, sums[q], 8);
        sums[q] += __shfl_xor_sync(0xffffffffu, sums[q], 16);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sse += __shfl_xor_sync(0xffffffffu, sse, o);
    if (lane < 8) {
#pragma unroll
        for (int q = 0; q < 8; ++q) cs[w][lane * 8 + q] = sums[q];
    }
    if (lane == 0) ss[w] = sse;
    __syncthreads();
    if (threadIdx.x < 64) {
        const int c = nc * 64 + threadIdx.x;
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += cs[k][threadIdx.x];
        if (c < N) bias_part[(size_t)mb * N + c] = s;
    }
    if (threadIdx.x == 64) {
        float s = 0.f;
#pragma unroll
        for (int k = 0; k < 8; ++k) s += ss[k];
        sse_part[(size_t)mb * gridDim.x + nc] = s;
    }
}

// Momentum update of Section 6.2.1: g = sum of partial changes (+ pending G);
// v = lr*gs*g + m*v; w += v; then the bf16 copy.  Mode 1 adds the partial changes
// into G instead.  Bound by DRAM: a block owns 2,048 consecutive weights, every
// thread two float4 pieces whose loads (weights, changes, up to two partial
// planes at a time) are all issued before the first store.
__global__ void __launch_bounds__(kUpdThreads) k_update_bf16(const __grid_constant__ UpdArgs a) {
    __shared__ float red[kUpdSlices * kUpdBiases];
    const int t = threadIdx.x;
    pdl_launch();
    pdl_wait();
    const int b = blockIdx.x;
    if (b >= a.blocks) {
        update_bias_block(a, b - a.blocks, t, red, [] { __syncthreads(); });
        return;
    }
    int l = 0;
    while (l + 1 < a.L && b >= a.ly[l + 1].block0) ++l;
    const LayerUpd& u = a.ly[l];
    const long long e0 = (long long)(b - u.block0) * kUpdFloats + t * 4;
    float4 g4[kUpdPieces], w4[kUpdPieces], v4[kUpdPieces];
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kUpdPieces; ++k) {
        const long long e = e0 + k * (kUpdThreads * 4);
        g4[k] = w4[k] = v4[k] = z;
        if (e >= u.nw) continue;
        if (a.mode != 1) w4[k] = *reinterpret_cast<const float4*>(a.theta + u.woff + e);
        if (a.mode == 0) v4[k] = *reinterpret_cast<const float4*>(a.V + u.woff + e);
        if (a.mode == 1 || a.fold_g) g4[k] = *reinterpret_cast<const float4*>(a.G + u.woff + e);
    }
    float4 p4[kUpdPieces];
#pragma unroll
    for (int k = 0; k < kUpdPieces; ++k) p4[k] = z;
#pragma unroll 2
    for (int s = 0; s < a.splits; ++s) {
#pragma unroll
        for (int k = 0; k < kUpdPieces; ++k) {
            const long long e = e0 + k * (kUpdThreads * 4);
            if (e < u.nw) p4[k] = add4(p4[k], __ldcs(reinterpret_cast<const float4*>(u.gpart + s * u.nw + e)));
        }
    }
#pragma unroll
    for (int k = 0; k < kUpdPieces; ++k) {
        const long long e = e0 + k * (kUpdThreads * 4);
        if (e >= u.nw) continue;
        const float4 g = add4(p4[k], g4[k]);
        if (a.mode == 1) {
            *reinterpret_cast<float4*>(a.G + u.woff + e) = g;
            continue;
        }
        if (a.mode == 0) {
            const float* gc = &g.x;
            float* wc = &w4[k].x;
            float* vc = &v4[k].x;
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float vel = a.lr_gs * guard_change(a, gc[c]) + a.momentum * vc[c];
                vc[c] = vel;
                wc[c] += vel;
            }
            *reinterpret_cast<float4*>(a.V + u.woff + e) = v4[k];
            *reinterpret_cast<float4*>(a.theta + u.woff + e) = w4[k];
            if (a.fold_g) *reinterpret_cast<float4*>(a.G + u.woff + e) = z;
        }
        __align__(8) __nv_bfloat162 h[2];
        h[0] = __floats2bfloat162_rn(w4[k].x, w4[k].y);
        h[1] = __floats2bfloat162_rn(w4[k].z, w4[k].w);
        *reinterpret_cast<uint2*>(u.wb + e) = *reinterpret_cast<const uint2*>(h);
    }
}

// ------------------------------------------------------------ host side
std::string g_msg;

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

bool get_encoder() {
    if (!g_encode) g_encode = tensor_map_encoder();
    return g_encode != nullptr;
}

// 2-D bf16 tensor map over a row-major [rows, cols] matrix (pitch cols), box =
// box_rows x 64 columns, 128-byte swizzle, zero fill.  box_rows is the tile edge
// for an operand whose rows run along K, BK for one whose rows run along M or N.
bool make_map(CUtensorMap* map, const void* base, int rows, int cols, int box_rows) {
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
    cuuint32_t box[2] = {64, (cuuint32_t)box_rows};
    cuuint32_t estr[2] = {1, 1};
    CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                          CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS;
}

template <int BN>
cudaError_t gemm_setup() {
    const void* fns[] = {(const void*)k_gemm<BN, MODE_FWD>, (const void*)k_gemm<BN, MODE_FWD_OUT>,
                         (const void*)k_gemm<BN, MODE_DX>, (const void*)k_gemm_dw<BN>, (const void*)k_gemm_dwu<BN>};
    for (const void* f : fns) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   GemmCfg<BN>::kSmemBytes);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

std::mutex g_mu;
bool g_ready[64];

cudaError_t setup_all(int device) {
    std::lock_guard<std::mutex> lk(g_mu);
    if (device < 64 && g_ready[device]) return cudaSuccess;
    cudaError_t e;
    if ((e = gemm_setup<64>()) != cudaSuccess) return e;
    if ((e = gemm_setup<128>()) != cudaSuccess) return e;
    if ((e = gemm_setup<256>()) != cudaSuccess) return e;
    if (device < 64) g_ready[device] = true;
    return cudaSuccess;
}

// Launch whose setup may overlap the previous kernel's tail (the kernel calls pdl_wait).
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), int grid_x, int grid_y, int threads, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid_x, grid_y);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, std::forward<A>(args)...);
}

}  // namespace

struct Bf16Net {
    int L = 0;
    int n[BP_MAX_SIZES] = {0};
    int cap = 0;
    int num_sms = 0;
    float* theta = nullptr;
    float* V = nullptr;
    float* G = nullptr;
    int* flags = nullptr;       // [0] error bits, [1] fault-guard count
    float guard = 0.f;          // fault guard of Section 8 (0: off)
    long long woff[BP_MAX_SIZES] = {0}, boff[BP_MAX_SIZES] = {0};
    bf16* wb[BP_MAX_SIZES] = {nullptr};     // W_l   [n_l, n_{l-1}]
    bf16* act[BP_MAX_SIZES] = {nullptr};    // A_l   [cap, n_l], l >= 1
    bf16* dlt[BP_MAX_SIZES] = {nullptr};    // delta_l [cap, n_l], l >= 1
    float* gpart[BP_MAX_SIZES] = {nullptr}; // [max_splits, n_l, n_{l-1}]
    int max_splits = 1;
    float* bpart[BP_MAX_SIZES] = {nullptr}; // [mtiles(cap), n_l]
    float* sse_part = nullptr;              // [mtiles(cap) * 64-column tiles along n_L]
    std::vector<void*> allocs;
};

namespace {

bool alloc(Bf16Net* b, void** p, size_t bytes) {
    if (cudaMalloc(p, bytes) != cudaSuccess) return false;
    b->allocs.push_back(*p);
    return true;
}

int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

int tiles_of(int M, int N, int bn) { return ceil_div(M, BM) * ceil_div(N, bn); }

// Clocks of a K block (64 of K) of a 128 x bn tile with every SM busy, fitted to
// whole steps at forced widths (the MMAs alone: 512, 256, 128).  Half the width costs
// more than half the time: each SM then re-reads A twice as often from L2, and the
// loops that issue copies and MMAs take about 300 clocks a block themselves (two 64s
// of K a block at the narrow widths were 1-3% slower).
constexpr double kb_clocks(int bn) { return bn == 256 ? 530 : bn == 128 ? 330 : 230; }

// Tile width of a launch.  A tile's time is its K loop or its epilogue, whichever
// is longer (they overlap across tiles), once per wave of tiles over the SMs, plus
// the other one at the end.  Narrow tiles fill the chip when the batch or the
// layer is small: the forward of 512 patterns of 208-1024-32 takes 9.3 / 10.7 / 14.7 us
// with all launches at 64 / 128 / 256 columns, of 1,001 of 1024-2048-2048-512 29.5 /
// 27.2 / 41.0 (25.5 by this rule); large batches want 256: a step of 8,192 of
// 1024-2048-2048-512 364 / 298 / 296.
int pick_bn(int M, int N, int kb, int num_sms) {
    const int bns[3] = {256, 128, 64};
    int best = 256;
    double best_t = 0;
    for (int bn : bns) {
        const double waves = ceil_div(tiles_of(M, N, bn), num_sms);
        const double k = kb * kb_clocks(bn), e = 800.0 + 900.0 * bn / 64;
        const double t = waves * (k > e ? k : e) + (k > e ? e : k);
        if (bn == 256 || t < best_t) {
            best = bn;
            best_t = t;
        }
    }
    return best;
}

template <int MODE>
cudaError_t launch_gemm(const Bf16Net* b, const bf16* A, const bf16* Bop, GemmArgs g, cudaStream_t s) {
    g.kb_total = ceil_div(g.K, BK);
    const int bn = pick_bn(g.M, g.N, g.kb_total, b->num_sms);
    g.num_m = ceil_div(g.M, BM);
    g.num_n = ceil_div(g.N, bn);
    g.flags = b->flags;
    CUtensorMap ma, mb;
    const bool ok = make_map(&ma, A, g.M, g.K, BM) &&
                    (MODE == MODE_DX ? make_map(&mb, Bop, g.K, g.N, BK) : make_map(&mb, Bop, g.N, g.K, bn));
    if (!ok) return cudaErrorInvalidValue;
    const int items = g.num_m * g.num_n;
    const int grid = items < b->num_sms ? items : b->num_sms;
    switch (bn) {
        case 64: return launch_pdl(k_gemm<64, MODE>, grid, 1, kGemmThreads, GemmCfg<64>::kSmemBytes, s, ma, mb, g);
        case 128: return launch_pdl(k_gemm<128, MODE>, grid, 1, kGemmThreads, GemmCfg<128>::kSmemBytes, s, ma, mb, g);
        default: return launch_pdl(k_gemm<256, MODE>, grid, 1, kGemmThreads, GemmCfg<256>::kSmemBytes, s, ma, mb, g);
    }
}

GemmArgs blank_args() {
    GemmArgs g;
    memset(&g, 0, sizeof g);
    return g;
}

// Forward pass of all layers.  With T, also the output deltas (training), which
// replace the outputs; without, the outputs go to act[L] (for a backward) and Y.
cudaError_t run_forward(Bf16Net* b, const bf16* X, int B, const bf16* T, bf16* Y, cudaStream_t s) {
    const int L = b->L;
    for (int l = 1; l <= L; ++l) {
        const bf16* A = (l == 1) ? X : b->act[l - 1];
        GemmArgs g = blank_args();
        g.M = B;
        g.N = b->n[l];
        g.K = b->n[l - 1];
        g.bias = b->theta + b->boff[l];
        cudaError_t e;
        if (l < L) {
            g.out = b->act[l];
            g.ldo = b->n[l];
            e = launch_gemm<MODE_FWD>(b, A, b->wb[l], g, s);
        } else {
            if (T != nullptr) {
                g.aux = T;
                g.ld_aux = b->n[L];
                g.out2 = b->dlt[L];
                g.bias_part = b->bpart[L];
                g.sse_part = b->sse_part;
            } else {
                g.out = b->act[L];
                g.ldo = b->n[L];
                g.out2 = Y;
            }
            g.ld2 = b->n[L];
            e = launch_gemm<MODE_FWD_OUT>(b, A, b->wb[l], g, s);
        }
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// K blocks that one sum of a layer's pooled change runs over in TMEM.  The tensor cores
// truncate as they accumulate, so that a sum's error grows with its chain: 2-norm error
// against float64 of the change of 4096 x 4096 weights, one chain / this rule, 8,192
// patterns 8.1e-6 / 3.7e-6, 16,384 1.7e-5 / 8.0e-6; 208 x 1024 by 512 3.4e-7 / 1.2e-7.
// The epilogue adds the chains' sums, rounding to nearest.  Their number s is the split of K
// that would be fastest with 128 x 256 tiles and a plane of partial sums each: the least of
//   ceil(tiles * s / num_sms) / s  (waves of 1/s-K items, in times of a full-K tile)
//   + s * tiles * plane            (writing and reading a plane; a tile's share of it over
//                                   its MMAs is 4 / K times the 1.87 bf16 flops an SM does
//                                   in the time of a byte of DRAM traffic),
// many for the few tiles of a small layer, one or two for a layer of several waves.  us,
// one chain / this rule: 25 steps of 8,192 of 1024-2048-2048-512 7,248 / 7,303, 50 steps of
// 4096^5 201,690 / 201,520, two epochs of 16,200 of 208-1024-32 by 512 1,332 / 1,333, an
// update of 208-128-32 by 512 16.7 / 17.2.
constexpr int kMaxChains = 16;
int sum_chain(int M, int N, int kb_total, int num_sms) {
    const int tiles = tiles_of(M, N, 256);
    const double plane = 4.0 * 1.87 / ((double)kb_total * BK);
    int best = 1;
    double best_cost = 0.0;
    for (int s = 1; s <= kMaxChains && s <= kb_total; ++s) {
        const double waves = (double)(((long long)tiles * s + num_sms - 1) / num_sms) / s;
        const double cost = waves + s * plane * tiles;
        if (s == 1 || cost < best_cost * (1.0 - 1e-9)) {
            best = s;
            best_cost = cost;
        }
    }
    return ceil_div(kb_total, best);
}

// How the pooled-change launch of a group of B patterns is cut: the tile width,
// the number of K splits, and whether the update runs in its epilogue (training, one
// split).  All layers share the launch, so their tiles fill the last wave together.
// The choice minimises, in clocks,
//   fused:   as pick_bn, with the update of a tile (18 bytes a weight through an SM's
//            share of DRAM) as the epilogue;
//   split:   ceil(tiles * s / num_sms) * K blocks / s * kb_clocks   (waves of 1/s-K items)
//            + s fp32 partial planes, written here and read by the update, at 3,285 B a
//            clock (the measured 6.8 TB/s copy rate at 2.07 GHz)
//            + the update kernel's 18 bytes a weight at the same rate and 8,000 clocks
//            of one more launch in the chain.
// us per step, split at its best / fused at 64 / 128 / 256 columns: 208-1024-32 at 512
// patterns 21.9 / 20.6 / 24.4 / 29.7; 1024-2048-2048-512 at 1,001 90.6 / 82.2 / 84.5 /
// 93.5, at 8,192 294.0 / 313.4 / 281.4 / 296.4; 2048-2048-2048 at 2,048 117.7 / 109.9 /
// 114.3 / 116.4; 128-256-256-64 at 8,192, whose 16 tiles leave the chip idle unsplit,
// 39.9 / 48.5 / 57.1 / 75.2.  (All with one chain per run of K blocks; in chains, see
// sum_chain, they change by less than 1%.)
constexpr int kMaxSplits = 16;
struct DwPlan {
    int bn, tiles, splits, kb_total, kb_per_split;
    bool fused;     // the update runs in the pooled-change launch's epilogue
};
DwPlan dw_plan(const int* n, int L, int B, int num_sms, int max_splits, bool may_fuse) {
    DwPlan p{};
    p.kb_total = ceil_div(B, BK);
    double best = 0, weights = 0;
    for (int l = 1; l <= L; ++l) weights += (double)n[l] * n[l - 1];
    auto take = [&](double t, int bn, int tiles, int splits, bool fused) {
        if (best != 0 && t >= best * (1.0 - 1e-9)) return;
        best = t;
        p.bn = bn;
        p.tiles = tiles;
        p.splits = splits;
        p.fused = fused;
    };
    const double hbm = 3285;   // bytes per clock
    const int bns[3] = {256, 128, 64};
    for (int bn : bns) {
        int tiles = 0;
        for (int l = 1; l <= L; ++l) tiles += tiles_of(n[l], n[l - 1], bn);
        const double loop = p.kb_total * kb_clocks(bn), plane = 8.0 * BM * bn * tiles / hbm;
        if (may_fuse) {
            const double upd = 7000.0 * bn / 64, waves = ceil_div(tiles, num_sms);
            take(waves * (loop > upd ? loop : upd) + (loop > upd ? upd : loop), bn, tiles, 1, true);
        }
        for (int s = 1; s <= max_splits && s <= p.kb_total; ++s) {
            const double waves = (double)(((long long)tiles * s + num_sms - 1) / num_sms) / s;
            take(waves * loop + s * plane + weights * 18 / hbm + 8000, bn, tiles, s, false);
        }
    }
    p.kb_per_split = ceil_div(p.kb_total, p.splits);
    p.splits = ceil_div(p.kb_total, p.kb_per_split);   // every split non-empty
    return p;
}

// Hidden deltas and pooled partial changes for every layer (deltas of layer L
// and the activations must already be in scratch).
cudaError_t run_backward(Bf16Net* b, const bf16* X, int B, const DwPlan& p, const UpdArgs* upd, cudaStream_t s) {
    const int L = b->L;
    for (int l = L; l >= 2; --l) {
        // delta_{l-1} = (delta_l W_l) * a (1 - a):  A = delta_l [B, n_l], B-operand = W_l along K
        GemmArgs g = blank_args();
        g.M = B;
        g.N = b->n[l - 1];
        g.K = b->n[l];
        g.out = b->dlt[l - 1];
        g.ldo = b->n[l - 1];
        g.aux = b->act[l - 1];
        g.ld_aux = b->n[l - 1];
        g.bias_part = b->bpart[l - 1];
        const cudaError_t e = launch_gemm<MODE_DX>(b, b->dlt[l], b->wb[l], g, s);
        if (e != cudaSuccess) return e;
    }
    // G_l = delta_l^T A_{l-1}
    DwArgs g{};
    DwMaps maps;
    memset(&maps, 0, sizeof maps);
    g.L = L;
    g.tiles = p.tiles;
    g.splits = p.splits;
    g.kb_per_split = p.kb_per_split;
    g.kb_total = p.kb_total;
    g.flags = b->flags;
    int tile = 0;
    for (int l = 1; l <= L; ++l) {
        DwLayer& y = g.ly[l - 1];
        y.M = b->n[l];
        y.N = b->n[l - 1];
        y.num_m = ceil_div(y.M, BM);
        y.num_n = ceil_div(y.N, p.bn);
        y.tile0 = tile;
        y.chain = sum_chain(y.M, y.N, p.kb_total, b->num_sms);
        tile += y.num_m * y.num_n;
        y.gpart = b->gpart[l];
        if (!make_map(&maps.a[l - 1], b->dlt[l], B, y.M, BK) ||
            !make_map(&maps.b[l - 1], l == 1 ? X : b->act[l - 1], B, y.N, BK))
            return cudaErrorInvalidValue;
    }
    const int items = p.tiles * p.splits;
    const int grid = items < b->num_sms ? items : b->num_sms;
    if (upd != nullptr) {
        switch (p.bn) {
            case 64: return launch_pdl(k_gemm_dwu<64>, grid, 1, kGemmThreads, GemmCfg<64>::kSmemBytes, s, maps, g, *upd);
            case 128: return launch_pdl(k_gemm_dwu<128>, grid, 1, kGemmThreads, GemmCfg<128>::kSmemBytes, s, maps, g, *upd);
            default: return launch_pdl(k_gemm_dwu<256>, grid, 1, kGemmThreads, GemmCfg<256>::kSmemBytes, s, maps, g, *upd);
        }
    }
    switch (p.bn) {
        case 64: return launch_pdl(k_gemm_dw<64>, grid, 1, kGemmThreads, GemmCfg<64>::kSmemBytes, s, maps, g);
        case 128: return launch_pdl(k_gemm_dw<128>, grid, 1, kGemmThreads, GemmCfg<128>::kSmemBytes, s, maps, g);
        default: return launch_pdl(k_gemm_dw<256>, grid, 1, kGemmThreads, GemmCfg<256>::kSmemBytes, s, maps, g);
    }
}

// splits, mtiles: partial changes pending (0: none).
UpdArgs upd_args(Bf16Net* b, int splits, int mtiles, int mode, bool fold, float lr_gs, float momentum, float* sse_out,
                 int n_sse) {
    UpdArgs a;
    memset(&a, 0, sizeof a);
    a.L = b->L;
    int blocks = 0, bias_blocks = 0;
    for (int l = 1; l <= b->L; ++l) {
        LayerUpd& u = a.ly[l - 1];
        u.n_out = b->n[l];
        u.nw = (long long)b->n[l] * b->n[l - 1];
        u.woff = b->woff[l];
        u.boff = b->boff[l];
        u.gpart = b->gpart[l];
        u.bias_part = b->bpart[l];
        u.wb = b->wb[l];
        u.block0 = blocks;
        u.bias0 = bias_blocks;
        blocks += ceil_div(u.nw, kUpdFloats);
        bias_blocks += ceil_div(u.n_out, kUpdBiases);
    }
    a.blocks = blocks;
    a.bias_blocks = bias_blocks;
    a.splits = splits;
    a.mtiles = mtiles;
    a.theta = b->theta;
    a.V = b->V;
    a.G = b->G;
    a.lr_gs = lr_gs;
    a.momentum = momentum;
    a.mode = mode;
    a.fold_g = fold ? 1 : 0;
    a.sse_part = b->sse_part;
    a.n_sse = n_sse;
    a.sse_out = sse_out;
    a.flags = b->flags;
    a.guard = b->guard;
    a.faults = reinterpret_cast<unsigned*>(b->flags + 1);
    return a;
}

cudaError_t launch_update(const UpdArgs& a, cudaStream_t s) {
    return launch_pdl(k_update_bf16, a.blocks + a.bias_blocks + (a.sse_out != nullptr ? 1 : 0), 1, kUpdThreads, 0, s, a);
}

}  // namespace

bp_status bf16_check_shape(const int* n, int L, int max_batch) {
    for (int l = 0; l <= L; ++l) {
        if (n[l] % 8 != 0) {
            char buf[200];
            snprintf(buf, sizeof buf,
                     "the bfloat16 path needs every layer size to be a multiple of 8 "
                     "(16-byte rows for TMA); layer %d has %d",
                     l, n[l]);
            g_msg = buf;
            return BP_ESHAPE;
        }
    }
    (void)max_batch;   // any batch works
    return BP_OK;
}

const char* bf16_last_message() { return g_msg.c_str(); }

bp_status bf16_create(const int* n, int L, int max_batch, int num_sms, float* theta, float* V,
                      float* G, Bf16Net** out) {
    if (!get_encoder()) {
        g_msg = "cuTensorMapEncodeTiled is not available from the driver";
        return BP_ECUDA;
    }
    int dev = 0;
    cudaGetDevice(&dev);
    if (setup_all(dev) != cudaSuccess) {
        g_msg = "could not set the shared-memory limit of the tensor-core kernels";
        return BP_ECUDA;
    }
    Bf16Net* b = new Bf16Net();
    b->L = L;
    for (int l = 0; l <= L; ++l) b->n[l] = n[l];
    b->cap = max_batch;
    b->num_sms = num_sms;
    b->theta = theta;
    b->V = V;
    b->G = G;
    long long pos = 0;
    for (int l = 1; l <= L; ++l) {
        b->woff[l] = pos;
        pos += (long long)n[l] * n[l - 1];
        b->boff[l] = pos;
        pos += n[l];
    }
    bool ok = true;
    const int mt = ceil_div(max_batch, BM);
    b->max_splits = dw_plan(n, L, max_batch, num_sms, kMaxSplits, false).splits;
    for (int l = 1; l <= L && ok; ++l) {
        ok = ok && alloc(b, (void**)&b->wb[l], (size_t)n[l] * n[l - 1] * 2);
        ok = ok && alloc(b, (void**)&b->act[l], (size_t)max_batch * n[l] * 2);
        ok = ok && alloc(b, (void**)&b->dlt[l], (size_t)max_batch * n[l] * 2);
        ok = ok && alloc(b, (void**)&b->gpart[l], (size_t)b->max_splits * n[l] * n[l - 1] * 4);
        ok = ok && alloc(b, (void**)&b->bpart[l], (size_t)mt * n[l] * 4);
    }
    ok = ok && alloc(b, (void**)&b->sse_part, (size_t)mt * ceil_div(n[L], 64) * 4);
    if (!ok) {
        g_msg = "cudaMalloc failed for the bfloat16 scratch buffers";
        bf16_destroy(b);
        return BP_ENOMEM;
    }
    *out = b;
    return BP_OK;
}

void bf16_destroy(Bf16Net* b) {
    if (b == nullptr) return;
    for (void* p : b->allocs) cudaFree(p);
    delete b;
}

void bf16_set_flags(Bf16Net* b, int* flags) { b->flags = flags; }
void bf16_set_guard(Bf16Net* b, float guard) { b->guard = guard; }

cudaError_t bf16_refresh_weights(Bf16Net* b, cudaStream_t s) {
    return launch_update(upd_args(b, 0, 0, 2, false, 0.f, 0.f, nullptr, 0), s);
}

cudaError_t bf16_forward(Bf16Net* b, const void* X, int batch, void* Y, cudaStream_t s) {
    // One layer: tiles still read rows of X that others have written to Y, so a Y that overlaps
    // X is copied to at the end.  (With more layers X is read before the last one writes.)
    const size_t nx = (size_t)batch * b->n[0] * sizeof(bf16), ny = (size_t)batch * b->n[b->L] * sizeof(bf16);
    const uintptr_t x = (uintptr_t)X, y = (uintptr_t)Y;
    if (b->L > 1 || Y == nullptr || y + ny <= x || x + nx <= y)
        return run_forward(b, (const bf16*)X, batch, nullptr, (bf16*)Y, s);
    const cudaError_t e = run_forward(b, (const bf16*)X, batch, nullptr, nullptr, s);
    return e != cudaSuccess ? e : cudaMemcpyAsync(Y, b->act[b->L], ny, cudaMemcpyDeviceToDevice, s);
}

cudaError_t bf16_backward(Bf16Net* b, const void* X, const void* T, int batch, float* sse,
                          bool /*g_dirty*/, cudaStream_t s) {
    const int L = b->L;
    const int nL = b->n[L];
    const int nc = ceil_div(nL, 64), mt = ceil_div(batch, BM);
    cudaError_t e = launch_pdl(k_output_delta, nc, mt, 256, 0, s, b->act[L], (const bf16*)T, batch, nL, b->dlt[L],
                               b->bpart[L], b->sse_part);
    if (e != cudaSuccess) return e;
    const DwPlan p = dw_plan(b->n, L, batch, b->num_sms, b->max_splits, false);
    e = run_backward(b, (const bf16*)X, batch, p, nullptr, s);
    if (e != cudaSuccess) return e;
    return launch_update(upd_args(b, p.splits, mt, 1, false, 0.f, 0.f, sse, mt * nc), s);
}

cudaError_t bf16_update(Bf16Net* b, float lr, float momentum, float grad_scale, cudaStream_t s) {
    // apply G only: no partial changes pending
    return launch_update(upd_args(b, 0, 0, 0, true, lr * grad_scale, momentum, nullptr, 0), s);
}

cudaError_t bf16_train(Bf16Net* b, const void* X, const void* T, int n_patterns, int minibatch,
                       float* sse, float lr, float momentum, float grad_scale, bool g_dirty,
                       cudaStream_t s) {
    const int L = b->L;
    const size_t xrow = (size_t)b->n[0], trow = (size_t)b->n[L];
    bool fold = g_dirty;
    for (long long p0 = 0, step = 0; p0 < n_patterns; p0 += minibatch, ++step) {
        const int B = (int)((n_patterns - p0) < minibatch ? (n_patterns - p0) : minibatch);
        const bf16* Xs = (const bf16*)X + p0 * xrow;
        const bf16* Ts = (const bf16*)T + p0 * trow;
        cudaError_t e = run_forward(b, Xs, B, Ts, nullptr, s);
        if (e != cudaSuccess) return e;
        const DwPlan p = dw_plan(b->n, L, B, b->num_sms, b->max_splits, true);
        const int n_sse = tiles_of(B, b->n[L], pick_bn(B, b->n[L], ceil_div(b->n[L - 1], BK), b->num_sms));
        const UpdArgs a = upd_args(b, p.fused ? 0 : p.splits, ceil_div(B, BM), 0, fold, lr * grad_scale, momentum,
                                   sse != nullptr ? sse + step : nullptr, n_sse);
        e = run_backward(b, Xs, B, p, p.fused ? &a : nullptr, s);
        if (e == cudaSuccess && !p.fused) e = launch_update(a, s);
        if (e != cudaSuccess) return e;
        fold = false;
    }
    return cudaSuccess;
}

}  // namespace bp
