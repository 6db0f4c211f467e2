// Learned surrogate of the RVE homogenisation (no counterpart in the paper).
//
// An ensemble of MLPs maps 8 features of a macro Gauss point to the 33
// Cholesky-factor entries of its normalised C (21), K (6) and D (6):
//   h_{l+1} = silu(h_l W_l + b_l), l = 0..3 (width 256), z = h_4 W_4 + b_4,
//   L = tril(z) with softplus on the diagonal, tensor = L L^T (always SPD).
// Weights and activations are BF16, every product accumulates in FP32 on the
// 5th-generation tensor cores (tcgen05.mma kind::f16, accumulator in tensor
// memory), master weights and Adam moments are FP32.
//
// GEMM convention: C[M][N] = A[M][K] * B, with A row-major and B supplied as
// Bt[N][K] row-major (K contiguous in both), M a multiple of 64, N 64 or a
// multiple of 128, K a multiple of 64.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>

#include "kernels.h"
#include "surrogate.h"

namespace rve {

namespace {

__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 lo, __nv_bfloat16 hi) {
    return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// a sigmoid(a) with the fast reciprocal division (a / inf -> 0 for very negative a)
__device__ __forceinline__ float silu_f(float a) { return __fdividef(a, 1.f + __expf(-a)); }
__device__ __forceinline__ float dsilu_f(float a) {
    const float s = 1.f / (1.f + __expf(-a));
    return s * (1.f + a * (1.f - s));
}

}  // namespace

// ------------------------------------------------ tcgen05 GEMM (sm_103a)
// C tile [128 rows x NT] = A [128 x K] * Bt [NT x K]^T on the 5th-generation tensor
// cores: BF16 operands staged by cp.async into 128-byte-swizzled K-major shared
// memory tiles (64 K values = 128 bytes per row), two K stages in flight, one
// thread issuing kind::f16 MMAs (M = 128, N = NT, K = 16) into an FP32 TMEM
// accumulator, thread t reading back row t for the epilogue.  Rows past M are
// zero-filled on load and not stored.
namespace {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint64_t gl_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool bar_try(uint32_t a, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait (1 s of the global timer, or a poll cap should the timer not advance)
__device__ __forceinline__ bool bar_wait(uint32_t a, uint32_t parity) {
    if (bar_try(a, parity)) return true;
    const uint64_t t0 = gl_ns();
    for (int i = 0; i < (1 << 26); ++i) {
        if (bar_try(a, parity)) return true;
        if (gl_ns() - t0 > 1000000000ull) return false;
    }
    return false;
}
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
    return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
__device__ __forceinline__ void mma_f16_tmem(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void tmem_ld16x(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

// set when a bounded wait of the GEMM gave up: a word of pinned host memory, which the host
// reads after any synchronisation without a copy of its own
__device__ int* g_gemm_timeout;
__device__ __forceinline__ void gemm_gave_up() { *(volatile int*)g_gemm_timeout = 1; }

}  // namespace

// epilogue: 0 = store FP32 only, 1 = bias + silu -> BF16 (pre-activation to Cf if non-null),
//           2 = bias, FP32 out,
//           4 = bias, FP32 out transposed (Cf[col * M + row]),
//           5 = times silu'(pre) -> BF16 (the backward pass through an activation)
//
// One launch runs up to GEMM_GROUP problems of the same N and K (the members of an
// ensemble; blockIdx.y is the problem), each with its own operands, outputs and M.  A
// training step's problems are a few tiles each, so a launch of one is bound by its own
// latency: grouped, an epoch of 64 steps of four members takes 4.0 ms instead of 20.6 ms
// (4 096 points in batches of 256).
//
// Persistent and warp-specialised: each CTA walks the output tiles
// blockIdx.x, blockIdx.x + gridDim.x, ... (the N tiles of one row block are
// neighbours, so the A rows are read from L2 once per row block).
//   warp 0   TMA producer: K steps of 64 values of A and Bt into a ring of
//            GemmShape::S stages (128-byte swizzle; rows past M zero-filled by the
//            tensor map's bounds), each stage a "full" barrier counting its bytes;
//   warp 1   MMA issuer: kind::f16 MMAs into one of two FP32 TMEM accumulators,
//            releasing each stage through an "empty" barrier and each finished
//            tile through "tmem full";
//   warps 2.. epilogue (NT / 8 of them): a warp reads 32 rows (its TMEM lane
//            quarter) x 32 columns of the finished accumulator, hands it back through
//            "tmem empty" and runs bias / SiLU / conversion and the stores while
//            the MMAs of the next tile fill the other accumulator.
// Every wait is bounded; a role that gives up sets *g_gemm_timeout and leaves its
// loop, after which the producer waits for its copies in flight and the MMA
// issuer for its MMAs, so the tensor memory is idle when it is freed.
template <int NT>
struct GemmShape {
    static constexpr int S = NT == 128 ? 6 : 8;
    static constexpr int A_BYTES = 128 * 128, B_BYTES = NT * 128, STAGE = A_BYTES + B_BYTES;
    // epilogue warps: four lane quarters x column groups of 32
    static constexpr int EPI_WARPS = 4 * (NT / 32), THREADS = 64 + 32 * EPI_WARPS;
    static constexpr int NBAR = 2 * S + 5;
    // bias vector staged in shared memory (N <= BIAS_MAX) behind the barriers
    static constexpr int BIAS_OFF = ((8 * NBAR + 16 + 15) / 16) * 16, BIAS_MAX = 256;
};

struct GemmGroup {
    CUtensorMap a[GEMM_GROUP], b[GEMM_GROUP];
    GemmProblem p[GEMM_GROUP];
    uint32_t stage_tx[GEMM_GROUP];
};

template <int NT>
__global__ void __launch_bounds__(GemmShape<NT>::THREADS, 1)
    k_gemm_tc(const __grid_constant__ GemmGroup P, int N, int K, int epilogue) {
    using G = GemmShape<NT>;
    const int prob = blockIdx.y;
    const CUtensorMap& tmA = P.a[prob];
    const CUtensorMap& tmB = P.b[prob];
    const int M = P.p[prob].M;
    const uint32_t stage_tx = P.stage_tx[prob];
    const float* __restrict__ bias = P.p[prob].bias;
    const float* __restrict__ pre = P.p[prob].pre;
    __nv_bfloat16* __restrict__ Cb = P.p[prob].Cb;
    float* __restrict__ Cf = P.p[prob].Cf;
    constexpr int S = G::S;
    extern __shared__ uint8_t gsm_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(gsm_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(base + S * G::STAGE);
    uint64_t* empty = full + S;
    uint64_t* tfull = empty + S;    // [2]
    uint64_t* tempty = tfull + 2;   // [2]
    uint64_t* done = tempty + 2;
    uint32_t* tslot = reinterpret_cast<uint32_t*>(done + 1);
    float* sbias = reinterpret_cast<float*>(base + S * G::STAGE + G::BIAS_OFF);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int KB = K / 64, n_tn = N / NT, n_tiles = ((M + 127) / 128) * n_tn;
    const bool bias_smem = bias != nullptr && (epilogue == 1 || epilogue == 2 || epilogue == 4) && N <= G::BIAS_MAX;
    if (bias_smem)
        for (int i = t; i < N; i += blockDim.x) sbias[i] = __ldg(bias + i);
    if (t == 0) {
        for (int k = 0; k < G::NBAR; ++k) {
            const uint32_t cnt = (k == 2 * S + 2 || k == 2 * S + 3) ? (uint32_t)G::EPI_WARPS : 1u;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(full + k)), "r"(cnt) : "memory");
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                     "r"((uint32_t)(2 * NT))
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer
            int it = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
                const int m0 = (tile / n_tn) * 128, n0 = (tile % n_tn) * NT;
                for (int kb = 0; kb < KB; ++kb, ++it) {
                    const int s = it % S;
                    if (it >= S && !bar_wait(smem_addr(empty + s), ((it / S) & 1) ^ 1)) {
                        ok = false;
                        break;
                    }
                    const uint32_t sa = smem_addr(base + s * G::STAGE), sb = sa + G::A_BYTES, fb = smem_addr(full + s);
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(stage_tx)
                                 : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                        "%3}], [%4];" ::"r"(sa),
                        "l"(reinterpret_cast<uint64_t>(&tmA)), "r"(kb * 64), "r"(m0), "r"(fb)
                        : "memory");
                    asm volatile(
                        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
                        "%3}], [%4];" ::"r"(sb),
                        "l"(reinterpret_cast<uint64_t>(&tmB)), "r"(kb * 64), "r"(n0), "r"(fb)
                        : "memory");
                }
            }
            if (!ok) gemm_gave_up();
            // the copies of the last min(S, it) steps may still be in flight
            for (int k = it - 1; k >= 0 && k >= it - S; --k)
                if (!bar_wait(smem_addr(full + k % S), (k / S) & 1)) gemm_gave_up();
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer: kind::f16, D FP32, A and B BF16, both K-major, N = NT, M = 128
            const uint32_t idesc =
                (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NT >> 3) << 17) | ((128u >> 4) << 24);
            int it = 0, i = 0;
            bool ok = true;
            for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x, ++i) {
                const int acc = i & 1;
                if (i >= 2 && !bar_wait(smem_addr(tempty + acc), ((i >> 1) & 1) ^ 1)) {
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d = tmem + (uint32_t)(acc * NT);
                for (int kb = 0; kb < KB; ++kb, ++it) {
                    const int s = it % S;
                    if (!bar_wait(smem_addr(full + s), (it / S) & 1)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t sa = smem_addr(base + s * G::STAGE), sb = sa + G::A_BYTES;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk)
                        mma_f16_tmem(d, desc_sw128(sa + kk * 32), desc_sw128(sb + kk * 32), idesc,
                                     (kb > 0 || kk > 0) ? 1u : 0u);
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                            smem_addr(empty + s))
                        : "memory");
                }
                if (ok)
                    asm volatile(
                        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                            smem_addr(tfull + acc))
                        : "memory");
            }
            if (!ok) gemm_gave_up();
            // every MMA issued has completed once this commit arrives
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             smem_addr(done))
                         : "memory");
            if (!bar_wait(smem_addr(done), 0)) gemm_gave_up();
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, column group (w - 2) / 4
        const int q = warp & 3, h = (warp - 2) >> 2;
        constexpr int HC = 32;
        int i = 0;
        for (int tile = blockIdx.x; tile < n_tiles; tile += gridDim.x, ++i) {
            __syncwarp();
            const int acc = i & 1;
            const int m0 = (tile / n_tn) * 128, n0 = (tile % n_tn) * NT;
            bool w = true;
            if (lane == 0) w = bar_wait(smem_addr(tfull + acc), (i >> 1) & 1);
            w = __shfl_sync(0xffffffffu, w ? 1 : 0, 0) != 0;
            if (!w) {
                if (lane == 0) gemm_gave_up();
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            uint32_t v[HC];
            const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(acc * NT + h * HC);
#pragma unroll
            for (int c = 0; c < HC; c += 16) tmem_ld16x(ta + c, *reinterpret_cast<uint32_t(*)[16]>(v + c));
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(tempty + acc)) : "memory");
            const int row = m0 + 32 * q + lane;
            if (row >= M) continue;   // (rows past M hold the zero fill or, for M < 128, stale data)
            const int col0 = n0 + h * HC;
            const int64_t o = (int64_t)row * N + col0;
#pragma unroll
            for (int c = 0; c < HC; c += 16) {
                float f[16];
#pragma unroll
                for (int u = 0; u < 16; ++u) f[u] = __uint_as_float(v[c + u]);
                if (bias_smem) {
#pragma unroll
                    for (int u = 0; u < 16; u += 4) {
                        const float4 b4 = *reinterpret_cast<const float4*>(sbias + col0 + c + u);
                        f[u] += b4.x;
                        f[u + 1] += b4.y;
                        f[u + 2] += b4.z;
                        f[u + 3] += b4.w;
                    }
                } else if (bias && epilogue != 0) {
#pragma unroll
                    for (int u = 0; u < 16; u += 4) {
                        const float4 b4 = __ldg(reinterpret_cast<const float4*>(bias + col0 + c + u));
                        f[u] += b4.x;
                        f[u + 1] += b4.y;
                        f[u + 2] += b4.z;
                        f[u + 3] += b4.w;
                    }
                }
                if (epilogue == 4) {   // bias, FP32, transposed: Cf[col][row] (rows adjacent across lanes)
#pragma unroll
                    for (int u = 0; u < 16; ++u) Cf[(int64_t)(col0 + c + u) * M + row] = f[u];
                    continue;
                }
                if (epilogue == 5) {
#pragma unroll
                    for (int u = 0; u < 16; u += 4) {
                        const float4 z4 = __ldg(reinterpret_cast<const float4*>(pre + o + c + u));
                        f[u] *= dsilu_f(z4.x);
                        f[u + 1] *= dsilu_f(z4.y);
                        f[u + 2] *= dsilu_f(z4.z);
                        f[u + 3] *= dsilu_f(z4.w);
                    }
                    uint32_t pk[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        pk[u] = pack_bf16(__float2bfloat16(f[2 * u]), __float2bfloat16(f[2 * u + 1]));
                    *reinterpret_cast<uint4*>(Cb + o + c) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(Cb + o + c + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                } else if (epilogue == 1) {
                    if (Cf)
#pragma unroll
                        for (int u = 0; u < 16; u += 4)
                            *reinterpret_cast<float4*>(Cf + o + c + u) = make_float4(f[u], f[u + 1], f[u + 2], f[u + 3]);
                    uint32_t pk[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        pk[u] = pack_bf16(__float2bfloat16(silu_f(f[2 * u])), __float2bfloat16(silu_f(f[2 * u + 1])));
                    *reinterpret_cast<uint4*>(Cb + o + c) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(Cb + o + c + 8) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                } else {
#pragma unroll
                    for (int u = 0; u < 16; u += 4)
                        *reinterpret_cast<float4*>(Cf + o + c + u) = make_float4(f[u], f[u + 1], f[u + 2], f[u + 3]);
                }
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)(2 * NT))
                     : "memory");
    }
}

// ------------------------------------------- fused ensemble inference (sm_103a)
// The whole network of up to MLP_MAXM members for 128-row tiles of features, with
// the activations kept in shared memory between the layers (only the features come
// in and the last layer's z goes out).  Per layer: kind::f16 MMAs (M = 128, N = 256
// or 64, K = 16) from the activation tile (A: 128-byte-swizzled K-major chunks of 64
// values, written by the epilogue in that layout) and a weight chunk W^T [N][64] (B,
// streamed by TMA through a two-stage ring from L2) into an FP32 accumulator of 256
// tensor-memory columns; the epilogue adds the bias, applies SiLU and writes the BF16
// activations back over the tile it came from (its layer's MMAs have completed), or,
// after the last layer, stores z transposed (zT[member][col][row]) for the head.
//
// Work items are (tile, member) pairs, walked persistently.  Two items are in flight
// per CTA, one per slot (own feature tile, activation tile and accumulator): the MMA
// warp alternates between the slots layer by layer, so that one slot's MMAs run while
// the other slot's epilogue works.  Warp 0 issues the TMA copies in the MMA's order,
// warp 1 the MMAs, and epilogue warps 2-9 serve slot 0 and 10-17 slot 1 (lane quarter
// w % 4, 128-column half).  Every wait is bounded.
constexpr int MLP_MAXM = 4, MLP_EPI = 16, MLP_THREADS = 64 + 32 * MLP_EPI;
constexpr int MLP_NL = 5;
constexpr int MLP_OFF_ACT = 0,        // [2][64 KB]
    MLP_OFF_X = 131072,               // [2][16 KB]
    MLP_OFF_W = 163840,               // [2][32 KB]
    MLP_OFF_BAR = 229376, MLP_SMEM = 1024 + MLP_OFF_BAR + 128;

struct MlpParams {
    CUtensorMap x;                       // features [M][64] BF16, box {64, x_rows}
    CUtensorMap w[MLP_MAXM][MLP_NL];     // member e, layer l: W^T [N_l][K_l] BF16, box {64, N_l}
    const float* bias[MLP_MAXM][MLP_NL];
    float* zT;                           // [members][64][ldz]
    int M, ldz, members;
    uint32_t x_tx;                       // bytes of one feature tile (x_rows x 128)
};

__device__ __forceinline__ int mlp_k(int l) { return l == 0 ? 64 : 256; }
__device__ __forceinline__ int mlp_n(int l) { return l == 4 ? 64 : 256; }

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__global__ void __launch_bounds__(MLP_THREADS, 1) k_mlp_fused(const __grid_constant__ MlpParams P) {
    extern __shared__ uint8_t msm_raw[];
    uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(msm_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(base + MLP_OFF_BAR);
    // per slot s: xfull[s], xempty[s], accfull[s], epidone[s]; the ring's wfull[2], wempty[2]; done
    auto B = [&](int k) { return smem_addr(bars + k); };
    const uint32_t b_xfull = B(0), b_xempty = B(2), b_acc = B(4), b_epi = B(6), b_wfull = B(8), b_wempty = B(10),
                   b_done = B(12);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 13);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int n_items = ((P.M + 127) / 128) * P.members;
    // this CTA's items k = 0 .. n_cta - 1 are blockIdx.x + k gridDim.x; slot s takes k = s (mod 2)
    const int n_cta = blockIdx.x < n_items ? (n_items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int ns0 = (n_cta + 1) / 2, ns1 = n_cta / 2;
    if (t == 0) {
        for (int k = 0; k < 13; ++k)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bars + k)),
                         "r"((k == 6 || k == 7) ? (uint32_t)(MLP_EPI / 2) : 1u)
                         : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                     "r"(512u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tslot;
    const uint32_t s_act = smem_addr(base + MLP_OFF_ACT), s_x = smem_addr(base + MLP_OFF_X),
                   s_w = smem_addr(base + MLP_OFF_W);

    if (warp == 0) {
        if (lane == 0) {
            // ---- TMA producer, in the MMA's order: round r gives slot 0, then slot 1,
            // layer r % 5 of its item r / 5; a layer-0 step also loads the item's features
            int wit = 0;
            bool ok = true;
            for (int r = 0; ok && r / 5 < ns0; ++r)
                for (int sl = 0; sl < 2 && ok; ++sl) {
                    const int idx = r / 5, l = r % 5;
                    if (idx >= (sl ? ns1 : ns0)) continue;
                    const int item = blockIdx.x + (2 * idx + sl) * gridDim.x;
                    const int tile = item / P.members, e = item % P.members;
                    if (l == 0) {
                        if (idx >= 1 && !bar_wait(b_xempty + 8 * sl, (idx - 1) & 1)) {
                            ok = false;
                            break;
                        }
                        bar_expect(b_xfull + 8 * sl, P.x_tx);
                        tma_2d(s_x + sl * 16384, &P.x, 0, tile * 128, b_xfull + 8 * sl);
                    }
                    for (int kc = 0; kc < mlp_k(l) / 64; ++kc, ++wit) {
                        const int st = wit & 1;
                        if (wit >= 2 && !bar_wait(b_wempty + 8 * st, ((wit >> 1) & 1) ^ 1)) {
                            ok = false;
                            break;
                        }
                        bar_expect(b_wfull + 8 * st, (uint32_t)mlp_n(l) * 128u);
                        tma_2d(s_w + st * 32768, &P.w[e][l], kc * 64, 0, b_wfull + 8 * st);
                    }
                }
            if (!ok) gemm_gave_up();
            // copies that may still be in flight: each slot's last feature tile and the
            // last weight chunks
            for (int sl = 0; sl < 2; ++sl) {
                const int n = sl ? ns1 : ns0;
                if (n >= 1 && !bar_wait(b_xfull + 8 * sl, (n - 1) & 1)) gemm_gave_up();
            }
            for (int k = wit - 1; k >= 0 && k >= wit - 2; --k)
                if (!bar_wait(b_wfull + 8 * (k & 1), (k >> 1) & 1)) gemm_gave_up();
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // ---- MMA issuer: the same round order as the producer.  A slot's step waits
            // for the epilogue of the slot's previous step, which both freed the slot's
            // accumulator and wrote this step's input activations.
            int wit = 0, ks[2] = {0, 0};
            bool ok = true;
            for (int r = 0; ok && r / 5 < ns0; ++r)
                for (int sl = 0; sl < 2 && ok; ++sl) {
                    const int idx = r / 5, l = r % 5;
                    if (idx >= (sl ? ns1 : ns0)) continue;
                    if (l == 0 && !bar_wait(b_xfull + 8 * sl, idx & 1)) {
                        ok = false;
                        break;
                    }
                    if (ks[sl] >= 1 && !bar_wait(b_epi + 8 * sl, (ks[sl] - 1) & 1)) {
                        ok = false;
                        break;
                    }
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    const uint32_t a_base = l == 0 ? s_x + sl * 16384 : s_act + sl * 65536;
                    const uint32_t d = tmem + (uint32_t)(256 * sl);
                    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                                           ((uint32_t)(mlp_n(l) >> 3) << 17) | ((128u >> 4) << 24);
                    for (int kc = 0; kc < mlp_k(l) / 64; ++kc, ++wit) {
                        const int st = wit & 1;
                        if (!bar_wait(b_wfull + 8 * st, (wit >> 1) & 1)) {
                            ok = false;
                            break;
                        }
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint32_t a = a_base + kc * 16384, b = s_w + st * 32768;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)
                            mma_f16_tmem(d, desc_sw128(a + kk * 32), desc_sw128(b + kk * 32), idesc,
                                         (kc > 0 || kk > 0) ? 1u : 0u);
                        mma_commit(b_wempty + 8 * st);
                    }
                    if (!ok) break;
                    if (l == 0) mma_commit(b_xempty + 8 * sl);
                    mma_commit(b_acc + 8 * sl);
                    ++ks[sl];
                }
            if (!ok) gemm_gave_up();
            // every MMA issued has completed once this commit arrives
            mma_commit(b_done);
            if (!bar_wait(b_done, 0)) gemm_gave_up();
        }
    } else {
        // ---- epilogue: warps 2-9 serve slot 0, 10-17 slot 1; lane quarter q, column half h
        const int sl = (warp - 2) >> 3, q = warp & 3, h = ((warp - 2) >> 2) & 1;
        const int r = 32 * q + lane;
        const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(256 * sl);
        uint8_t* act = base + MLP_OFF_ACT + sl * 65536;
        const int n_slot = sl ? ns1 : ns0;
        int ks = 0;
        bool ok = true;
        for (int idx = 0; idx < n_slot && ok; ++idx) {
            const int item = blockIdx.x + (2 * idx + sl) * gridDim.x;
            const int tile = item / P.members, e = item % P.members;
            const int grow = tile * 128 + r;
            for (int l = 0; l < MLP_NL; ++l, ++ks) {
                __syncwarp();
                bool w = true;
                if (lane == 0) w = bar_wait(b_acc + 8 * sl, ks & 1);
                w = __shfl_sync(0xffffffffu, w ? 1 : 0, 0) != 0;
                if (!w) {
                    if (lane == 0) gemm_gave_up();
                    ok = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const float* bias = P.bias[e][l];
                if (l < MLP_NL - 1) {
                    // columns 128 h + 64 j .. + 63: activation chunk 2 h + j
#pragma unroll 1
                    for (int j = 0; j < 2; ++j) {
                        const int c0 = 128 * h + 64 * j;
                        uint32_t v[64];
#pragma unroll
                        for (int jj = 0; jj < 4; ++jj)
                            tmem_ld16x(lane_base + (uint32_t)(c0 + 16 * jj),
                                       *reinterpret_cast<uint32_t(*)[16]>(v + 16 * jj));
                        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                        uint8_t* out = act + (c0 / 64) * 16384 + r * 128;
#pragma unroll
                        for (int u = 0; u < 8; ++u) {
                            const float4 b0 = __ldg(reinterpret_cast<const float4*>(bias + c0 + 8 * u));
                            const float4 b1 = __ldg(reinterpret_cast<const float4*>(bias + c0 + 8 * u + 4));
                            const float bb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
                            uint32_t pk[4];
#pragma unroll
                            for (int hh = 0; hh < 4; ++hh)
                                pk[hh] = pack_bf16(
                                    __float2bfloat16(silu_f(__uint_as_float(v[8 * u + 2 * hh]) + bb[2 * hh])),
                                    __float2bfloat16(silu_f(__uint_as_float(v[8 * u + 2 * hh + 1]) + bb[2 * hh + 1])));
                            // 128-byte swizzle of the K-major operand layout: 16-byte unit u of row r
                            *reinterpret_cast<uint4*>(out + ((u ^ (r & 7)) << 4)) =
                                make_uint4(pk[0], pk[1], pk[2], pk[3]);
                        }
                    }
                    // the next layer's MMAs read these writes through the async proxy
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                } else {
                    // N = 64: columns 32 h .. + 31
                    uint32_t v[32];
                    tmem_ld16x(lane_base + (uint32_t)(32 * h), *reinterpret_cast<uint32_t(*)[16]>(v));
                    tmem_ld16x(lane_base + (uint32_t)(32 * h + 16), *reinterpret_cast<uint32_t(*)[16]>(v + 16));
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    if (grow < P.M) {
                        float* zt = P.zT + ((int64_t)e * 64 + 32 * h) * P.ldz + grow;
#pragma unroll
                        for (int u = 0; u < 32; ++u)
                            zt[(int64_t)u * P.ldz] = __uint_as_float(v[u]) + __ldg(bias + 32 * h + u);
                    }
                }
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0)
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(b_epi + 8 * sl) : "memory");
            }
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
    }
}

template <int NT>
static size_t gemm_smem() {
    return 1024 + (size_t)GemmShape<NT>::S * GemmShape<NT>::STAGE + GemmShape<NT>::BIAS_OFF +
           4 * GemmShape<NT>::BIAS_MAX;
}

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link to the driver library)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
    static EncodeTiledFn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    });
    return fn;
}

// 2-D BF16 row-major matrix [rows][cols] (cols contiguous), box of 64 columns x box_rows
// rows with the 128-byte swizzle; rows past `rows` read as zero
static bool make_map(CUtensorMap* m, const __nv_bfloat16* base, int rows, int cols, int box_rows) {
    EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {(cuuint64_t)cols * sizeof(__nv_bfloat16)};
    const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
    const cuuint32_t estr[2] = {1u, 1u};
    return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<__nv_bfloat16*>(base), dims, strides, box, estr,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

namespace {
std::atomic<int*> g_timeout_host{nullptr};   // the word g_gemm_timeout points to
}

cudaError_t gemm_tc_prepare() {
    static std::mutex mu;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!g_timeout_host.load()) {
            void* w = nullptr;
            const cudaError_t e = cudaHostAlloc(&w, 64, cudaHostAllocPortable | cudaHostAllocMapped);
            if (e != cudaSuccess) return e;
            *static_cast<int*>(w) = 0;
            g_timeout_host.store(static_cast<int*>(w));
        }
    }
    void* d = nullptr;   // (each device keeps its own pointer to the one word)
    cudaError_t e = cudaHostGetDevicePointer(&d, g_timeout_host.load(), 0);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_gemm_timeout, &d, sizeof(d));
    if (e != cudaSuccess) return e;
    cudaFuncSetAttribute(k_gemm_tc<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<128>());
    cudaFuncSetAttribute(k_gemm_tc<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem<64>());
    cudaFuncSetAttribute(k_mlp_fused, cudaFuncAttributeMaxDynamicSharedMemorySize, MLP_SMEM);
    return cudaSuccess;
}

int mlp_fused_max_members() { return MLP_MAXM; }

// The fused inference of `members` networks on M feature rows (M a multiple of 64):
// weights of member e at wt[e] + w_off[l] (W^T [N_l][K_l] BF16), biases bias[e * 5 + l].
cudaError_t launch_mlp_fused(int M, int members, const __nv_bfloat16* X, const __nv_bfloat16* const* wt,
                             const int64_t* w_off, const float* const* bias, float* zT, int ldz, cudaStream_t s) {
    if (M <= 0 || M % 64 || members < 1 || members > MLP_MAXM || ldz < M) return cudaErrorInvalidValue;
    static const int KL[MLP_NL] = {64, 256, 256, 256, 256}, NL[MLP_NL] = {256, 256, 256, 256, 64};
    MlpParams P;
    std::memset(&P, 0, sizeof(P));
    const int x_rows = M < 128 ? M : 128;
    if (!make_map(&P.x, X, M, 64, x_rows)) return cudaErrorInvalidValue;
    for (int e = 0; e < members; ++e)
        for (int l = 0; l < MLP_NL; ++l) {
            if (!make_map(&P.w[e][l], wt[e] + w_off[l], NL[l], KL[l], NL[l])) return cudaErrorInvalidValue;
            P.bias[e][l] = bias[e * MLP_NL + l];
        }
    P.zT = zT;
    P.M = M;
    P.ldz = ldz;
    P.members = members;
    P.x_tx = (uint32_t)x_rows * 128u;
    const int items = ((M + 127) / 128) * members;
    const int grid = std::min(items, sm_count());
    k_mlp_fused<<<grid, MLP_THREADS, MLP_SMEM, s>>>(P);
    return cudaGetLastError();
}

int gemm_tc_timed_out() {
    const int* w = g_timeout_host.load();
    return w ? *const_cast<const volatile int*>(w) : 0;
}

int gemm_tc_set_timed_out(int v) {
    int* w = g_timeout_host.load();
    if (!w) return -1;
    const int old = *const_cast<volatile int*>(w);
    *const_cast<volatile int*>(w) = v;
    return old;
}

// M a multiple of 64 (rows past a 128-row tile are zero-filled), N 64 or a multiple of
// 128, K a multiple of 64; A and Bt 16-byte aligned.  At most one CTA per tile and SM,
// two accumulators of NT TMEM columns each.
cudaError_t launch_gemm_group(int count, const GemmProblem* probs, int N, int K, int epilogue, cudaStream_t s) {
    const int NT = N == 64 ? 64 : 128;
    if (count < 1 || count > GEMM_GROUP || K <= 0 || K % 64 || (N != 64 && N % 128)) return cudaErrorInvalidValue;
    GemmGroup P;
    std::memset(static_cast<void*>(&P), 0, sizeof(P));
    int tiles = 0;
    for (int i = 0; i < count; ++i) {
        const int M = probs[i].M;
        if (M <= 0 || M % 64) return cudaErrorInvalidValue;
        // with M = 64 the A box is 64 rows and the MMA's rows 64..127 are never stored
        const int a_rows = M < 128 ? M : 128;
        if (!make_map(&P.a[i], probs[i].A, M, K, a_rows) || !make_map(&P.b[i], probs[i].Bt, N, K, NT))
            return cudaErrorInvalidValue;
        P.p[i] = probs[i];
        P.stage_tx[i] = (uint32_t)(a_rows + NT) * 128u;
        tiles = std::max(tiles, (N / NT) * ((M + 127) / 128));
    }
    const dim3 grid(std::min(tiles, std::max(1, sm_count() / count)), count);
    if (NT == 64)
        k_gemm_tc<64><<<grid, GemmShape<64>::THREADS, gemm_smem<64>(), s>>>(P, N, K, epilogue);
    else
        k_gemm_tc<128><<<grid, GemmShape<128>::THREADS, gemm_smem<128>(), s>>>(P, N, K, epilogue);
    return cudaGetLastError();
}

cudaError_t launch_gemm_bf16(int M, int N, int K, const __nv_bfloat16* A, const __nv_bfloat16* Bt,
                             const float* bias, int epilogue, __nv_bfloat16* Cb, float* Cf, cudaStream_t s) {
    GemmProblem p;
    p.A = A;
    p.Bt = Bt;
    p.bias = bias;
    p.Cb = Cb;
    p.Cf = Cf;
    p.M = M;
    return launch_gemm_group(1, &p, N, K, epilogue, s);
}

// Sum of a double over the block's 256 threads (every thread gets it), in a fixed order.
__device__ __forceinline__ double block_sum_256(double v, double* buf) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += buf[k];
    __syncthreads();
    return t;
}

// Adds one step's partial sums (part [n], non-negative, one per warp of k_head_loss) to the
// FP32 running sum *loss of an epoch.  Added one by one, each is rounded to the last place of
// the sum, and the sum depends on their order only where it passes a power of two: which
// of them come before, at the finer rounding, and which after.  Here every one takes part in
// each binade by the share of the step that falls into it, which is the mean over all orders:
// the same in every run, where atomic additions in the order the blocks finish scatter
// by 1e-7 around it.  One pass over the partial sums per binade, 1.7 a step.
__device__ __forceinline__ void add_step_loss(const float* __restrict__ part, int n, float* loss) {
    __shared__ double buf[8];
    double v = 0.0;
    for (int i = threadIdx.x; i < n; i += 256) v += (double)part[i];
    const double total = block_sum_256(v, buf);
    double s = (double)*loss, rest = 1.0;
    if (isfinite(total) && isfinite(s) && total > 0.0) {
        if (s == 0.0) {   // the first of n equal shares is exact
            s = total / n;
            rest = 1.0 - 1.0 / n;
        }
        for (;;) {
            const float at = (float)s;
            v = 0.0;
            for (int i = threadIdx.x; i < n; i += 256) v += (double)((at + part[i]) - at);
            const double r = block_sum_256(v, buf), top = at > 0.f ? ldexp(1.0, ilogbf(at) + 1) : 0.0;
            if (!(top > s) || !isfinite(r) || s + rest * r <= top) {
                s += rest * (isfinite(r) ? r : total);
                break;
            }
            rest -= (top - s) / r;
            s = top;
        }
    } else {
        s += total;
    }
    __syncthreads();
    if (threadIdx.x == 0) *loss = (float)s;
}

// One of the jobs in front of the weight-gradient GEMMs, per block plane z: the
// transposes of a layer's output gradient G [M][N] and input H [M][K], G's column
// sums (the bias gradient), and a member's loss.  The column sums run over the rows in
// order: the tile is staged in shared memory so that the serial FP32 sum is not a chain
// of global loads.
__global__ void __launch_bounds__(256) k_backward_prep(const __grid_constant__ PrepJobs J) {
    const PrepJob& j = J.job[blockIdx.z];
    if (j.part) {
        if (blockIdx.x == 0 && blockIdx.y == 0) add_step_loss(j.part, j.rows, j.sum);
        return;
    }
    const int bx = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    if (bx >= j.cols) return;
    if (j.out) {
        const int by = blockIdx.y * 32;
        if (by >= j.rows) return;
        __shared__ __nv_bfloat16 tile[32][33];
        for (int r = ty; r < 32; r += 8) {
            const int row = by + r, c = bx + tx;
            tile[r][tx] = (row < j.rows && c < j.cols) ? j.in[(int64_t)row * j.cols + c] : __float2bfloat16(0.f);
        }
        __syncthreads();
        for (int r = ty; r < 32; r += 8) {
            const int c = bx + r, row = by + tx;
            if (c < j.cols && row < j.rows) j.out[(int64_t)c * j.rows + row] = tile[tx][r];
        }
    } else {
        if (blockIdx.y != 0) return;
        __shared__ float st[256][33];
        float sum = 0.f;
        for (int r0 = 0; r0 < j.rows; r0 += 256) {
            const int n = min(256, j.rows - r0);
            for (int r = ty; r < n; r += 8)
                st[r][tx] = bx + tx < j.cols ? __bfloat162float(j.in[(int64_t)(r0 + r) * j.cols + bx + tx]) : 0.f;
            __syncthreads();
            if (ty == 0)
                for (int r = 0; r < n; ++r) sum += st[r][tx];
            __syncthreads();
        }
        if (ty == 0 && bx + tx < j.cols) j.sum[bx + tx] = sum;
    }
}

void launch_backward_prep(const PrepJobs& J, int count, int max_cols, int max_rows, cudaStream_t s) {
    dim3 grid((max_cols + 31) / 32, (max_rows + 31) / 32, count);
    k_backward_prep<<<grid, 256, 0, s>>>(J);
}

// Output head loss: z [M][NOUTP] (FP32), target rows [.][33] (row r takes target
// rows[r], or r without a list), sigma [33]; dz = d loss / d z (BF16, padded columns
// zero); loss partial per warp, in warp order.  blockIdx.y is the member.
__global__ void k_head_loss(int M, int noutp, const __grid_constant__ HeadArgs A, const float* __restrict__ target,
                            const float* __restrict__ sigma, const uint8_t* __restrict__ diag) {
    const float* __restrict__ z = A.z[blockIdx.y];
    const int32_t* __restrict__ rows = A.rows[blockIdx.y];
    __nv_bfloat16* __restrict__ dz = A.dz[blockIdx.y];
    float* __restrict__ part = A.part[blockIdx.y];
    float local = 0.f;
    const float inv = 1.f / ((float)M * 33.f);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)M * noutp;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int row = (int)(i / noutp), c = (int)(i % noutp);
        float g = 0.f;
        if (c < 33) {
            const int64_t src = rows ? rows[row] : row;
            const float zz = z[i];
            const float L = diag[c] ? (zz > 20.f ? zz : log1pf(__expf(zz))) : zz;
            const float r = (L - target[src * 33 + c]) / sigma[c];
            local += r * r * inv;
            g = 2.f * r / sigma[c] * inv;
            if (diag[c]) g *= 1.f / (1.f + __expf(-zz));
        }
        dz[i] = __float2bfloat16(g);
    }
    for (int o = 16; o > 0; o >>= 1) local += __shfl_down_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0) part[blockIdx.x * 8 + (threadIdx.x >> 5)] = local;
}

int head_loss_parts(int M, int noutp) { return 8 * std::min((int)(((int64_t)M * noutp + 255) / 256), 2048); }

void launch_head_loss(int members, int M, int noutp, const HeadArgs& A, const float* target, const float* sigma,
                      const uint8_t* diag, cudaStream_t s) {
    k_head_loss<<<dim3(head_loss_parts(M, noutp) / 8, members), 256, 0, s>>>(M, noutp, A, target, sigma, diag);
}

// Adam on FP32 master weights W [K][N] with gradient G given transposed [N][K]
// (dW^T from the GEMM); refreshes both BF16 layouts Wt [N][K] and Wn [K][N].  One job
// per layer and member (blockIdx.y); the bias [N] of the layer follows its weights.
__global__ void __launch_bounds__(256) k_adam(const __grid_constant__ AdamJobs J, float lr, float b1, float b2, float c1,
                                              float c2, float eps) {
    const AdamJob& j = J.job[blockIdx.y];
    const int K = j.K, N = j.N;
    const int64_t nw = (int64_t)K * N, n = nw + (j.gb ? N : 0);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool weight = i < nw;
        const int k = weight ? (int)(i / N) : 0, c = weight ? (int)(i % N) : (int)(i - nw);
        float g = weight ? (j.Gt ? j.Gt[(int64_t)c * K + k] : 0.f) : j.gb[c];
        if (c >= j.n_valid) g = 0.f;
        // the product that is rounded before the fused add is fixed: weights the gradient's,
        // biases the moment's (a free choice of the compiler would differ between builds, and
        // Adam carries a last-bit difference of a moment into the whole trajectory)
        const float m = j.m1[i], q = j.m2[i], gm = 1.f - b1, gq = __fmul_rn(1.f - b2, g);
        const float a = weight ? __fmaf_rn(b1, m, __fmul_rn(gm, g)) : __fmaf_rn(gm, g, __fmul_rn(b1, m));
        const float v = weight ? __fmaf_rn(b2, q, __fmul_rn(gq, g)) : __fmaf_rn(gq, g, __fmul_rn(b2, q));
        j.m1[i] = a;
        j.m2[i] = v;
        float w = j.W[i];
        if (c < j.n_valid) w -= lr * (a / c1) / (sqrtf(v / c2) + eps);
        j.W[i] = w;
        if (weight) {
            j.Wt[(int64_t)c * K + k] = __float2bfloat16(w);
            j.Wn[i] = __float2bfloat16(w);
        }
    }
}

void launch_adam(const AdamJobs& J, int count, float lr, int step, cudaStream_t s) {
    const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
    const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
    k_adam<<<dim3(64, count), 256, 0, s>>>(J, lr, b1, b2, c1, c2, eps);
}

// features [.][8] (FP64) -> normalised BF16 rows of width kin (padded with zeros), rows up
// to M; row r takes source row rows[r] (r without a list).  blockIdx.y is the member.
__global__ void k_features(int n, int M, int kin, const double* __restrict__ feat, const __grid_constant__ FeatureArgs A,
                           const float* __restrict__ mean, const float* __restrict__ inv_std) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (int64_t)M * kin) return;
    const int r = (int)(i / kin), c = (int)(i % kin);
    const int32_t* __restrict__ rows = A.rows[blockIdx.y];
    float v = 0.f;
    if (r < n && c < 8) v = ((float)feat[(int64_t)(rows ? rows[r] : r) * 8 + c] - mean[c]) * inv_std[c];
    A.X[blockIdx.y][i] = __float2bfloat16(v);
}

void launch_features(int members, int n, int M, int kin, const double* feat, const FeatureArgs& A, const float* mean,
                     const float* inv_std, cudaStream_t s) {
    const int64_t tot = (int64_t)M * kin;
    k_features<<<dim3((unsigned)((tot + 255) / 256), members), 256, 0, s>>>(n, M, kin, feat, A, mean, inv_std);
}

// Head and ensemble in one pass.  Per point and member the last layer's output (zT of the
// member, [noutp][ldz], so that adjacent threads touch adjacent words) gives the factor
// entries (softplus diagonals); the member tensors L L^T are formed twice from the
// factors in registers, for the mean and for the deviations from it, instead of being
// written out and read back twice (at four members 2.6 KB a point of traffic against
// 0.5 KB in and 0.45 KB out).  Head and ensemble as two kernels took 173 + 314 us for
// 300 000 points and four members, this one 170 us.  FP32 arithmetic (the network is BF16
// with FP32 accumulation).
constexpr int ENS_BLOCK = 64, ENS_LD = 55;

// entry (i, j) of L L^T, the factor stored row by row
template <int NN>
__device__ __forceinline__ float llt(const float* L, int i, int j) {
    float acc = 0.f;
#pragma unroll
    for (int q = 0; q < NN; ++q)
        if (q <= (i < j ? i : j)) acc = fmaf(L[i * (i + 1) / 2 + q], L[j * (j + 1) / 2 + q], acc);
    return acc;
}

// One tensor (size NN, factor entries from OFF on): the mean over the members into the
// block's staging row from OO on, and the largest relative member deviation
// max_e ||T_e - mean|| / ||mean||.
template <int NN, int OFF, int OO, int MM>
__device__ __forceinline__ float ensemble_tensor(int r, int ldz, int members, const float* __restrict__ z,
                                                 int64_t zstride, const uint8_t* __restrict__ diag,
                                                 double* __restrict__ stage) {
    constexpr int NF = NN * (NN + 1) / 2;
    float L[MM][NF];
#pragma unroll
    for (int e = 0; e < MM; ++e)
        if (e < members)
#pragma unroll
            for (int c = 0; c < NF; ++c) {
                const float zz = __ldg(z + e * zstride + (int64_t)(OFF + c) * ldz + r);
                L[e][c] = diag[OFF + c] ? (zz > 20.f ? zz : log1pf(expf(zz))) : zz;
            }
    const float inv = 1.f / (float)members;
    float mean[NN * NN], den = 0.f;
#pragma unroll
    for (int i = 0; i < NN; ++i)
#pragma unroll
        for (int j = 0; j < NN; ++j) {
            float sacc = 0.f;
#pragma unroll
            for (int e = 0; e < MM; ++e)
                if (e < members) sacc += llt<NN>(L[e], i, j);
            mean[i * NN + j] = __fmul_rn(sacc, inv);
            stage[OO + i * NN + j] = (double)mean[i * NN + j];
        }
#pragma unroll
    for (int c = 0; c < NN * NN; ++c) den = fmaf(mean[c], mean[c], den);
    float worst = 0.f;
#pragma unroll
    for (int e = 0; e < MM; ++e)
        if (e < members) {
            float num = 0.f;
#pragma unroll
            for (int i = 0; i < NN; ++i)
#pragma unroll
                for (int j = 0; j < NN; ++j) {
                    const float d = __fsub_rn(llt<NN>(L[e], i, j), mean[i * NN + j]);
                    num = fmaf(d, d, num);
                }
            const float q = den > 0.f ? sqrtf(num / den) : 0.f;
            worst = q > worst ? q : worst;
        }
    return worst;
}

// The same for any number of members: one member's factors at a time, formed again for the
// deviations.  (Kept for all of up to 16 members they are 1.3 KB a thread of local memory:
// 65 536 points, whole inference, 8 members 1.08 ms, this way 0.91; 16 members 2.08 and 1.77.)
// The additions run in the same order.
template <int NN, int OFF, int OO>
__device__ __forceinline__ float ensemble_tensor_any(int r, int ldz, int members, const float* __restrict__ z,
                                                     int64_t zstride, const uint8_t* __restrict__ diag,
                                                     double* __restrict__ stage) {
    constexpr int NF = NN * (NN + 1) / 2;
    float L[NF], mean[NN * NN], den = 0.f, worst = 0.f;
    auto factors = [&](int e) {
#pragma unroll
        for (int c = 0; c < NF; ++c) {
            const float zz = __ldg(z + e * zstride + (int64_t)(OFF + c) * ldz + r);
            L[c] = diag[OFF + c] ? (zz > 20.f ? zz : log1pf(expf(zz))) : zz;
        }
    };
#pragma unroll
    for (int c = 0; c < NN * NN; ++c) mean[c] = 0.f;
#pragma unroll 1
    for (int e = 0; e < members; ++e) {
        factors(e);
#pragma unroll
        for (int c = 0; c < NN * NN; ++c) mean[c] += llt<NN>(L, c / NN, c % NN);
    }
    const float inv = 1.f / (float)members;
#pragma unroll
    for (int c = 0; c < NN * NN; ++c) {
        mean[c] = __fmul_rn(mean[c], inv);
        stage[OO + c] = (double)mean[c];
        den = fmaf(mean[c], mean[c], den);
    }
#pragma unroll 1
    for (int e = 0; e < members; ++e) {
        factors(e);
        float num = 0.f;
#pragma unroll
        for (int c = 0; c < NN * NN; ++c) {
            const float d = __fsub_rn(llt<NN>(L, c / NN, c % NN), mean[c]);
            num = fmaf(d, d, num);
        }
        const float q = den > 0.f ? sqrtf(num / den) : 0.f;
        worst = q > worst ? q : worst;
    }
    return worst;
}

// C [n][36], K [n][9], D [n][9] = mean over the members times the reference scales (SI
// units, FP64), spread[n] the largest of the three tensors'.  The means of a block's
// points are staged in shared memory and each output is stored as one contiguous run of
// rows.  MM: at most so many members, whose factors stay in registers (0: any number).
template <int MM>
__global__ void __launch_bounds__(ENS_BLOCK) k_ensemble(int n, int ldz, int members, const float* __restrict__ z,
                                                        int64_t zstride, const uint8_t* __restrict__ diag, double rc,
                                                        double rk, double rd, double* __restrict__ C,
                                                        double* __restrict__ K, double* __restrict__ D,
                                                        double* __restrict__ spread) {
    __shared__ double stage[ENS_BLOCK * ENS_LD];
    const int r0 = blockIdx.x * ENS_BLOCK, r = r0 + threadIdx.x;
    if (r < n) {
        double* st = stage + threadIdx.x * ENS_LD;
        float a, b, c;
        if constexpr (MM > 0) {
            a = ensemble_tensor<6, 0, 0, MM>(r, ldz, members, z, zstride, diag, st);
            b = ensemble_tensor<3, 21, 36, MM>(r, ldz, members, z, zstride, diag, st);
            c = ensemble_tensor<3, 27, 45, MM>(r, ldz, members, z, zstride, diag, st);
        } else {
            a = ensemble_tensor_any<6, 0, 0>(r, ldz, members, z, zstride, diag, st);
            b = ensemble_tensor_any<3, 21, 36>(r, ldz, members, z, zstride, diag, st);
            c = ensemble_tensor_any<3, 27, 45>(r, ldz, members, z, zstride, diag, st);
        }
        spread[r] = (double)fmaxf(a, fmaxf(b, c));
    }
    __syncthreads();
    const int rows = min(ENS_BLOCK, n - r0);
    for (int i = threadIdx.x; i < rows * 36; i += ENS_BLOCK)
        C[(int64_t)r0 * 36 + i] = stage[(i / 36) * ENS_LD + i % 36] * rc;
    for (int i = threadIdx.x; i < rows * 9; i += ENS_BLOCK) {
        K[(int64_t)r0 * 9 + i] = stage[(i / 9) * ENS_LD + 36 + i % 9] * rk;
        D[(int64_t)r0 * 9 + i] = stage[(i / 9) * ENS_LD + 45 + i % 9] * rd;
    }
}

// members' outputs z + e zstride
void launch_ensemble(int n, int ldz, int members, const float* z, int64_t zstride, const uint8_t* diag, double rc,
                     double rk, double rd, double* C, double* K, double* D, double* spread, cudaStream_t s) {
    const int grid = (n + ENS_BLOCK - 1) / ENS_BLOCK;
    if (members <= 4)
        k_ensemble<4><<<grid, ENS_BLOCK, 0, s>>>(n, ldz, members, z, zstride, diag, rc, rk, rd, C, K, D, spread);
    else
        k_ensemble<0><<<grid, ENS_BLOCK, 0, s>>>(n, ldz, members, z, zstride, diag, rc, rk, rd, C, K, D, spread);
}

}  // namespace rve
