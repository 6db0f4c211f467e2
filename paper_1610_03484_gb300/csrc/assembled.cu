// Assembled operator (sm_103a), orders 1 and 2.
//
// Within a batch the stiffness of column c is s_0(c) K_0 + s_1(c) K_1 with the two
// phases' matrices K_0, K_1 shared by every column (degradation scales the matrix
// modulus only, Sec. 5).  Both are assembled once per mesh, boundary condition and
// materials; a row lists its phase-0 entries, then its phase-1 entries, so nodes
// inside one phase store each block once.
//
// Per scalar DOF node a row holds about 15 blocks at p = 1 and 28 at p = 2, i.e. 23
// and 336 FMAs per tetrahedron and column, against about 130 and 610 element by
// element, and rows are gathered and stored once where elements scatter 12 and 30
// atomic additions.  At p = 3 a row holds about 51 blocks of 4.5 nodes per
// tetrahedron (2065 FMAs against 2080, and 7 times the matrix), so the element form
// stays the better one there.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <vector>

#include "assembled.h"
#include "rve_internal.h"

namespace rve {
namespace {

__host__ __device__ constexpr int aut6(int i, int j) {
    return i <= j ? (i * 6 - i * (i - 1) / 2 + (j - i)) : (j * 6 - j * (j - 1) / 2 + (i - j));
}
__host__ __device__ constexpr int avoigt(int i, int j) {
    return i == j ? i : (i + j == 1 ? 3 : (i + j == 3 ? 4 : 5));
}

// One warp per row: the FP64 sums over the elements of the row's node that hold the coupled
// node and belong to the entry's phase,
//   |T| sum_lm D_{cl,dm} g_lm,  g = J^-T R_ab J^-1,  R_ab[k][l] = sum_m A[k][m][a] A[l][m][b],
// written in FP64 and / or FP32.  Bound by the FP64 pipe, which takes as long for one lane of
// a warp as for all: a lane first forms the block of one pair (element, local function), so
// that all have work, and the blocks then meet in the entries through shared memory, a lane
// per entry and the elements in order.  (With a lane per entry from the start, 4 of 17 entries
// of a row at p = 1 meet in an element: 40x40x16, p = 1, mechanics 4.8 ms, this way 0.98; 24x24x8,
// p = 2 3.2 and 1.40.)
template <int NE, int NC>
__global__ void __launch_bounds__(128) k_assemble(AsmGraph G, const int32_t* __restrict__ edofs,
                                                  const uint8_t* __restrict__ phase,
                                                  const double* __restrict__ geo, const double* __restrict__ mat,
                                                  const double* __restrict__ rtab, double* __restrict__ ent64,
                                                  float* __restrict__ ent32) {
    constexpr int NV = NC == 3 ? 9 : 2, ST = NC == 3 ? 9 : 3, EL = 32 / NE;   // elements a pass
    __shared__ double blocks[4][32 * ST];
    __shared__ uint32_t keys[4][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t row = (int64_t)blockIdx.x * 4 + warp;
    if (row >= G.n) return;   // (whole warps)
    double* blk = blocks[warp];
    uint32_t* key = keys[warp];
    const int node = G.order[row], sp = G.split[row], q0 = G.eptr[node], q1 = G.eptr[node + 1], k1 = G.ptr[row + 1];
    for (int k0 = G.ptr[row]; k0 < k1; k0 += 64) {
        // this lane's entries k0 + lane and k0 + 32 + lane: coupled node and phase
        uint32_t mine[2];
        int col[2];
        double A[2][NV];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = k0 + 32 * h + lane;
            col[h] = k < k1 ? G.col[k] : 0;
            mine[h] = k < k1 ? 2u * (uint32_t)col[h] + (k >= sp ? 1u : 0u) : 0xfffffffeu;
#pragma unroll
            for (int i = 0; i < NV; ++i) A[h][i] = 0.0;
        }
        for (int qb = q0; qb < q1; qb += EL) {
            const int q = qb + lane / NE;
            uint32_t found = 0xffffffffu;
            if (lane < EL * NE && q < q1) {
                const int64_t e = G.inc[q] / NE;
                const int a = G.inc[q] % NE, b = lane % NE;
                found = 2u * (uint32_t)__ldg(edofs + e * NE + b) + (phase[e] != 0 ? 1u : 0u);
                const double* R = rtab + (a * NE + b) * 9;
                const double* J = geo + e * 10;
                const double vol = J[9];
                double t[9], g[9];
#pragma unroll
                for (int i = 0; i < 3; ++i)
#pragma unroll
                    for (int m = 0; m < 3; ++m)
                        t[i * 3 + m] = R[i * 3] * J[m] + R[i * 3 + 1] * J[3 + m] + R[i * 3 + 2] * J[6 + m];
#pragma unroll
                for (int l = 0; l < 3; ++l)
#pragma unroll
                    for (int m = 0; m < 3; ++m)
                        g[l * 3 + m] = vol * (J[l] * t[m] + J[3 + l] * t[3 + m] + J[6 + l] * t[6 + m]);
                if constexpr (NC == 3) {
                    const double* D = mat + e * 21;
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int d = 0; d < 3; ++d) {
                            double v = 0.0;
#pragma unroll
                            for (int l = 0; l < 3; ++l)
#pragma unroll
                                for (int m = 0; m < 3; ++m) v += D[aut6(avoigt(i, l), avoigt(d, m))] * g[l * 3 + m];
                            blk[lane * ST + i * 3 + d] = v;
                        }
                } else {
                    const double* D = mat + e * 12;
#pragma unroll
                    for (int f = 0; f < 2; ++f) {
                        double v = 0.0;
#pragma unroll
                        for (int l = 0; l < 3; ++l)
#pragma unroll
                            for (int m = 0; m < 3; ++m) v += D[6 * f + avoigt(l, m)] * g[l * 3 + m];
                        blk[lane * ST + f] = v;
                    }
                }
            }
            key[lane] = found;
            __syncwarp();
#pragma unroll
            for (int el = 0; el < EL; ++el) {
                int at[2] = {-1, -1};
#pragma unroll
                for (int b = 0; b < NE; ++b) {
                    const uint32_t u = key[el * NE + b];
                    if (u == mine[0]) at[0] = el * NE + b;
                    if (u == mine[1]) at[1] = el * NE + b;
                }
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    if (at[h] >= 0)
#pragma unroll
                        for (int i = 0; i < NV; ++i) A[h][i] += blk[at[h] * ST + i];
            }
            __syncwarp();
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int64_t k = k0 + 32 * h + lane;
            if (k >= k1) continue;
            if (ent64) {
                double* o = ent64 + k * AsmEntry<double, NC>::WORDS;
#pragma unroll
                for (int i = 0; i < NV; ++i) o[i] = A[h][i];
                o[NV] = __longlong_as_double((long long)col[h]);
            }
            if (ent32) {
                float* o = ent32 + k * AsmEntry<float, NC>::WORDS;
#pragma unroll
                for (int i = 0; i < NV; ++i) o[i] = (float)A[h][i];
                o[NV] = __int_as_float(col[h]);
            }
        }
    }
}

// ------------------------------------------------------------- the product
template <typename T, int VEC>
struct Pack;
template <typename T>
struct Pack<T, 1> {
    using V = T;
};
template <>
struct Pack<float, 2> {
    using V = float2;
};
template <>
struct Pack<float, 4> {
    using V = float4;
};
template <>
struct Pack<double, 2> {
    using V = double2;
};

template <typename T, int VEC>
__device__ __forceinline__ void load_pack(const T* p, T (&v)[VEC]) {
    *reinterpret_cast<typename Pack<T, VEC>::V*>(v) = *reinterpret_cast<const typename Pack<T, VEC>::V*>(p);
}
template <typename T, int VEC>
__device__ __forceinline__ void store_pack(T* p, const T (&v)[VEC]) {
    *reinterpret_cast<typename Pack<T, VEC>::V*>(p) = *reinterpret_cast<const typename Pack<T, VEC>::V*>(v);
}

// the entry's values and coupled node
template <int NC>
__device__ __forceinline__ int load_entry(const float* p, float (&a)[NC == 3 ? 9 : 2]) {
    const float4* q = reinterpret_cast<const float4*>(p);
    if constexpr (NC == 3) {
        const float4 u = __ldg(q), v = __ldg(q + 1), w = __ldg(q + 2);
        a[0] = u.x; a[1] = u.y; a[2] = u.z;
        a[3] = u.w; a[4] = v.x; a[5] = v.y;
        a[6] = v.z; a[7] = v.w; a[8] = w.x;
        return __float_as_int(w.y);
    } else {
        const float4 u = __ldg(q);
        a[0] = u.x;
        a[1] = u.y;
        return __float_as_int(u.z);
    }
}
template <int NC>
__device__ __forceinline__ int load_entry(const double* p, double (&a)[NC == 3 ? 9 : 2]) {
    const double2* q = reinterpret_cast<const double2*>(p);
    if constexpr (NC == 3) {
        double2 u[5];
#pragma unroll
        for (int i = 0; i < 5; ++i) u[i] = __ldg(q + i);
#pragma unroll
        for (int i = 0; i < 9; ++i) a[i] = (i & 1) ? u[i / 2].y : u[i / 2].x;
        return (int)__double_as_longlong(u[4].y);
    } else {
        const double2 u = __ldg(q), v = __ldg(q + 1);
        a[0] = u.x;
        a[1] = u.y;
        return (int)__double_as_longlong(v.x);
    }
}

// A thread takes VEC adjacent columns of one row and every KS-th of its entries: per
// entry it loads the block (the same words for the lanes of a row) and NC VEC values
// of x and does NC NC VEC FMAs.  With KS > 1 the partial rows are added by shuffles:
// the first exchange leaves one of the two columns with each lane, so that the sums,
// the scaling and the energies are spread over the lanes too (each of these is an FP64
// instruction, and FP64 runs at two lanes per clock and SM).
// Columns come in chunks of ASM_CHUNK per block, of which only groups with an active
// column take lanes; a block walks a contiguous run of rows, which are stored along a
// space-filling curve, so that its gathers of x meet in L1.
//
// What follows the row's product, MODE:
//   PRODUCT   y = A x, energies x . A x
//   RESIDUAL  y = b - A x
//   STEP      one step of the Chebyshev recurrence (see launch_cheb_step): x is z,
//             d = c1 d_in + c2 D^-1 (b - A z), y = z + d
//   LAST      the same, d not kept, and (r64, y) per column into eacc
enum AsmMode { PRODUCT, RESIDUAL, STEP, LAST };
constexpr int ASM_THREADS = 256, ASM_CHUNK = 48;

template <typename T, int NC, int VEC, int KS, int MODE>
__global__ void __launch_bounds__(ASM_THREADS, sizeof(T) == 8 ? 3 : (NC == 3 && VEC == 4 ? 2 : 4))
    k_asm_product(AsmView<T> A, const T* __restrict__ x, const T* __restrict__ b, T* __restrict__ y, int ncols,
                  const int32_t* __restrict__ active, double* __restrict__ eacc, ChebArgs ch) {
    static_assert(KS == 1 || VEC == 2, "split rows exchange two columns");
    constexpr int NV = NC == 3 ? 9 : 2, W = AsmEntry<T, NC>::WORDS;
    constexpr int VO = KS == 1 ? VEC : 1;   // columns a lane finishes
    constexpr int UNROLL = sizeof(T) == 8 ? 2 : (NC == 3 ? 2 : 4);
    __shared__ int glist[ASM_CHUNK / VEC];
    __shared__ int n_groups;
    const int c0 = blockIdx.x * ASM_CHUNK, ng = min(ASM_CHUNK, ncols - c0) / VEC;
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        bool on = lane < ng;
        if (on && active) {
            on = false;
#pragma unroll
            for (int v = 0; v < VEC; ++v) on = on || active[c0 + lane * VEC + v] != 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (on) glist[__popc(m & ((1u << lane) - 1u))] = lane;
        if (lane == 0) n_groups = __popc(m);
    }
    __syncthreads();
    const int G = n_groups;
    if (G == 0) return;
    const int L = G * KS, R = ASM_THREADS / L, rr = threadIdx.x / L, g = (threadIdx.x % L) / KS;
    const int part = KS == 1 ? 0 : (int)threadIdx.x % KS;
    const bool live = rr < R;
    const int col = c0 + glist[g] * VEC;
    const int ocol = KS == 1 ? col : col + (part & 1);
    const bool owner = live && (part >> 1) == 0;
    T s0[VO], s1[VO], e[VO], ec[VO];   // energies, FP32 with a compensation word
    double rz[VO];
#pragma unroll
    for (int v = 0; v < VO; ++v) {
        s0[v] = A.scale[2 * (ocol + v)];
        s1[v] = A.scale[2 * (ocol + v) + 1];
        e[v] = ec[v] = T(0);
        rz[v] = 0.0;
    }
    bool second[VEC];   // scalar fields: the column takes the second value (diffusivity)
#pragma unroll
    for (int v = 0; v < VEC; ++v) second[v] = (col + v) % 6 >= 3;
    const int64_t lo = A.n * blockIdx.y / gridDim.y, hi = A.n * (blockIdx.y + 1) / gridDim.y;
    // every lane of a warp runs the same number of rows (shuffles below)
    for (int64_t row0 = lo; row0 < hi; row0 += R) {
        const int64_t row = row0 + rr;
        const bool on = live && row < hi;
        int k0 = 0, ks = 0, k1 = 0;
        if (on) {
            k0 = __ldg(A.ptr + row);
            ks = __ldg(A.split + row);
            k1 = __ldg(A.ptr + row + 1);
        }
        T acc[NC][VEC], out[NC][VO];
        auto run = [&](int from, int to) {
#pragma unroll
            for (int i = 0; i < NC; ++i)
#pragma unroll
                for (int v = 0; v < VEC; ++v) acc[i][v] = T(0);
#pragma unroll (UNROLL)
            for (int k = from + part; k < to; k += KS) {
                T a[NV];
                const int c = load_entry<NC>(A.ent + (int64_t)k * W, a);
                const uint32_t at = (uint32_t)c * (uint32_t)(NC * ncols) + (uint32_t)col;
#pragma unroll
                for (int j = 0; j < NC; ++j) {
                    T xv[VEC];
                    load_pack<T, VEC>(x + at + (uint32_t)(j * ncols), xv);
#pragma unroll
                    for (int i = 0; i < NC; ++i)
#pragma unroll
                        for (int v = 0; v < VEC; ++v) {
                            const T m = NC == 3 ? a[i * 3 + j] : (second[v] ? a[1] : a[0]);
                            acc[i][v] = fma(m, xv[v], acc[i][v]);
                        }
                }
            }
        };
        // the row's sums over its lanes: column part & 1 stays here
        auto gather = [&](int i, int v) -> T {
            if constexpr (KS == 1) {
                return acc[i][v];
            } else {
                const T keep = part & 1 ? acc[i][1] : acc[i][0], give = part & 1 ? acc[i][0] : acc[i][1];
                T t = keep + __shfl_xor_sync(0xffffffffu, give, 1);
#pragma unroll
                for (int o = 2; o < KS; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                return t;
            }
        };
        run(k0, ks);
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
            for (int v = 0; v < VO; ++v) out[i][v] = s0[v] * gather(i, v);
        if (__any_sync(0xffffffffu, ks < k1)) {
            run(ks, k1);
#pragma unroll
            for (int i = 0; i < NC; ++i)
#pragma unroll
                for (int v = 0; v < VO; ++v) out[i][v] = fma(s1[v], gather(i, v), out[i][v]);
        }
        if (!on || !owner) continue;
        const int node = __ldg(A.order + row);
        const uint32_t at = (uint32_t)node * (uint32_t)(NC * ncols) + (uint32_t)ocol;
        T dot[VO];
#pragma unroll
        for (int v = 0; v < VO; ++v) dot[v] = T(0);
#pragma unroll
        for (int i = 0; i < NC; ++i) {
            const uint32_t ai = at + (uint32_t)(i * ncols);
            T o[VO];
            if constexpr (MODE == RESIDUAL) {
                load_pack<T, VO>(b + ai, o);
#pragma unroll
                for (int v = 0; v < VO; ++v) o[v] -= out[i][v];
            } else if constexpr (MODE == STEP || MODE == LAST) {
                const int64_t ri = (int64_t)node * NC + i;
                T zv[VO], dv[VO], rv[VO];
                load_pack<T, VO>(x + ai, zv);
                load_pack<T, VO>(ch.d_in + ai, dv);
                load_pack<T, VO>(b + ai, rv);
#pragma unroll
                for (int v = 0; v < VO; ++v) {
                    const int grp = NC == 3 ? (ocol + v) / 6 : ((ocol + v) % 6 >= 3 ? 1 : 0);
                    const T di = __ldg(ch.dinv + ri * ch.groups + grp);
                    dv[v] = fma(ch.c1, dv[v], ch.c2 * (di * (rv[v] - out[i][v])));
                    o[v] = zv[v] + dv[v];
                }
                if constexpr (MODE == STEP) {
                    store_pack<T, VO>(ch.d_out + ai, dv);
                } else {
#pragma unroll
                    for (int v = 0; v < VO; ++v) rz[v] = fma(ch.r64[ai + v], (double)o[v], rz[v]);
                }
            } else {
                T xv[VO];
                load_pack<T, VO>(x + ai, xv);
#pragma unroll
                for (int v = 0; v < VO; ++v) {
                    o[v] = out[i][v];
                    dot[v] = fma(xv[v], o[v], dot[v]);
                }
            }
            store_pack<T, VO>(y + ai, o);
        }
        if constexpr (MODE == PRODUCT) {
#pragma unroll
            for (int v = 0; v < VO; ++v) {
                if constexpr (sizeof(T) == 8) {
                    e[v] += dot[v];
                } else {
                    const float yv = dot[v] - ec[v], t = e[v] + yv;
                    ec[v] = (t - e[v]) - yv;
                    e[v] = t;
                }
            }
        }
    }
    if constexpr (MODE == PRODUCT || MODE == LAST) {
        if (eacc) {
            // the rows of the block per column: eight partial sums, then one
            __shared__ double buf[ASM_THREADS];
            double* acc_out = eacc + (size_t)(blockIdx.y % ACC_SLOTS) * ncols;
            const int parts = min(R, 8), C = KS == 1 ? G : 2 * G, ci = KS == 1 ? g : 2 * g + (part & 1);
#pragma unroll
            for (int v = 0; v < VO; ++v) {
                if (owner) buf[rr * C + ci] = MODE == LAST ? rz[v] : (double)e[v] - (double)ec[v];
                __syncthreads();
                double t = 0.0;
                if (owner && rr < parts)
                    for (int q = rr; q < R; q += parts) t += buf[q * C + ci];
                __syncthreads();
                if (owner && rr < parts) buf[rr * C + ci] = t;
                __syncthreads();
                if (owner && rr == 0) {
                    t = 0.0;
                    for (int q = 0; q < parts; ++q) t += buf[q * C + ci];
                    atomicAdd(acc_out + ocol + v, t);
                }
                if (v + 1 < VO) __syncthreads();
            }
        }
    }
}

template <typename T, int NC, int VEC, int KS, int MODE>
void run_product(const AsmView<T>& A, const T* x, const T* b, T* y, int ncols, const int32_t* active, double* eacc,
                 cudaStream_t s, const ChebArgs& ch = ChebArgs()) {
    static std::atomic<int> cached{0};   // resident blocks per SM of this instance
    int per_sm = cached.load(std::memory_order_relaxed);
    if (per_sm == 0) {
        int v = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_asm_product<T, NC, VEC, KS, MODE>, ASM_THREADS, 0) !=
                cudaSuccess ||
            v < 1)
            v = 1;
        per_sm = v;
        cached.store(v, std::memory_order_relaxed);
    }
    const int gx = (ncols + ASM_CHUNK - 1) / ASM_CHUNK;
    const int lanes = std::min(ncols, ASM_CHUNK) / VEC * KS, rows = ASM_THREADS / lanes;
    // FP32: one wave, so that a block's run of rows shares its gathers in L1.  FP64: a
    // block per pass, since rows differ in length and the FP64 pipe wants them balanced.
    const int64_t wave = std::max<int64_t>(1, (int64_t)per_sm * sm_count() / gx);
    const int64_t passes = (A.n + rows - 1) / rows;
    const int64_t gy = std::max<int64_t>(1, sizeof(T) == 8 ? std::min<int64_t>(passes, 65535) : std::min(wave, passes));
    k_asm_product<T, NC, VEC, KS, MODE><<<dim3(gx, (unsigned)gy), ASM_THREADS, 0, s>>>(A, x, b, y, ncols, active, eacc, ch);
}

// d[row][g] = 1 / (s_0 diag_0 + s_1 diag_1), 0 on Dirichlet rows; times f in FP32
__global__ void __launch_bounds__(256) k_jacobi_inverse(RowView<double> rv, int groups, double* __restrict__ dinv,
                                                        float* __restrict__ dinv32, double f32) {
    const int64_t n = rv.n_rows * groups;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / groups;
        const int g = (int)(i % groups);
        const int f = rv.nfield == 2 ? g : 0, col = rv.nfield == 2 ? 3 * g : 6 * g;
        double d = fma(rv.scale[2 * col], rv.diag[(int64_t)(2 * f) * rv.n_rows + row],
                       __dmul_rn(rv.scale[2 * col + 1], rv.diag[(int64_t)(2 * f + 1) * rv.n_rows + row]));
        d = d > 0.0 ? 1.0 / d : 0.0;
        if (rv.mask && rv.mask[row / rv.nc]) d = 0.0;
        dinv[i] = d;
        if (dinv32) dinv32[i] = (float)(f32 * d);
    }
}

}  // namespace

void launch_assemble(int p, int nc, const AsmGraph& g, const int32_t* edofs, const uint8_t* phase,
                     const double* geo64, const double* mat64, double* rtab, double* ent64, float* ent32,
                     cudaStream_t s) {
    const Basis& B = basis(p);
    const int ne = B.ne, nm = B.nm;
    std::vector<double> R((size_t)ne * ne * 9, 0.0);
    // reference gradient of function j on mode m: the vertex functions (j < 4) are
    // linear, with the constant mode only
    auto grad = [&](int k, int m, int j) -> double {
        if (j < 4) return m == 0 ? (j == k + 1 ? 1.0 : (j == 0 ? -1.0 : 0.0)) : 0.0;
        return B.A[(size_t)(k * nm + m) * ne + j];
    };
    for (int a = 0; a < ne; ++a)
        for (int b = 0; b < ne; ++b)
            for (int k = 0; k < 3; ++k)
                for (int l = 0; l < 3; ++l) {
                    double v = 0.0;
                    for (int m = 0; m < nm; ++m) v += grad(k, m, a) * grad(l, m, b);
                    R[(size_t)(a * ne + b) * 9 + 3 * k + l] = v;
                }
    cudaMemcpyAsync(rtab, R.data(), R.size() * 8, cudaMemcpyHostToDevice, s);
    const unsigned grid = (unsigned)((g.n + 3) / 4);
#define RVE_ASSEMBLE(PP, NEE, NCC) \
    if (p == PP && nc == NCC) k_assemble<NEE, NCC><<<grid, 128, 0, s>>>(g, edofs, phase, geo64, mat64, rtab, ent64, ent32);
    RVE_ASSEMBLE(1, 4, 3) RVE_ASSEMBLE(2, 10, 3) RVE_ASSEMBLE(1, 4, 1) RVE_ASSEMBLE(2, 10, 1)
#undef RVE_ASSEMBLE
}

// Columns per thread and lanes per row.  Four columns per thread need 16-byte aligned
// rows and eight warps per SM: with fewer, each thread's serial walk along its row bounds
// the product (6x7x8, p = 1, 108 columns: a mixed call of 18 points took 2.68 ms with four
// columns a thread, 2.27 with split rows).  Otherwise the entries of a row are split over
// four lanes, or eight where even then the chip has less than four warps per scheduler.
#define RVE_ASM_RUN(MODE, ...)                                                              \
    do {                                                                                    \
        const bool few = A.n * ncols / 2 < (int64_t)sm_count() * 4 * 32;                    \
        if constexpr (sizeof(T) == 4) {                                                     \
            if (ncols % 4 == 0 && ncols >= 24 && A.n * ncols / 4 >= (int64_t)sm_count() * 256) { \
                if (nc == 3) return run_product<T, 3, 4, 1, MODE>(__VA_ARGS__);             \
                return run_product<T, 1, 4, 1, MODE>(__VA_ARGS__);                          \
            }                                                                               \
        }                                                                                   \
        if (few && ncols <= 12) {                                                           \
            if (nc == 3) return run_product<T, 3, 2, 8, MODE>(__VA_ARGS__);                 \
            return run_product<T, 1, 2, 8, MODE>(__VA_ARGS__);                              \
        }                                                                                   \
        if (nc == 3) return run_product<T, 3, 2, 4, MODE>(__VA_ARGS__);                     \
        return run_product<T, 1, 2, 4, MODE>(__VA_ARGS__);                                  \
    } while (0)

template <typename T>
void launch_asm_product(int nc, const AsmView<T>& A, const T* x, T* y, int ncols, const int32_t* active,
                        double* energy_acc, cudaStream_t s) {
    RVE_ASM_RUN(PRODUCT, A, x, nullptr, y, ncols, active, energy_acc, s);
}
template void launch_asm_product<float>(int, const AsmView<float>&, const float*, float*, int, const int32_t*,
                                        double*, cudaStream_t);
template void launch_asm_product<double>(int, const AsmView<double>&, const double*, double*, int, const int32_t*,
                                         double*, cudaStream_t);

template <typename T>
void launch_asm_residual(int nc, const AsmView<T>& A, const T* x, const T* b, T* y, int ncols, cudaStream_t s) {
    RVE_ASM_RUN(RESIDUAL, A, x, b, y, ncols, nullptr, nullptr, s);
}
template void launch_asm_residual<double>(int, const AsmView<double>&, const double*, const double*, double*, int,
                                          cudaStream_t);

void launch_jacobi_inverse(const RowView<double>& rv, int groups, double* dinv, float* dinv32, double f32,
                           cudaStream_t s) {
    const int64_t n = rv.n_rows * groups;
    const int64_t b = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sm_count() * 8));
    k_jacobi_inverse<<<(unsigned)b, 256, 0, s>>>(rv, groups, dinv, dinv32, f32);
}

void launch_cheb_step(int nc, const AsmView<float>& A, const float* z, const float* r32, float* z_new,
                      const ChebArgs& ch, int ncols, const int32_t* active, double* rz_acc, cudaStream_t s) {
    using T = float;
    if (rz_acc) RVE_ASM_RUN(LAST, A, z, r32, z_new, ncols, active, rz_acc, s, ch);
    RVE_ASM_RUN(STEP, A, z, r32, z_new, ncols, active, nullptr, s, ch);
}

// ------------------------------------------------ vector passes of that iteration
// x += alpha p, r -= alpha q (apply), then the Chebyshev start z = w D^-1 r in FP32,
// r in FP32, and (r, D^-1 r) per column into rj_acc (the stopping test's norm).
__global__ void __launch_bounds__(256) k_cheb_update(RowView<double> rv, const float* __restrict__ dinv32,
                                                     double* __restrict__ x, double* __restrict__ r,
                                                     const double* __restrict__ p, const double* __restrict__ q,
                                                     float* __restrict__ r32, float* __restrict__ z, float w,
                                                     ColState cs, int ncols, int cpb, int apply) {
    const int rows = blockDim.x / cpb;
    const int cl = threadIdx.x % cpb, rr = threadIdx.x / cpb;
    const int col = blockIdx.x * cpb + cl;
    __shared__ double s_alpha[256];
    __shared__ int s_on[256];
    __shared__ double buf[256];
    if (rr == 0) {
        const bool act = cs.active[col] != 0;
        double a = 0.0;
        int on = act ? 1 : 0;
        if (act && apply) {
            double pq = 0.0;
#pragma unroll
            for (int k = 0; k < ACC_SLOTS; ++k) pq += cs.pq_acc[(size_t)k * ncols + col];
            a = cs.rz[col] / pq;
            if (!(pq > 0.0) || !isfinite(a)) on = 2;
        }
        s_alpha[cl] = a;
        s_on[cl] = on;
    }
    __syncthreads();
    const double a = s_alpha[cl];
    const int on = s_on[cl];
    if (apply && blockIdx.y == 0 && rr == 0) {
        if (on == 1) {
            cs.alpha[col] = a;
            cs.iters[col] += 1;
        } else if (on == 2) {
            atomicOr(cs.flags, 8);   // the loop control stops the column
            cs.beta[col] = -1.0;
        }
    }
    double acc = 0.0;
    if (on == 1) {
        const int g = rv.nfield == 2 ? ((col % 6) >= 3 ? 1 : 0) : col / 6;
        for (int64_t i = (int64_t)blockIdx.y * rows + rr; i < rv.n_rows; i += (int64_t)gridDim.y * rows) {
            const int64_t idx = i * ncols + col;
            double ri = r[idx];
            if (apply) {
                x[idx] = fma(a, p[idx], x[idx]);
                ri = fma(-a, q[idx], ri);
                r[idx] = ri;
            }
            const double di = __ldg(rv.dinv + i * rv.dinv_groups + g);
            acc = fma(ri, ri * di, acc);
            const float rf = (float)ri;
            r32[idx] = rf;
            z[idx] = w * (__ldg(dinv32 + i * rv.dinv_groups + g) * rf);
        }
    }
    buf[threadIdx.x] = acc;
    __syncthreads();
    if (rr == 0) {
        double t = 0.0;
        for (int k = 0; k < rows; ++k) t += buf[k * cpb + cl];
        atomicAdd(cs.rj_acc + (size_t)(blockIdx.y % ACC_SLOTS) * ncols + col, t);
    }
}

// The Chebyshev step behind an element-by-element product y = A z (added into y, which
// is cleared for the next one): d = c1 d + c2 D^-1 (r - y), z += d; with rz_acc the last
// one: (r64, z) per column is added.  A thread takes two adjacent columns of a row
// (column counts are even); bound by memory latency and bandwidth.
template <bool LAST_>
__global__ void __launch_bounds__(256) k_cheb_vector(int64_t n_rows, int nfield, const float* __restrict__ r32,
                                                     const float* d_in, float* d_out,
                                                     const float* __restrict__ dinv, int groups, float c1, float c2,
                                                     const double* __restrict__ r64, float* __restrict__ z,
                                                     float* __restrict__ y, const int32_t* __restrict__ active,
                                                     int ncols, int cpb, double* __restrict__ rz_acc) {
    const int half = cpb / 2, rows = blockDim.x / half;
    const int cl = threadIdx.x % half, rr = threadIdx.x / half;
    const int col = blockIdx.x * cpb + 2 * cl;
    int g[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) g[v] = nfield == 2 ? ((col + v) % 6 >= 3 ? 1 : 0) : (col + v) / 6;
    double acc[2] = {0.0, 0.0};
    const bool on = rr < rows && (active[col] | active[col + 1]) != 0;
    const int64_t stride = (int64_t)gridDim.y * rows;
    if (on)
        for (int64_t i = (int64_t)blockIdx.y * rows + rr; i < n_rows; i += stride) {
            const int64_t idx = i * ncols + col;
            const float2 dv = *reinterpret_cast<const float2*>(d_in + idx);
            const float2 rv = *reinterpret_cast<const float2*>(r32 + idx);
            const float2 yv = *reinterpret_cast<const float2*>(y + idx);
            const float2 zv = *reinterpret_cast<const float2*>(z + idx);
            const float i0 = __ldg(dinv + i * groups + g[0]), i1 = __ldg(dinv + i * groups + g[1]);
            const float d0 = fmaf(c1, dv.x, c2 * (i0 * (rv.x - yv.x)));
            const float d1 = fmaf(c1, dv.y, c2 * (i1 * (rv.y - yv.y)));
            const float2 zn = make_float2(zv.x + d0, zv.y + d1);
            *reinterpret_cast<float2*>(y + idx) = make_float2(0.f, 0.f);
            *reinterpret_cast<float2*>(z + idx) = zn;
            if constexpr (LAST_) {
                const double2 w = *reinterpret_cast<const double2*>(r64 + idx);
                acc[0] = fma(w.x, (double)zn.x, acc[0]);
                acc[1] = fma(w.y, (double)zn.y, acc[1]);
            } else {
                *reinterpret_cast<float2*>(d_out + idx) = make_float2(d0, d1);
            }
        }
    if constexpr (LAST_) {
        __shared__ double buf[2][256];
        buf[0][threadIdx.x] = acc[0];
        buf[1][threadIdx.x] = acc[1];
        __syncthreads();
        if (threadIdx.x < cpb) {
            const int c = threadIdx.x / 2, v = threadIdx.x & 1;
            double t = 0.0;
            for (int k = 0; k < rows; ++k) t += buf[v][k * half + c];
            atomicAdd(rz_acc + (size_t)(blockIdx.y % ACC_SLOTS) * ncols + blockIdx.x * cpb + threadIdx.x, t);
        }
    }
}

// One block: per active column (r, z) and (r, D^-1 r) from their accumulators, beta and
// the stopping test on the latter (rj <= tol^2 rz0 with rz0 its initial value); a column
// whose (r, z) is not positive stops with flag bit 3, the breakdown of the preconditioner;
// clears the accumulators; with CTL the loop control of the graph's WHILE node.
template <bool CTL>
__global__ void __launch_bounds__(1024) k_cheb_beta(ColState cs, int ncols, int first, cudaGraphConditionalHandle h,
                                                    int32_t* __restrict__ counter, int max_iter) {
    const double tol = *cs.tol;
    bool any = false;
    for (int c = threadIdx.x; c < ncols; c += blockDim.x) {
        double rz = 0.0, rj = 0.0;
#pragma unroll
        for (int k = 0; k < ACC_SLOTS; ++k) {
            rz += cs.rz_acc[(size_t)k * ncols + c];
            rj += cs.rj_acc[(size_t)k * ncols + c];
            cs.rz_acc[(size_t)k * ncols + c] = 0.0;
            cs.rj_acc[(size_t)k * ncols + c] = 0.0;
            cs.pq_acc[(size_t)k * ncols + c] = 0.0;
        }
        if (!cs.active[c]) continue;
        if (!first && cs.beta[c] == -1.0) {   // the update met a direction of no curvature
            cs.active[c] = 0;
            continue;
        }
        const bool done = first ? rj == 0.0 : rj <= tol * tol * cs.rz0[c];
        const bool sound = rz > 0.0 && isfinite(rz);   // (not NaN)
        if (!isfinite(rj)) atomicOr(cs.flags, 1);
        else if (!done && !sound) atomicOr(cs.flags, 8);
        if (done || !sound || !isfinite(rj)) {
            cs.active[c] = 0;
            continue;
        }
        cs.beta[c] = first ? 0.0 : rz / cs.rz[c];
        cs.rz[c] = rz;
        any = true;
    }
    const int more = __syncthreads_or(any ? 1 : 0);
    // the active columns in ascending order (the element operators take lanes for them)
    __shared__ int counts[32], base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int c0 = 0; c0 < ncols; c0 += blockDim.x) {
        const int c = c0 + threadIdx.x;
        const bool on = c < ncols && cs.active[c] != 0;
        const unsigned m = __ballot_sync(0xffffffffu, on);
        if (lane == 0) counts[warp] = __popc(m);
        __syncthreads();
        int off = base;
        for (int w = 0; w < warp; ++w) off += counts[w];
        if (on) cs.list[off + __popc(m & ((1u << lane) - 1u))] = c;
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) base += counts[w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *cs.n_list = base;
    if constexpr (CTL) {
        if (threadIdx.x == 0) {
            const int n = *counter + 1;
            *counter = n;
            cudaGraphSetConditional(h, (more && n < max_iter) ? 1u : 0u);
        }
    }
}

// p = z + beta p (first: p = z, and 0 in columns that take no part); q = 0 when given
// (for an operator that adds into it)
__global__ void __launch_bounds__(256) k_cheb_direction(int64_t n_rows, const float* __restrict__ z,
                                                        double* __restrict__ p, double* __restrict__ q, ColState cs,
                                                        int ncols, int cpb, int first) {
    const int rows = blockDim.x / cpb;
    const int col = blockIdx.x * cpb + threadIdx.x % cpb, rr = threadIdx.x / cpb;
    const bool act = cs.active[col] != 0;
    if (!act && !first) return;
    const double beta = first ? 0.0 : cs.beta[col];
    for (int64_t i = (int64_t)blockIdx.y * rows + rr; i < n_rows; i += (int64_t)gridDim.y * rows) {
        const int64_t idx = i * ncols + col;
        p[idx] = !act ? 0.0 : (first ? (double)z[idx] : fma(beta, p[idx], (double)z[idx]));
        if (q) q[idx] = 0.0;
    }
}

void launch_cheb_update(const RowView<double>& rv, const float* dinv32, double* x, double* r, const double* p,
                        const double* q, float* r32, float* z, float w, ColState cs, bool apply, const Launch& L) {
    dim3 grid(L.ncols / L.cpb, L.nby), block(L.cpb * L.rows_per_block);
    k_cheb_update<<<grid, block, 0, L.stream>>>(rv, dinv32, x, r, p, q, r32, z, w, cs, L.ncols, L.cpb, apply);
}

void launch_cheb_beta(ColState cs, int ncols, bool first, cudaGraphConditionalHandle h, int32_t* counter,
                      int max_iter, bool ctl, cudaStream_t s) {
    const int threads = std::min(1024, ((ncols + 31) / 32) * 32);
    if (ctl)
        k_cheb_beta<true><<<1, threads, 0, s>>>(cs, ncols, first, h, counter, max_iter);
    else
        k_cheb_beta<false><<<1, threads, 0, s>>>(cs, ncols, first, 0, nullptr, 0);
}

void launch_cheb_direction(int64_t n_rows, const float* z, double* p, double* q, ColState cs, bool first,
                           const Launch& L) {
    dim3 grid(L.ncols / L.cpb, L.nby), block(L.cpb * L.rows_per_block);
    k_cheb_direction<<<grid, block, 0, L.stream>>>(n_rows, z, p, q, cs, L.ncols, L.cpb, first);
}

void launch_cheb_vector(int64_t n_rows, int nfield, const float* r32, const ChebArgs& ch, float* z, float* y,
                        const int32_t* active, double* rz_acc, const Launch& L) {
    const int half = L.cpb / 2, rows = 256 / half;
    const int64_t want = (n_rows + rows - 1) / rows;
    dim3 grid(L.ncols / L.cpb, (unsigned)std::min<int64_t>(want, std::max<int64_t>(1, sm_count() * 16 / (L.ncols / L.cpb))));
    if (rz_acc)
        k_cheb_vector<true><<<grid, 256, 0, L.stream>>>(n_rows, nfield, r32, ch.d_in, ch.d_out, ch.dinv, ch.groups, ch.c1,
                                                        ch.c2, ch.r64, z, y, active, L.ncols, L.cpb, rz_acc);
    else
        k_cheb_vector<false><<<grid, 256, 0, L.stream>>>(n_rows, nfield, r32, ch.d_in, ch.d_out, ch.dinv, ch.groups,
                                                         ch.c1, ch.c2, ch.r64, z, y, active, L.ncols, L.cpb, nullptr);
}

// ------------------------------------------------- the largest eigenvalue of D^-1 A
// Power iteration on six columns: a third to a half of them on each phase alone.  For
// any positive scales the largest eigenvalue of D^-1 A is at most the larger of the
// phases' own (numerator and denominator are the same combination of the phases).
namespace {
// columns that run on phase ph only; scalar fields have a conductivity and a
// diffusivity column for each phase
__host__ __device__ inline int power_phase(int nc, int c) { return nc == 3 ? c / 3 : (c % 3 == 1 ? 1 : 0); }

__global__ void k_power_start(int64_t n_rows, float* __restrict__ x) {
    const int64_t n = n_rows * 6;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t h = (uint32_t)i * 2654435761u + 12345u;
        h ^= h >> 15;
        h *= 2246822519u;
        h ^= h >> 13;
        x[i] = (float)(h & 0xffffu) * (1.f / 32768.f) - 1.f;
    }
}

// x <- D^-1 y / 2 of the column's phase; with sums: out[c] += (x, y), out[6 + c] += (x, D x)
__global__ void __launch_bounds__(192) k_power_next(int64_t n_rows, int nc, const double* __restrict__ diag,
                                                    float* __restrict__ x, const float* __restrict__ y,
                                                    double* __restrict__ out) {
    __shared__ double part[2][192];
    const int c = threadIdx.x % 6;
    const int f = nc == 3 ? 0 : (c >= 3 ? 1 : 0);
    const double* dg = diag + (int64_t)(2 * f + power_phase(nc, c)) * n_rows;
    double xy = 0.0, xx = 0.0;
    for (int64_t row = (int64_t)blockIdx.x * 32 + threadIdx.x / 6; row < n_rows; row += (int64_t)gridDim.x * 32) {
        const float d = (float)dg[row], yv = y[row * 6 + c], xv = x[row * 6 + c];
        if (out) {
            xy += (double)xv * yv;
            xx += (double)xv * (double)(xv * d);
        } else {
            x[row * 6 + c] = d > 0.f ? 0.5f * yv / d : 0.f;
        }
    }
    if (!out) return;
    part[0][threadIdx.x] = xy;
    part[1][threadIdx.x] = xx;
    __syncthreads();
    if (threadIdx.x < 6)
        for (int k = 0; k < 2; ++k) {
            double t = 0.0;
            for (int q = 0; q < 32; ++q) t += part[k][q * 6 + threadIdx.x];
            atomicAdd(out + 6 * k + threadIdx.x, t);
        }
}
}  // namespace

void power_scales(int nc, float* scale) {
    for (int c = 0; c < 6; ++c)
        for (int ph = 0; ph < 2; ++ph) scale[2 * c + ph] = power_phase(nc, c) == ph ? 1.f : 0.f;
}

void launch_power_start(int64_t n_rows, float* x, cudaStream_t s) {
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_rows + 31) / 32, (int64_t)sm_count() * 8));
    k_power_start<<<g, 256, 0, s>>>(n_rows, x);
}

void launch_power_next(int nc, int64_t n_rows, const double* diag, float* x, const float* y, double* out,
                       cudaStream_t s) {
    const unsigned g = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n_rows + 31) / 32, (int64_t)sm_count() * 8));
    k_power_next<<<g, 192, 0, s>>>(n_rows, nc, diag, x, y, out);
}

// ------------------------------------------------- uniform traction without rows
// r[row][6 b + j] = constraint row first + j mod n (n = 6 strain rows, or 3 flux rows for
// each of the two scalar fields) on the support, 0 elsewhere (the caller clears r)
__global__ void __launch_bounds__(256) k_traction_loads(int64_t n_sup, int m, int first, int n,
                                                        const int64_t* __restrict__ row,
                                                        const double* __restrict__ coef, int ncols,
                                                        double* __restrict__ r) {
    const int64_t total = n_sup * ncols;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = i / ncols;
        const int col = (int)(i % ncols);
        r[row[s] * ncols + col] = coef[s * m + first + (col % 6) % n];
    }
}

// x[row][6 b + i] = sum_j x[row][6 b + j] mu[b][j][i] + sum_k R_k(node) mu[b][6 + k][i]
// - X_i(node), R_k the rigid modes (three translations and rotations; the constant for a
// scalar field) and X_i the unit macro field of load case i (on vertex nodes: in the
// hierarchic basis a linear field lives there)
__global__ void __launch_bounds__(256) k_traction_combine(int64_t n_rows, int nc, int nrve,
                                                          const double* __restrict__ mu,
                                                          const int32_t* __restrict__ vertex,
                                                          const double* __restrict__ xyz, double* __restrict__ x) {
    const int64_t total = n_rows * nrve;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = i / nrve;
        const int b = (int)(i % nrve);
        double* v = x + row * 6 * nrve + 6 * b;
        const double* M = mu + (int64_t)b * 72;
        double in[6], out[6];
#pragma unroll
        for (int j = 0; j < 6; ++j) in[j] = v[j];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            double t = 0.0;
#pragma unroll
            for (int j = 0; j < 6; ++j) t = fma(in[j], M[j * 6 + k], t);
            out[k] = t;
        }
        const int vert = vertex[row / nc];
        if (vert >= 0) {
            const double* y = xyz + 3 * (int64_t)vert;
            if (nc == 3) {
                const int c = (int)(row % 3);
                out[c] -= y[c];
                // engineering shears 12, 23, 31: E_ab = E_ba = 1/2
                if (c == 0) { out[3] -= 0.5 * y[1]; out[5] -= 0.5 * y[2]; }
                if (c == 1) { out[3] -= 0.5 * y[0]; out[4] -= 0.5 * y[2]; }
                if (c == 2) { out[4] -= 0.5 * y[1]; out[5] -= 0.5 * y[0]; }
                // translations, and rotations e_k x y
                const double rot[3] = {c == 0 ? 0.0 : (c == 1 ? -y[2] : y[1]), c == 0 ? y[2] : (c == 1 ? 0.0 : -y[0]),
                                       c == 0 ? -y[1] : (c == 1 ? y[0] : 0.0)};
#pragma unroll
                for (int k = 0; k < 6; ++k)
                    out[k] += M[(6 + c) * 6 + k] + rot[0] * M[54 + k] + rot[1] * M[60 + k] + rot[2] * M[66 + k];
            } else {
#pragma unroll
                for (int k = 0; k < 6; ++k) out[k] += M[36 + k] - y[k % 3];
            }
        }
#pragma unroll
        for (int k = 0; k < 6; ++k) v[k] = out[k];
    }
}

void launch_traction_loads(int64_t n_sup, int m, int first, int n, const int64_t* row, const double* coef, int ncols,
                           double* r, cudaStream_t s) {
    const int64_t g = std::max<int64_t>(1, std::min<int64_t>((n_sup * ncols + 255) / 256, (int64_t)sm_count() * 8));
    k_traction_loads<<<(unsigned)g, 256, 0, s>>>(n_sup, m, first, n, row, coef, ncols, r);
}

void launch_traction_combine(int64_t n_rows, int nc, int nrve, const double* mu, const int32_t* vertex,
                             const double* xyz, double* x, cudaStream_t s) {
    const int64_t g = std::max<int64_t>(1, std::min<int64_t>((n_rows * nrve + 255) / 256, (int64_t)sm_count() * 8));
    k_traction_combine<<<(unsigned)g, 256, 0, s>>>(n_rows, nc, nrve, mu, vertex, xyz, x);
}

}  // namespace rve
