// Coupled macro time step on the GPU (Secs. 3, 4, 5): heat and moisture
// transport on a linear-tetrahedron macro mesh with the homogenised tensors
// (Eq. Eq_field discretised as Eq. Eq_field_disc, one backward-Euler step), then
// the degradation field 1 - omega at the macro Gauss points by backward Euler of
// the rate form (Eq. Eq_Model_RateForm) and the equivalent exposure time that
// hands each Gauss point to the RVE path (macro_update_gauss_points[_dev] or the
// surrogate) as (T, c, t_eq).
//
// Both fields are solved together as two columns of one assembled operator:
// vectors v[node * 2 + field], field 0 temperature [C], field 1 moisture [wt%].
//
// The macro mechanical problem of the fully nested FE^2 step (Sec. 5) uses the
// same mesh: linear elasticity with the homogenised stiffness C_bar of every
// macro Gauss point, vectors u[node * 3 + component], with a per-DOF held mask,
// solved by PCG with a Chebyshev preconditioner.
// Everything here is FP64 but that preconditioner, which is evaluated in FP32.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <vector>

#include "api_internal.h"
#include "chebyshev.h"
#include "node_graph.h"

struct rve_macro_s {
    rve_ctx ctx = nullptr;
    int64_t nv = 0, nt = 0;
    rve::DevBuf tets, geo, mask, hold, x, b, r, p, q, acc, gp, W, flags;
    std::vector<int32_t> tets_h;
    double KT[6] = {}, Dc[6] = {};          // symmetric (xx, yy, zz, xy, yz, zx)
    double rho_cp = 0;
    bool have_transport = false, have_face = false, have_state = false;
    // assembled operators on the node graph, sliced by 32 rows (see "assembled
    // operators" below); built on the first solve
    int64_t n_slices = 0, n_ell = 0;
    rve::DevBuf g_base, g_col, g_len, g_eptr, g_inc;
    bool have_graph = false;
    bool element_form = false;   // no matrices: the operators element by element
    size_t mat_limit = 0;        // bytes the graph and the matrices may take (0: by the free memory)
    rve::DevBuf t_mass, t_stiff, t_mat, t_dinv;
    rve::DevBuf c_r, c_z, c_z2, c_d, c_dinv;   // FP32 vectors of the elastic preconditioner
    bool have_stiff = false;
    double mat_dt = -1;                     // dt [s] that t_mat and t_dinv were formed for
    // macro mechanics: held DOFs and their values, traction load, inverse Jacobi
    // diagonal, displacement, per-tet mean stiffness [nt][36], the assembled
    // stiffness, Gauss-point stiffness staged from the host [nt*4][36] and stresses
    // [nt*4][6]
    rve::DevBuf mfix, mval, mload, mdinv, mu, cm, mmat, mmat32, cgp, msig;
    bool have_mech_bc = false, have_mech_load = false, have_mech_u = false, have_mech_sig = false;
    // instantiated PCG loops (0 transport, 1 mechanics, 2 its Jacobi iteration), reused while
    // the captured launch parameters stay the same
    struct Loop {
        cudaGraphExec_t exec = nullptr;
        std::vector<unsigned char> key;
    } loop[3];
    ~rve_macro_s() {
        for (auto& l : loop)
            if (l.exec) cudaGraphExecDestroy(l.exec);
    }
};

namespace rve {
namespace {

constexpr double kKelvin = 273.15;

struct TransportTensors {
    double KT[6], Dc[6];
};

__device__ __forceinline__ double sym3(const double* k, int i, int j) {
    if (i == j) return k[i];
    const int s = i + j;   // (0,1) -> 3, (1,2) -> 4, (0,2) -> 5
    return k[s == 1 ? 3 : (s == 3 ? 4 : 5)];
}

// --------------------------------------------------- assembled operators
// Both macro problems are solved with assembled matrices.  On linear tetrahedra a
// node couples to about 15 nodes, so a row of the elastic matrix costs 15 x 9 FMAs
// per node, 24 per tetrahedron, where the element-by-element product takes about 117
// and 12 atomic additions; the transport pair needs 30 per node against 120 per
// tetrahedron.  FP64 runs at two FMAs per clock and SM here, which is what bounds
// both forms: on 480k tetrahedra (200 x 40 x 10 cells) one product element by element
// takes 109 us for either problem; assembled 39 us (mechanics) and 13 us (transport),
// cold cache.
//
// Storage: rows in slices of 32 nodes (sliced ELL); slice s holds ELL rows
// base[s] .. base[s + 1], ELL row k of a slice the k-th coupled node of its 32 rows,
// one per lane, so that every load of a warp is contiguous.  Short rows are padded
// with their own node and zero values.

// y += C/dt x etc. need the consistent capacity and the stiffness of both fields per
// entry: mass [ell][32], stiff [ell][32] (conductivity, diffusivity).
// One thread per (ELL row of the slice, lane).
__global__ void __launch_bounds__(256) k_transport_entries(int64_t nv, const int64_t* __restrict__ base,
                                                           const int32_t* __restrict__ col,
                                                           const int32_t* __restrict__ len,
                                                           const int32_t* __restrict__ eptr,
                                                           const int32_t* __restrict__ inc,
                                                           const int32_t* __restrict__ tets,
                                                           const double* __restrict__ geo, TransportTensors prm,
                                                           double* __restrict__ mass, double2* __restrict__ stiff) {
    const int lane = threadIdx.x & 31;
    const int64_t s = blockIdx.x, i = s * 32 + lane, row0 = base[s], row1 = base[s + 1];
    const int n_len = i < nv ? len[i] : 0;
    for (int64_t row = row0 + (threadIdx.x >> 5); row < row1; row += blockDim.x >> 5) {
        double m = 0.0, kt = 0.0, kc = 0.0;
        if (row - row0 < n_len) {
            const int c = col[row * 32 + lane];
            for (int q = eptr[i]; q < eptr[i + 1]; ++q) {
                const int e = inc[q] >> 2, a = inc[q] & 3;
                for (int b = 0; b < 4; ++b) {
                    if (tets[(int64_t)e * 4 + b] != c) continue;
                    const double vol = geo[(int64_t)e * 13];
                    const double* ga = geo + (int64_t)e * 13 + 1 + a * 3;
                    const double* gb = geo + (int64_t)e * 13 + 1 + b * 3;
                    m += (a == b ? 2.0 : 1.0) * vol / 20.0;
                    double ft = 0.0, fc = 0.0;
#pragma unroll
                    for (int j = 0; j < 3; ++j) {
                        ft += ga[j] * (sym3(prm.KT, j, 0) * gb[0] + sym3(prm.KT, j, 1) * gb[1] + sym3(prm.KT, j, 2) * gb[2]);
                        fc += ga[j] * (sym3(prm.Dc, j, 0) * gb[0] + sym3(prm.Dc, j, 1) * gb[1] + sym3(prm.Dc, j, 2) * gb[2]);
                    }
                    kt += vol * ft;
                    kc += vol * fc;
                }
            }
        }
        mass[row * 32 + lane] = m;
        stiff[row * 32 + lane] = make_double2(kt, kc);
    }
}

// mat = cap mass + stiff for the two fields' capacities per time step, and the
// inverse diagonal; one warp per slice
__global__ void __launch_bounds__(256) k_transport_matrix(int64_t nv, int64_t n_slices,
                                                          const int64_t* __restrict__ base,
                                                          const int32_t* __restrict__ col,
                                                          const int32_t* __restrict__ len,
                                                          const double* __restrict__ mass,
                                                          const double2* __restrict__ stiff, double capT, double capC,
                                                          double2* __restrict__ mat, double2* __restrict__ dinv) {
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, i = s * 32 + lane;
    if (s >= n_slices) return;
    const int64_t row0 = base[s], row1 = base[s + 1];
    const int n_len = i < nv ? len[i] : 0;
    for (int64_t row = row0; row < row1; ++row) {
        const double m = mass[row * 32 + lane];
        const double2 k = stiff[row * 32 + lane];
        const double2 v = make_double2(fma(capT, m, k.x), fma(capC, m, k.y));
        mat[row * 32 + lane] = v;
        if (row - row0 < n_len && col[row * 32 + lane] == i) dinv[i] = make_double2(1.0 / v.x, 1.0 / v.y);
    }
}

// b = C/dt x
__global__ void __launch_bounds__(256) k_transport_rhs(int64_t nv, int64_t n_slices, const int64_t* __restrict__ base,
                                                       const int32_t* __restrict__ col,
                                                       const double* __restrict__ mass, double capT, double capC,
                                                       const double2* __restrict__ x, double2* __restrict__ b) {
    const int lane = threadIdx.x & 31;
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, i = s * 32 + lane;
    if (s >= n_slices) return;
    double at = 0.0, ac = 0.0;
#pragma unroll 4
    for (int64_t row = base[s]; row < base[s + 1]; ++row) {
        const double m = mass[row * 32 + lane];
        const double2 v = x[col[row * 32 + lane]];
        at = fma(m, v.x, at);
        ac = fma(m, v.y, ac);
    }
    if (i < nv) b[i] = make_double2(capT * at, capC * ac);
}

// ---------------------------------------------------------- element form
// Without room for the matrices (or past their 32-bit indices) both operators are applied
// element by element, one per thread, with FP64 atomics: see apply_element_form.

// y += (capacity + stiffness) x over both fields
__global__ void __launch_bounds__(256) k_transport_apply(int64_t nt, const int32_t* __restrict__ tets,
                                                         const double* __restrict__ geo, TransportTensors prm,
                                                         double capT, double capC, int stiff,
                                                         const double2* __restrict__ x, double2* __restrict__ y) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nt; e += (int64_t)gridDim.x * blockDim.x) {
        int v[4];
        double2 xa[4], sum = make_double2(0.0, 0.0);
        double gt[3] = {0, 0, 0}, gc[3] = {0, 0, 0};
        const double vol = geo[e * 13];
        const double* g = geo + e * 13 + 1;   // grad lambda_a, [4][3]
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = tets[e * 4 + a];
            xa[a] = x[v[a]];
            sum.x += xa[a].x;
            sum.y += xa[a].y;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                gt[i] = fma(g[a * 3 + i], xa[a].x, gt[i]);
                gc[i] = fma(g[a * 3 + i], xa[a].y, gc[i]);
            }
        }
        double ft[3], fc[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            ft[i] = stiff ? vol * (sym3(prm.KT, i, 0) * gt[0] + sym3(prm.KT, i, 1) * gt[1] + sym3(prm.KT, i, 2) * gt[2]) : 0.0;
            fc[i] = stiff ? vol * (sym3(prm.Dc, i, 0) * gc[0] + sym3(prm.Dc, i, 1) * gc[1] + sym3(prm.Dc, i, 2) * gc[2]) : 0.0;
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const double* ga = g + a * 3;
            atomicAdd(&y[v[a]].x, capT * vol / 20.0 * (sum.x + xa[a].x) + ga[0] * ft[0] + ga[1] * ft[1] + ga[2] * ft[2]);
            atomicAdd(&y[v[a]].y, capC * vol / 20.0 * (sum.y + xa[a].y) + ga[0] * fc[0] + ga[1] * fc[1] + ga[2] * fc[2]);
        }
    }
}

// its diagonal, added into d
__global__ void __launch_bounds__(256) k_transport_diag(int64_t nt, const int32_t* __restrict__ tets,
                                                        const double* __restrict__ geo, TransportTensors prm,
                                                        double capT, double capC, double2* __restrict__ d) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nt * 4; k += (int64_t)gridDim.x * blockDim.x) {
        const double vol = geo[(k >> 2) * 13];
        const double* g = geo + (k >> 2) * 13 + 1 + (k & 3) * 3;
        double kt = capT / 10.0, kc = capC / 10.0;
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) {
                kt += g[i] * sym3(prm.KT, i, j) * g[j];
                kc += g[i] * sym3(prm.Dc, i, j) * g[j];
            }
        atomicAdd(&d[tets[k]].x, vol * kt);
        atomicAdd(&d[tets[k]].y, vol * kc);
    }
}

// d = 1 / d, 0 where d is 0 (nodes of no element)
__global__ void __launch_bounds__(256) k_invert(int64_t n, double* __restrict__ d) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (d[i] != 0.0) d[i] = 1.0 / d[i];
}

// Scalars of the PCG loop (doubles in device memory).  Two fields each:
//   [0] (r, z) of this iteration, [2] (p, q), [4] (r, z) of the previous one,
//   [6] the reference max((b, M^-1 b), (r0, M^-1 r0)), [8] 1 while the field iterates,
//   [10] the same for the next iteration, [12] iterations, [14] (b, M^-1 b);
//   [16] iterations of the loop, [17] their limit, [18] the squared tolerance,
//   [20] (r, D^-1 r) of this iteration where M is not the Jacobi diagonal D (the stopping
//   test's norm, also of [6] and [14]); [22], [23] not 0: the iteration broke down (a
//   direction without curvature; a preconditioned residual whose (r, z) is not positive);
//   [24] the scale of the next residual in FP32.
// An iteration is the product (which also moves (r, z) and the active flags on), the x/r
// update, the preconditioner's steps if any and the p update (which also runs the loop
// control).  Every scalar is written by one thread in a kernel whose other blocks do
// not read it.
constexpr int PCG_SCALARS = 25;

// moves the scalars on to the next iteration; one thread per field of one block
__device__ __forceinline__ void pcg_roll(double* acc, int f) {
    acc[4 + f] = acc[f];
    acc[f] = 0.0;
    acc[20 + f] = 0.0;
    acc[8 + f] = acc[10 + f];
}

// The polynomial's residual is narrowed to FP32 times a power of two s that makes its norm
// about 1, so that it stays inside FP32's range whatever the units and however far the
// iteration has come.  With z = s M^-1 r and p = s (M^-1 r + beta p / s_old), alpha and beta
// are the quotients of the (r, z) formed with that z, as without the scale.
// rj: (r, D^-1 r).
__device__ __forceinline__ double pcg_narrow_scale(double rj) {
    return rj > 0.0 && isfinite(rj) ? ldexp(1.0, -(ilogb(rj) / 2)) : 1.0;
}

// block sums of up to two values per thread, added atomically to out[0..nf-1]
template <int NF>
__device__ __forceinline__ void block_add(const double (&a)[NF], double* out) {
    __shared__ double part[NF][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int f = 0; f < NF; ++f) {
        double v = a[f];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if (lane == 0) part[f][warp] = v;
    }
    __syncthreads();
    if (threadIdx.x < NF) {
        double v = 0.0;
        for (int w = 0; w < nw; ++w) v += part[threadIdx.x][w];
        atomicAdd(out + threadIdx.x, v);
    }
    __syncthreads();
}

// acc[2 + f] += (x, y) of field f = i mod NF, behind a product element by element
template <int NF>
__global__ void __launch_bounds__(256) k_macro_dot(int64_t n, const double* __restrict__ x, const double* __restrict__ y,
                                                   double* __restrict__ acc) {
    if (blockIdx.x == 0 && threadIdx.x < NF) pcg_roll(acc, threadIdx.x);
    double a[NF];
#pragma unroll
    for (int f = 0; f < NF; ++f) a[f] = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n / NF; i += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
        for (int f = 0; f < NF; ++f) a[f] = fma(x[i * NF + f], y[i * NF + f], a[f]);
    block_add<NF>(a, acc + 2);
}

// q = A x for the transport pair and (x, q) per field into acc[2..3]; one warp per
// slice, one lane per node.  acc null: the product alone.
__global__ void __launch_bounds__(256) k_transport_product(int64_t nv, int64_t n_slices,
                                                           const int64_t* __restrict__ base,
                                                           const int32_t* __restrict__ col,
                                                           const double2* __restrict__ mat,
                                                           const double2* __restrict__ x, double2* __restrict__ y,
                                                           double* __restrict__ acc) {
    if (acc && blockIdx.x == 0 && threadIdx.x < 2) pcg_roll(acc, threadIdx.x);
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    double dot[2] = {0.0, 0.0};
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < n_slices; s += nw) {
        const int64_t i = s * 32 + lane, row1 = base[s + 1];
        double at = 0.0, ac = 0.0;
#pragma unroll 4
        for (int64_t row = base[s]; row < row1; ++row) {
            const double2 m = mat[row * 32 + lane];
            const double2 v = x[col[row * 32 + lane]];
            at = fma(m.x, v.x, at);
            ac = fma(m.y, v.y, ac);
        }
        if (i < nv) {
            const double2 v = x[i];
            y[i] = make_double2(at, ac);
            dot[0] = fma(v.x, at, dot[0]);
            dot[1] = fma(v.y, ac, dot[1]);
        }
    }
    if (acc) block_add<2>(dot, acc + 2);
}

// The transport pair's vector passes, Jacobi-preconditioned, a thread per node (both
// fields, 16-byte loads).
//
// r = b - y on free nodes (0 on held ones), p = D^-1 r, acc[0] += (r, p) and
// acc[14] += (b, D^-1 b) over the free nodes (the reference norm)
__global__ void __launch_bounds__(256) k_transport_residual(int64_t nv, const double2* __restrict__ b,
                                                            const double2* __restrict__ y,
                                                            const uint8_t* __restrict__ mask,
                                                            const double2* __restrict__ dinv, double2* __restrict__ r,
                                                            double2* __restrict__ p, double* __restrict__ acc) {
    double a[2] = {0.0, 0.0}, bb[2] = {0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
        const bool held = mask[i] != 0;
        const double2 bi = b[i], yi = y[i], di = dinv[i];
        const double2 ri = held ? make_double2(0.0, 0.0) : make_double2(bi.x - yi.x, bi.y - yi.y);
        const double2 zi = make_double2(ri.x * di.x, ri.y * di.y);
        r[i] = ri;
        p[i] = zi;
        a[0] = fma(ri.x, zi.x, a[0]);
        a[1] = fma(ri.y, zi.y, a[1]);
        if (!held) {
            bb[0] = fma(bi.x, bi.x * di.x, bb[0]);
            bb[1] = fma(bi.y, bi.y * di.y, bb[1]);
        }
    }
    block_add<2>(a, acc);
    block_add<2>(bb, acc + 14);
}

// x += alpha p, r -= alpha q (held nodes stay 0), acc[0] += (r, D^-1 r)
__global__ void __launch_bounds__(256) k_transport_update(int64_t nv, const uint8_t* __restrict__ mask,
                                                          const double2* __restrict__ dinv, double2* __restrict__ x,
                                                          double2* __restrict__ r, const double2* __restrict__ p,
                                                          const double2* __restrict__ q, double* __restrict__ acc) {
    __shared__ double alpha[2];
    if (threadIdx.x < 2) {
        const double pq = acc[2 + threadIdx.x];
        const bool ok = acc[8 + threadIdx.x] != 0.0 && pq > 0.0;
        alpha[threadIdx.x] = ok ? acc[4 + threadIdx.x] / pq : 0.0;
    }
    __syncthreads();
    const double al = alpha[0], be = alpha[1];
    double a[2] = {0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 pi = p[i], qi = q[i], di = dinv[i];
        double2 xi = x[i], ri = r[i];
        const bool held = mask[i] != 0;
        xi.x = fma(al, pi.x, xi.x);
        xi.y = fma(be, pi.y, xi.y);
        ri.x = held ? 0.0 : fma(-al, qi.x, ri.x);
        ri.y = held ? 0.0 : fma(-be, qi.y, ri.y);
        x[i] = xi;
        r[i] = ri;
        a[0] = fma(ri.x, ri.x * di.x, a[0]);
        a[1] = fma(ri.y, ri.y * di.y, a[1]);
    }
    block_add<2>(a, acc);
}

// Per-field tail of an iteration, NF fields: whether the field goes on (the norm at
// acc[norm + f]), beta, and by one thread of the grid the flags and the loop control.
template <int NF>
__device__ __forceinline__ void pcg_tail(double* acc, int norm, cudaGraphConditionalHandle h, double (&beta)[NF],
                                         int (&on)[NF]) {
    __shared__ int broke;
    if (threadIdx.x == 0) broke = 0;
    __syncthreads();
    if (threadIdx.x < NF) {
        const int f = threadIdx.x;
        const double rz = acc[f], old = acc[4 + f];
        const bool open = acc[8 + f] != 0.0 && acc[norm + f] > acc[18] * acc[6 + f];
        const bool sound = rz > 0.0 && isfinite(rz);
        if (open && !sound) broke = 1;
        on[f] = open && sound && acc[22] == 0.0;
        beta[f] = old > 0.0 ? rz / old : 0.0;
    }
    __syncthreads();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        bool any = false;
        for (int f = 0; f < NF; ++f) {
            acc[12 + f] += acc[8 + f];
            acc[10 + f] = on[f] ? 1.0 : 0.0;
            acc[2 + f] = 0.0;
            any = any || on[f];
        }
        if (broke) acc[23] = 1.0;
        const double it = acc[16] + 1.0;
        acc[16] = it;
        cudaGraphSetConditional(h, any && it < acc[17] ? 1u : 0u);
    }
}

// p = D^-1 r + beta p for fields still iterating; loop control
__global__ void __launch_bounds__(256) k_transport_pupdate(int64_t nv, const double2* __restrict__ dinv,
                                                           const double2* __restrict__ r, double2* __restrict__ p,
                                                           double* __restrict__ acc, cudaGraphConditionalHandle h) {
    __shared__ double beta[2];
    __shared__ int on[2];
    pcg_tail<2>(acc, 0, h, beta, on);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
        const double2 di = dinv[i], ri = r[i];
        double2 pi = p[i];
        if (on[0]) pi.x = fma(beta[0], pi.x, ri.x * di.x);
        if (on[1]) pi.y = fma(beta[1], pi.y, ri.y * di.y);
        p[i] = pi;
    }
}

// Convergence is relative to the larger of the right-hand side and the initial residual
// (which carries the held values): a field already at rest (rounding-level residual)
// takes no iteration.  One thread per field; `norm` as in pcg_tail, ref a lower bound of
// the reference.
__global__ void k_macro_start(double* acc, int nf, int norm, double tol2, int max_iter, double ref) {
    const int f = threadIdx.x;
    const double rj = f < nf ? acc[norm + f] : 0.0, bb = f < nf ? acc[14 + f] : 0.0;
    acc[6 + f] = fmax(fmax(bb, rj), ref);
    acc[10 + f] = rj > tol2 * acc[6 + f] ? 1.0 : 0.0;
    acc[2 + f] = 0.0;
    acc[12 + f] = 0.0;
    if (f == 0) {
        if (norm) {   // the norm is formed again with the preconditioner's start
            acc[24] = pcg_narrow_scale(rj);
            acc[norm] = 0.0;
        }
        acc[16] = 0.0;
        acc[17] = (double)max_iter;
        acc[18] = tol2;
    }
}

// The mechanics' vector passes, with the Chebyshev preconditioner below (POLY) or Jacobi's;
// the norm (r, D^-1 r) at acc[norm], which without the polynomial is (r, z) itself.
//
// r = b - y on free rows (0 on held rows), acc[norm] += (r, D^-1 r) and acc[14] +=
// (b, D^-1 b) over the free rows
__global__ void __launch_bounds__(256) k_mech_residual(int64_t n, const double* __restrict__ b,
                                                       const double* __restrict__ y, const uint8_t* __restrict__ mask,
                                                       const double* __restrict__ dinv, double* __restrict__ r,
                                                       float* __restrict__ dinv32, int norm, double* __restrict__ acc) {
    double a[1] = {0.0}, bb[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const bool held = mask[i] != 0;
        const double bi = b[i], di = dinv[i];
        const double ri = held ? 0.0 : bi - y[i];
        r[i] = ri;
        if (dinv32) dinv32[i] = held ? 0.f : (float)di;   // the polynomial leaves held rows alone
        a[0] = fma(ri, ri * di, a[0]);
        if (!held) bb[0] = fma(bi, bi * di, bb[0]);
    }
    block_add<1>(a, acc + norm);
    block_add<1>(bb, acc + 14);
}

// p = z
template <bool POLY>
__global__ void __launch_bounds__(256) k_mech_first(int64_t n, const float* __restrict__ z, const double* __restrict__ r,
                                                    const double* __restrict__ dinv, double* __restrict__ p) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = POLY ? (double)z[i] : r[i] * dinv[i];
}

// x += alpha p, r -= alpha q (held rows stay 0), acc[norm] += (r, D^-1 r); POLY: the
// preconditioner's start r32 = r, z = w D^-1 r (scaled).  Without a step (alpha 0: at the
// start, or where the iteration breaks down) x and r stay as they are.
template <bool POLY>
__global__ void __launch_bounds__(256) k_mech_update(int64_t n, const uint8_t* __restrict__ mask,
                                                     const double* __restrict__ dinv, double* __restrict__ x,
                                                     double* __restrict__ r, const double* __restrict__ p,
                                                     const double* __restrict__ q, float* __restrict__ r32,
                                                     float* __restrict__ z, const float* __restrict__ dinv32, float w,
                                                     double* __restrict__ acc) {
    __shared__ double alpha, scale;
    if (threadIdx.x == 0) {
        const double pq = acc[2], rz = acc[4];
        const bool sound = pq > 0.0 && isfinite(pq) && rz > 0.0 && isfinite(rz / pq);
        alpha = acc[8] != 0.0 && sound ? rz / pq : 0.0;
        scale = acc[24];
        if (blockIdx.x == 0 && acc[8] != 0.0 && !sound) acc[22] = 1.0;
    }
    __syncthreads();
    const double al = alpha, sc = scale;
    double a[1] = {0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double ri = r[i];
        if (al != 0.0) {
            x[i] = fma(al, p[i], x[i]);
            ri = mask[i] ? 0.0 : fma(-al, q[i], ri);
            r[i] = ri;
        }
        if constexpr (POLY) {
            const float rf = (float)(ri * sc);
            r32[i] = rf;
            z[i] = w * (dinv32[i] * rf);
        }
        a[0] = fma(ri, ri * dinv[i], a[0]);
    }
    block_add<1>(a, acc + (POLY ? 20 : 0));
}

// p = z + beta p; loop control
template <bool POLY>
__global__ void __launch_bounds__(256) k_mech_pupdate(int64_t n, const float* __restrict__ z, const double* __restrict__ r,
                                                      const double* __restrict__ dinv, double* __restrict__ p,
                                                      double* __restrict__ acc, cudaGraphConditionalHandle h) {
    __shared__ double beta[1];
    __shared__ int on[1];
    pcg_tail<1>(acc, POLY ? 20 : 0, h, beta, on);
    if (!on[0]) return;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = fma(beta[0], p[i], POLY ? (double)z[i] : r[i] * dinv[i]);
}

// The elastic solve's preconditioner: a Chebyshev polynomial in D^-1 K evaluated in FP32
// with an FP32 copy of the matrix.  An FP32 product is bound by reading that copy, an
// FP64 one by the FP64 pipe, so the polynomial's products cost less than the FP64
// iterations they replace.  (Not for the transport pair: the equivalent time of a Gauss
// point ahead of the moisture front is a ratio of quantities at the solver's tolerance,
// which another preconditioner leaves elsewhere.)  One kernel per step: d = c1 d_in +
// c2 D^-1 (r - K z), z_new = z + d; the last one adds (r64, z_new) into acc instead of
// storing d.  A warp takes one displacement component of 32 nodes, as the FP64 product.
struct MechCheb {
    const float* z;
    float* z_new;
    const float* d_in;
    float* d_out;
    const float* r;
    const float* dinv;
    const double* r64;
    float c1, c2;
    double* acc;   // null: not the last step
};

__global__ void __launch_bounds__(192) k_mech_cheb(int64_t nv, int64_t n_slices, const int64_t* __restrict__ base,
                                                   const int32_t* __restrict__ col, const float* __restrict__ val,
                                                   MechCheb ch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = warp % 3;
    const int64_t s = (int64_t)blockIdx.x * 2 + warp / 3, i = s * 32 + lane;
    double dot[1] = {0.0};
    if (s < n_slices) {
        const int64_t row1 = base[s + 1];
        float a = 0.f;
#pragma unroll 4
        for (int64_t row = base[s]; row < row1; ++row) {
            const int64_t c = 3 * (int64_t)__ldg(col + row * 32 + lane);
            const float* v = val + (row * 9 + 3 * r) * 32 + lane;
            a = fmaf(__ldg(v), __ldg(ch.z + c), a);
            a = fmaf(__ldg(v + 32), __ldg(ch.z + c + 1), a);
            a = fmaf(__ldg(v + 64), __ldg(ch.z + c + 2), a);
        }
        if (i < nv) {
            const int64_t k = i * 3 + r;
            const float d = fmaf(ch.c1, ch.d_in[k], ch.c2 * (ch.dinv[k] * (ch.r[k] - a)));
            const float zn = ch.z[k] + d;
            ch.z_new[k] = zn;
            if (ch.acc)
                dot[0] = ch.r64[k] * (double)zn;
            else
                ch.d_out[k] = d;
        }
    }
    if (ch.acc) block_add<1>(dot, ch.acc);
}

// Power iteration for the largest eigenvalue of D^-1 K over all rows (held rows can only
// lower it): the step kernel with d_in = r = 0 and c2 = 1 gives d = -D^-1 K x, then
// x = -d / 2; k_power_sums adds (x, K x) and (x, D x).
__global__ void __launch_bounds__(256) k_power_start(int64_t n, const double* __restrict__ dinv, float* __restrict__ x,
                                                     float* __restrict__ zero, float* __restrict__ dinv32) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t h = (uint32_t)i * 2654435761u + 12345u;
        h ^= h >> 15;
        h *= 2246822519u;
        h ^= h >> 13;
        x[i] = (float)(h & 0xffffu) * (1.f / 32768.f) - 1.f;
        zero[i] = 0.f;
        dinv32[i] = (float)dinv[i];
    }
}
__global__ void __launch_bounds__(256) k_power_next(int64_t n, const float* __restrict__ d, float* __restrict__ x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        x[i] = -0.5f * d[i];
}
__global__ void __launch_bounds__(256) k_power_sums(int64_t n, const float* __restrict__ x, const float* __restrict__ d,
                                                    const float* __restrict__ dinv, double* __restrict__ out) {
    double a[2] = {0.0, 0.0};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (dinv[i] > 0.f) {
            const double w = 1.0 / (double)dinv[i];
            a[0] += (double)x[i] * (double)(-d[i]) * w;
            a[1] += (double)x[i] * (double)x[i] * w;
        }
    block_add<2>(a, out);
}

__global__ void k_narrow(int64_t n, const double* __restrict__ a, float* __restrict__ b) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        b[i] = (float)a[i];
}

// held rows take their prescribed values (hold[node * 2 + field])
__global__ void k_macro_hold(int64_t nv, const uint8_t* __restrict__ mask, const double* __restrict__ hold,
                             double* __restrict__ x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x)
        if (mask[i]) {
            x[i * 2] = hold[i * 2];
            x[i * 2 + 1] = hold[i * 2 + 1];
        }
}

// grad psi of one field per tetrahedron (constant on a linear element)
__global__ void k_macro_gradient(int64_t nt, const int32_t* __restrict__ tets, const double* __restrict__ geo,
                                 const double* __restrict__ x, int field, double* __restrict__ out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nt; e += (int64_t)gridDim.x * blockDim.x) {
        const double* g = geo + e * 13 + 1;
        double gr[3] = {0, 0, 0};
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const double v = x[(int64_t)tets[e * 4 + a] * 2 + field];
#pragma unroll
            for (int i = 0; i < 3; ++i) gr[i] += g[a * 3 + i] * v;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) out[e * 3 + i] = gr[i];
    }
}

__global__ void k_macro_fill(int64_t nv, double T, double c, double* __restrict__ x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
        x[i * 2] = T;
        x[i * 2 + 1] = c;
    }
}

// Gauss-point states: gp[k][e*4 + g] for k = T, c, W, t_eq.  W is advanced by
// backward Euler of Eq. Eq_Model_RateForm at the new T and c; t_eq [h] solves
// the closed form for that W.  Where there is no moisture now (lambda = 0: the
// capacity-consistent transport undershoots slightly ahead of the front) t_eq = 0
// hands the point over as undegraded; such points with W < 1 are counted in
// bad[0] and the largest 1 - W among them (the hand-over error) is kept in
// errbits as the bit pattern of a non-negative double.
__global__ void k_macro_gauss(int64_t nt, const int32_t* __restrict__ tets, const double* __restrict__ x,
                              double* __restrict__ Wst, double* __restrict__ gp, double dt_h, double beta,
                              double Tg_C, double c_sat, int advance, int* __restrict__ bad,
                              unsigned long long* __restrict__ errbits) {
    const double A = 0.5854101966249685, Bc = 0.1381966011250105;
    const int64_t n = nt * 4;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / 4;
        const int g = (int)(i % 4);
        double T = 0, c = 0;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const double N = a == g ? A : Bc;
            const int v = tets[e * 4 + a];
            T += N * x[(int64_t)v * 2];
            c += N * x[(int64_t)v * 2 + 1];
        }
        const double cn = fmin(fmax(c / c_sat, 0.0), 1.0);
        const double lam = cn * beta * log(1.0 - (T + kKelvin) / (Tg_C + kKelvin));
        double W = Wst[i];
        if (advance) {
            W = W / (1.0 + dt_h / 24.0 * lam);
            Wst[i] = W;
        }
        double teq = 0.0;
        if (lam > 0.0) {
            teq = -24.0 * log(W) / lam;
        } else if (W < 1.0) {
            atomicAdd(bad, 1);
            atomicMax(errbits, (unsigned long long)__double_as_longlong(1.0 - W));
        }
        gp[i] = T;
        gp[n + i] = c;
        gp[2 * n + i] = W;
        gp[3 * n + i] = teq;
    }
}

// ---------------------------------------------------------- macro mechanics
// Voigt order [xx, yy, zz, xy, yz, zx] with engineering shear, as C_bar of the
// RVE path.  On a linear tetrahedron the strain is constant, so the 4-point
// Gauss rule of K = sum_g |T| / 4 B^T C_g B collapses to |T| B^T (mean_g C_g) B.

// Voigt strain from the displacement gradient H_ij = du_i / dx_j
__device__ __forceinline__ void mech_strain(const double* g, const double* ua, double eps[6]) {
    double H[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) H[i][j] += ua[a * 3 + i] * g[a * 3 + j];
    eps[0] = H[0][0];
    eps[1] = H[1][1];
    eps[2] = H[2][2];
    eps[3] = H[0][1] + H[1][0];
    eps[4] = H[1][2] + H[2][1];
    eps[5] = H[2][0] + H[0][2];
}

// B^T sigma for node a with gradient (gx, gy, gz)
__device__ __forceinline__ void mech_bt(double gx, double gy, double gz, const double* sg, double f[3]) {
    f[0] = gx * sg[0] + gy * sg[3] + gz * sg[5];
    f[1] = gy * sg[1] + gx * sg[3] + gz * sg[4];
    f[2] = gz * sg[2] + gy * sg[4] + gx * sg[5];
}

// Per tetrahedron: cm = mean over its Gauss points of the symmetric part of C_g
__global__ void k_mech_material(int64_t nt, const double* __restrict__ Cgp, double* __restrict__ cm) {
    const int64_t n = nt * 36;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / 36;
        const int J = (int)(i % 36) / 6, K = (int)(i % 36) % 6;
        const double* Cq = Cgp + e * 4 * 36;
        double c = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) c += 0.125 * (Cq[q * 36 + J * 6 + K] + Cq[q * 36 + K * 6 + J]);
        cm[i] = c;
    }
}

// Element form: y += K x, per tetrahedron eps = B x_T, sigma = cm eps, y_a += |T| B_a^T sigma
__global__ void __launch_bounds__(256) k_mech_apply(int64_t nt, const int32_t* __restrict__ tets,
                                                    const double* __restrict__ geo, const double* __restrict__ cm,
                                                    const double* __restrict__ x, double* __restrict__ y) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nt; e += (int64_t)gridDim.x * blockDim.x) {
        int v[4];
        double ua[12], eps[6], sg[6];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = tets[e * 4 + a];
#pragma unroll
            for (int i = 0; i < 3; ++i) ua[a * 3 + i] = x[(int64_t)v[a] * 3 + i];
        }
        const double vol = geo[e * 13];
        const double* g = geo + e * 13 + 1;
        mech_strain(g, ua, eps);
        const double* C = cm + e * 36;
#pragma unroll
        for (int J = 0; J < 6; ++J) {
            double t = 0.0;
#pragma unroll
            for (int K = 0; K < 6; ++K) t = fma(C[J * 6 + K], eps[K], t);
            sg[J] = vol * t;
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            double f[3];
            mech_bt(g[a * 3], g[a * 3 + 1], g[a * 3 + 2], sg, f);
#pragma unroll
            for (int i = 0; i < 3; ++i) atomicAdd(y + (int64_t)v[a] * 3 + i, f[i]);
        }
    }
}

// its diagonal |T| b^T cm b (b the DOF's column of B), added into d
__global__ void __launch_bounds__(256) k_mech_diag(int64_t nt, const int32_t* __restrict__ tets,
                                                   const double* __restrict__ geo, const double* __restrict__ cm,
                                                   double* __restrict__ d) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nt * 4; k += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = k >> 2;
        const double vol = geo[e * 13];
        const double* g = geo + e * 13 + 1 + (k & 3) * 3;
        const double* C = cm + e * 36;
        for (int i = 0; i < 3; ++i) {
            double b[6] = {0, 0, 0, 0, 0, 0}, t = 0.0;
            b[i] = g[i];
            b[i == 2 ? 5 : 3] = i == 0 ? g[1] : g[0];
            b[i == 0 ? 5 : 4] = i == 2 ? g[1] : g[2];
            for (int J = 0; J < 6; ++J)
                for (int K = 0; K < 6; ++K) t += b[J] * C[J * 6 + K] * b[K];
            atomicAdd(d + (int64_t)tets[k] * 3 + i, vol * t);
        }
    }
}

// The assembled stiffness: 3 x 3 blocks sum_T |T| B_a^T cm B_b of every entry, stored
// val[(ell row * 9 + 3 r + c) * 32 + lane] (block row r), and the inverse Jacobi
// diagonal.  One thread per (ELL row of the slice, lane).
__global__ void __launch_bounds__(256) k_mech_entries(int64_t nv, const int64_t* __restrict__ base,
                                                      const int32_t* __restrict__ col,
                                                      const int32_t* __restrict__ len,
                                                      const int32_t* __restrict__ eptr,
                                                      const int32_t* __restrict__ inc,
                                                      const int32_t* __restrict__ tets,
                                                      const double* __restrict__ geo, const double* __restrict__ cm,
                                                      double* __restrict__ val, double* __restrict__ dinv) {
    const int lane = threadIdx.x & 31;
    const int64_t s = blockIdx.x, i = s * 32 + lane, row0 = base[s], row1 = base[s + 1];
    const int n_len = i < nv ? len[i] : 0;
    for (int64_t row = row0 + (threadIdx.x >> 5); row < row1; row += blockDim.x >> 5) {
        double A[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) A[k] = 0.0;
        int c = -1;
        if (row - row0 < n_len) {
            c = col[row * 32 + lane];
            for (int q = eptr[i]; q < eptr[i + 1]; ++q) {
                const int e = inc[q] >> 2, a = inc[q] & 3;
                for (int b = 0; b < 4; ++b) {
                    if (tets[(int64_t)e * 4 + b] != c) continue;
                    const double vol = geo[(int64_t)e * 13];
                    const double* ga = geo + (int64_t)e * 13 + 1 + a * 3;
                    const double* gb = geo + (int64_t)e * 13 + 1 + b * 3;
                    const double* C = cm + (int64_t)e * 36;
                    const double gx = vol * gb[0], gy = vol * gb[1], gz = vol * gb[2];
#pragma unroll
                    for (int d = 0; d < 3; ++d) {
                        // |T| C times the strain of the unit displacement d of node b
                        double sg[6], f[3];
#pragma unroll
                        for (int J = 0; J < 6; ++J)
                            sg[J] = d == 0   ? C[J * 6] * gx + C[J * 6 + 3] * gy + C[J * 6 + 5] * gz
                                    : d == 1 ? C[J * 6 + 1] * gy + C[J * 6 + 3] * gx + C[J * 6 + 4] * gz
                                             : C[J * 6 + 2] * gz + C[J * 6 + 4] * gy + C[J * 6 + 5] * gx;
                        mech_bt(ga[0], ga[1], ga[2], sg, f);
#pragma unroll
                        for (int r = 0; r < 3; ++r) A[3 * r + d] += f[r];
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 9; ++k) val[(row * 9 + k) * 32 + lane] = A[k];
        if (c == i)
#pragma unroll
            for (int r = 0; r < 3; ++r) dinv[i * 3 + r] = 1.0 / A[4 * r];
    }
}

// y = K x and (x, y) into acc[2] (norm: as in pcg_tail).  A warp takes one of the three displacement
// components of a slice's 32 nodes (three warps share the slice's column indices and
// gathered values in L1): three times the warps of one lane per node, which is what
// covers the latency of the gathers.  Bound by the FP64 pipe.  acc null: the product
// alone.
constexpr int MECH_THREADS = 192;
__global__ void __launch_bounds__(MECH_THREADS) k_mech_product(int64_t nv, int64_t n_slices,
                                                               const int64_t* __restrict__ base,
                                                               const int32_t* __restrict__ col,
                                                               const double* __restrict__ val,
                                                               const double* __restrict__ x, double* __restrict__ y,
                                                               int norm, double* __restrict__ acc) {
    if (acc && blockIdx.x == 0 && threadIdx.x == 0) {
        if (norm) acc[24] = pcg_narrow_scale(acc[norm]);
        pcg_roll(acc, 0);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = warp % 3;
    double dot[1] = {0.0};
    for (int64_t s = (int64_t)blockIdx.x * (MECH_THREADS / 96) + warp / 3; s < n_slices;
         s += (int64_t)gridDim.x * (MECH_THREADS / 96)) {
        const int64_t i = s * 32 + lane, row1 = base[s + 1];
        double a = 0.0;
#pragma unroll 4
        for (int64_t row = base[s]; row < row1; ++row) {
            const int64_t c = 3 * (int64_t)col[row * 32 + lane];
            const double* v = val + (row * 9 + 3 * r) * 32 + lane;
            a = fma(v[0], x[c], a);
            a = fma(v[32], x[c + 1], a);
            a = fma(v[64], x[c + 2], a);
        }
        if (i < nv) {
            y[i * 3 + r] = a;
            dot[0] = fma(x[i * 3 + r], a, dot[0]);
        }
    }
    if (acc) block_add<1>(dot, acc + 2);
}

// Consistent nodal forces of a uniform traction t on every tetrahedron face
// whose three vertices are all marked: t |F| / 3 on each, with the face area
// |F_a| = 3 |T| |grad lambda_a| of the face opposite vertex a.
__global__ void k_mech_traction(int64_t nt, const int32_t* __restrict__ tets, const double* __restrict__ geo,
                                const uint8_t* __restrict__ face, double tx, double ty, double tz,
                                double* __restrict__ f) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nt; e += (int64_t)gridDim.x * blockDim.x) {
        int v[4];
        bool on[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            v[a] = tets[e * 4 + a];
            on[a] = face[v[a]] != 0;
        }
        const double vol = geo[e * 13];
        const double* g = geo + e * 13 + 1;
        for (int a = 0; a < 4; ++a) {
            bool all = true;
            for (int k = 0; k < 4; ++k)
                if (k != a) all = all && on[k];
            if (!all) continue;
            const double gx = g[a * 3], gy = g[a * 3 + 1], gz = g[a * 3 + 2];
            const double third = vol * sqrt(gx * gx + gy * gy + gz * gz);   // |F_a| / 3
            for (int k = 0; k < 4; ++k)
                if (k != a) {
                    atomicAdd(f + (int64_t)v[k] * 3, tx * third);
                    atomicAdd(f + (int64_t)v[k] * 3 + 1, ty * third);
                    atomicAdd(f + (int64_t)v[k] * 3 + 2, tz * third);
                }
        }
    }
}

// held DOFs take their prescribed values
__global__ void k_mech_hold(int64_t n, const uint8_t* __restrict__ fix, const double* __restrict__ val,
                            double* __restrict__ x) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (fix[i]) x[i] = val[i];
}

// sigma_g = sym(C_g) B u_T at every Gauss point [nt*4][6]
__global__ void k_mech_stress(int64_t nt, const int32_t* __restrict__ tets, const double* __restrict__ geo,
                              const double* __restrict__ Cgp, const double* __restrict__ u,
                              double* __restrict__ sig) {
    const int64_t n = nt * 4;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t e = i / 4;
        double ua[12];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int k = 0; k < 3; ++k) ua[a * 3 + k] = u[(int64_t)tets[e * 4 + a] * 3 + k];
        double eps[6];
        mech_strain(geo + e * 13 + 1, ua, eps);
        const double* C = Cgp + i * 36;
#pragma unroll
        for (int J = 0; J < 6; ++J) {
            double t = 0.0;
#pragma unroll
            for (int K = 0; K < 6; ++K) t += 0.5 * (C[J * 6 + K] + C[K * 6 + J]) * eps[K];
            sig[i * 6 + J] = t;
        }
    }
}

unsigned grid_for(int64_t n) {
    int64_t b = (n + 255) / 256;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, (int64_t)sm_count() * 4));
}

bool sym_pos_def(const double k[9]) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            if (std::fabs(k[i * 3 + j] - k[j * 3 + i]) > 1e-12 * (std::fabs(k[i * 3 + j]) + std::fabs(k[j * 3 + i])))
                return false;
    const double d1 = k[0];
    const double d2 = k[0] * k[4] - k[1] * k[3];
    const double d3 = k[0] * (k[4] * k[8] - k[5] * k[7]) - k[1] * (k[3] * k[8] - k[5] * k[6]) +
                      k[2] * (k[3] * k[7] - k[4] * k[6]);
    return d1 > 0 && d2 > 0 && d3 > 0;
}

void to_sym6(const double k[9], double out[6]) {
    out[0] = k[0];
    out[1] = k[4];
    out[2] = k[8];
    out[3] = k[1];
    out[4] = k[5];
    out[5] = k[2];
}

// Whether the matrices' share may grow by so many bytes: a quarter of the free memory, since
// results and the caller want room too.
int room_for(rve_macro m, size_t bytes) {
    size_t room = m->mat_limit, all = 0;
    if (room == 0) {
        room = (size_t)1 << 30;   // (the query takes up to a millisecond: not for small matrices)
        if (bytes > room) {
            RVE_CUDA(cudaMemGetInfo(&room, &all));
            room /= 4;
        }
    }
    if (bytes <= room) return RVE_OK;
    set_error("no room for the macro mesh's matrices");
    return RVE_ERR_OUT_OF_MEMORY;
}

// Node graph of the mesh in slices of 32 rows, on the device (once per mesh).
// RVE_ERR_OUT_OF_MEMORY where it does not fit, in memory or in 32-bit indices, or where a
// node couples to so many others that the slices are mostly padding.
int ensure_graph(rve_macro m) {
    if (m->have_graph) return RVE_OK;
    NodeGraph g;
    if (!build_node_graph(m->tets_h.data(), m->nt, 4, nullptr, m->nv, g)) {
        set_error("macro mesh too large for 32-bit matrix indices");
        return RVE_ERR_OUT_OF_MEMORY;
    }
    const int64_t ns = (m->nv + 31) / 32;
    std::vector<int64_t> base(ns + 1, 0);
    std::vector<int32_t> len(m->nv);
    for (int64_t i = 0; i < m->nv; ++i) len[i] = g.ptr[i + 1] - g.ptr[i];
    for (int64_t s = 0; s < ns; ++s) {
        int32_t most = 0;
        for (int64_t i = s * 32; i < std::min(m->nv, s * 32 + 32); ++i) most = std::max(most, len[i]);
        base[s + 1] = base[s] + most;
    }
    if (base[ns] * 32 > 4 * (int64_t)g.col.size() + 4096) {
        set_error("a node of the macro mesh couples to too many others");
        return RVE_ERR_OUT_OF_MEMORY;
    }
    RVE_TRY(room_for(m, (size_t)base[ns] * 32 * 4 + (size_t)m->nt * 16));
    std::vector<int32_t> col((size_t)base[ns] * 32);
    for (int64_t s = 0; s < ns; ++s)
        for (int lane = 0; lane < 32; ++lane) {
            const int64_t i = std::min(s * 32 + lane, m->nv - 1);
            for (int64_t k = 0; k < base[s + 1] - base[s]; ++k)
                col[(base[s] + k) * 32 + lane] = k < len[i] ? g.col[g.ptr[i] + k] : (int32_t)i;
        }
    cudaStream_t s = m->ctx->stream;
    RVE_TRY(upload(m->g_base, base.data(), base.size(), s));
    RVE_TRY(upload(m->g_col, col.data(), col.size(), s));
    RVE_TRY(upload(m->g_len, len.data(), len.size(), s));
    RVE_TRY(upload(m->g_eptr, g.eptr.data(), g.eptr.size(), s));
    RVE_TRY(upload(m->g_inc, g.inc.data(), g.inc.size(), s));
    RVE_CUDA(cudaStreamSynchronize(s));
    m->n_slices = ns;
    m->n_ell = base[ns];
    m->have_graph = true;
    return RVE_OK;
}

// From here on the operators are applied element by element, as in a call that needs the
// matrices and finds no room for them.
int apply_element_form(rve_macro m) {
    cudaGetLastError();
    RVE_CUDA(cudaStreamSynchronize(m->ctx->stream));
    for (DevBuf* b : {&m->g_base, &m->g_col, &m->g_len, &m->g_eptr, &m->g_inc, &m->t_mass, &m->t_stiff, &m->t_mat,
                      &m->mmat, &m->mmat32})
        b->release();
    for (auto& l : m->loop)   // (their captured launches hold pointers that the keys do not list)
        if (l.exec) {
            cudaGraphExecDestroy(l.exec);
            l.exec = nullptr;
        }
    m->have_graph = m->have_stiff = false;
    m->element_form = true;
    m->mat_dt = -1;
    return RVE_OK;
}

// The transport matrix and inverse diagonal for one time step length.
int ensure_transport_matrix(rve_macro m, double dt_s) {
    RVE_TRY(ensure_graph(m));
    cudaStream_t s = m->ctx->stream;
    if (!m->have_stiff && m->t_mat.bytes < (size_t)m->n_ell * 32 * 16) RVE_TRY(room_for(m, (size_t)m->n_ell * 32 * 40));
    const int64_t *base = m->g_base.as<int64_t>();
    const int32_t *col = m->g_col.as<int32_t>(), *len = m->g_len.as<int32_t>();
    if (!m->have_stiff) {
        RVE_TRY(m->t_mass.ensure((size_t)m->n_ell * 32 * 8));
        RVE_TRY(m->t_stiff.ensure((size_t)m->n_ell * 32 * 16));
        RVE_TRY(m->t_mat.ensure((size_t)m->n_ell * 32 * 16));
        RVE_TRY(m->t_dinv.ensure((size_t)m->nv * 16));
        RVE_CUDA(cudaMemsetAsync(m->t_dinv.p, 0, (size_t)m->nv * 16, s));   // nodes of no element: z = 0
        TransportTensors prm;
        std::memcpy(prm.KT, m->KT, sizeof(prm.KT));
        std::memcpy(prm.Dc, m->Dc, sizeof(prm.Dc));
        k_transport_entries<<<(unsigned)m->n_slices, 256, 0, s>>>(m->nv, base, col, len, m->g_eptr.as<int32_t>(),
                                                                  m->g_inc.as<int32_t>(), m->tets.as<int32_t>(),
                                                                  m->geo.as<double>(), prm, m->t_mass.as<double>(),
                                                                  m->t_stiff.as<double2>());
        RVE_CUDA(cudaGetLastError());
        m->have_stiff = true;
        m->mat_dt = -1;
    }
    if (m->mat_dt != dt_s) {
        k_transport_matrix<<<(unsigned)((m->n_slices + 7) / 8), 256, 0, s>>>(
            m->nv, m->n_slices, base, col, len, m->t_mass.as<double>(), m->t_stiff.as<double2>(), m->rho_cp / dt_s,
            1.0 / dt_s, m->t_mat.as<double2>(), m->t_dinv.as<double2>());
        RVE_CUDA(cudaGetLastError());
        m->mat_dt = dt_s;
    }
    return RVE_OK;
}

// Room for the elastic matrix in both precisions and the preconditioner's vectors.
int ensure_mech_matrix(rve_macro m) {
    RVE_TRY(ensure_graph(m));
    const size_t e = (size_t)m->n_ell * 9 * 32;
    if (m->mmat.bytes < e * 8 || m->mmat32.bytes < e * 4) RVE_TRY(room_for(m, e * 12));
    RVE_TRY(m->mmat.ensure(e * 8));
    RVE_TRY(m->mmat32.ensure(e * 4));
    for (DevBuf* b : {&m->c_r, &m->c_z, &m->c_z2, &m->c_d, &m->c_dinv}) RVE_TRY(b->ensure((size_t)m->nv * 12));
    return RVE_OK;
}

// The PCG iterations of one problem (slot 0 transport, 1 mechanics) as a CUDA graph with
// a conditional WHILE node that ends on the device: body(stream, handle) launches one
// iteration.  The instantiated graph is kept while `key`, every captured pointer and
// number, stays the same.  Then the iterations and final relative residuals per field, the
// first one's reference norm, and whether the iteration broke down.
template <class Body>
int macro_loop(rve_macro mm, int slot, const void* key, size_t key_bytes, int nf, int norm, Body body, int its[2],
               double rel[2], bool& conv, double* ref = nullptr, bool* broke = nullptr) {
    cudaStream_t s = mm->ctx->stream;
    const unsigned char* kb = static_cast<const unsigned char*>(key);
    auto& loop = mm->loop[slot];
    if (!loop.exec || loop.key.size() != key_bytes || std::memcmp(loop.key.data(), kb, key_bytes) != 0) {
        if (loop.exec) {
            cudaGraphExecDestroy(loop.exec);
            loop.exec = nullptr;
        }
        cudaGraph_t graph = nullptr;
        RVE_CUDA(cudaGraphCreate(&graph, 0));
        struct GraphGuard {
            cudaGraph_t g;
            ~GraphGuard() { cudaGraphDestroy(g); }
        } guard{graph};
        cudaGraphConditionalHandle handle;
        RVE_CUDA(cudaGraphConditionalHandleCreate(&handle, graph, 1, cudaGraphCondAssignDefault));
        cudaGraphNodeParams np = {};
        np.type = cudaGraphNodeTypeConditional;
        np.conditional.handle = handle;
        np.conditional.type = cudaGraphCondTypeWhile;
        np.conditional.size = 1;
        cudaGraphNode_t node;
        RVE_CUDA(cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &np));
        cudaGraph_t inner = np.conditional.phGraph_out[0];
        cudaStream_t cap = mm->ctx->capture;
        RVE_CUDA(cudaStreamBeginCaptureToGraph(cap, inner, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal));
        body(cap, handle);
        RVE_CUDA(cudaStreamEndCapture(cap, &inner));
        RVE_CUDA(cudaGraphInstantiate(&loop.exec, graph, 0));
        loop.key.assign(kb, kb + key_bytes);
    }
    RVE_CUDA(cudaGraphLaunch(loop.exec, s));
    double h[PCG_SCALARS];
    RVE_CUDA(cudaMemcpyAsync(h, mm->acc.p, sizeof(h), cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    conv = true;
    for (int f = 0; f < 2; ++f) {
        its[f] = f < nf ? (int)h[12 + f] : 0;
        rel[f] = f < nf && h[6 + f] > 0 ? std::sqrt(std::max(h[norm + f], 0.0) / h[6 + f]) : 0.0;
        // (a field also stops where its residual is not finite or the iteration broke down)
        if (f < nf && (h[10 + f] != 0.0 || !std::isfinite(h[norm + f]))) conv = false;
    }
    if (h[22] != 0.0 || h[23] != 0.0) conv = false;
    if (ref) *ref = h[6];
    if (broke) *broke = h[22] != 0.0 || h[23] != 0.0;
    return RVE_OK;
}

// Polynomial of the elastic solve's preconditioner: it covers [lambda / ratio, lambda]
// of the spectrum with the odd degree next to sqrt(ratio).  Measured on the 200 x 40 x 10 plate
// (degree, ratio: ms for solve and results), the rule's choice first: 39, 1500: 27.1; 33, 1500:
// 27.3; 33, 1000: 28.1; 25, 600: 29.0; 51, 2500: 26.5.  The condition number grows with the square
// of the nodes along the longest side, at most as the 2/3 power of their number for a cube.
double mech_cheb_ratio(int64_t nv) { return std::min(1500.0, std::max(10.0, 0.75 * std::pow((double)nv, 2.0 / 3.0))); }

// Estimate of the largest eigenvalue of D^-1 K by power iteration with the preconditioner's
// step kernel, rounded up to eighths (the quotient approaches the eigenvalue from below,
// and the captured loop's coefficients then stay the same from solve to solve).
template <class Step>
int mech_spectrum(rve_macro m, int64_t n, Step step, double& lambda) {
    cudaStream_t s = m->ctx->stream;
    const unsigned g = grid_for(n);
    float *x = m->c_z.as<float>(), *d = m->c_d.as<float>(), *zero = m->c_r.as<float>(), *dinv = m->c_dinv.as<float>();
    double* acc = m->acc.as<double>();
    RVE_CUDA(cudaMemsetAsync(acc, 0, 2 * 8, s));
    k_power_start<<<g, 256, 0, s>>>(n, m->mdinv.as<double>(), x, zero, dinv);
    const int steps = 30;
    for (int k = 0; k <= steps; ++k) {
        step(s, MechCheb{x, m->c_z2.as<float>(), zero, d, zero, dinv, nullptr, 0.f, 1.f, nullptr});
        if (k < steps) k_power_next<<<g, 256, 0, s>>>(n, d, x);
    }
    k_power_sums<<<g, 256, 0, s>>>(n, x, d, dinv, acc);
    double h[2];
    RVE_CUDA(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    const double q = h[1] > 0.0 ? h[0] / h[1] : 0.0;
    lambda = std::isfinite(q) && q > 0.0 ? std::ceil(8.0 * 1.1 * q) / 8.0 : 12.0;
    return RVE_OK;
}

// FP64 PCG of the elastic problem: converged when (r, D^-1 r) <= rtol^2 max((f, D^-1 f),
// (r0, D^-1 r0)) over the free rows.  The polynomial preconditioner is evaluated in FP32;
// where that breaks down (a stiffness outside FP32's range, 1e-38 to 1e38, makes
// it so) the Jacobi iteration, all in FP64, takes over from the displacements reached.
// product(stream, in, out, norm, acc) forms out = K in and adds (in, out) to acc[2].
template <class Product, class Step>
int mech_pcg(rve_macro mm, int64_t n, double* x, const double* b, Product product, Step step, double rtol,
             int max_iter, int its[2], double rel[2], bool& conv) {
    cudaStream_t s = mm->ctx->stream;
    const bool with_poly = !mm->element_form;   // (which has no FP32 matrix)
    double lambda = 1.0;
    if (with_poly) RVE_TRY(mech_spectrum(mm, n, step, lambda));
    double *r = mm->r.as<double>(), *p = mm->p.as<double>(), *q = mm->q.as<double>(), *acc = mm->acc.as<double>();
    float *r32 = mm->c_r.as<float>(), *zb[2] = {mm->c_z.as<float>(), mm->c_z2.as<float>()};
    float *d = mm->c_d.as<float>(), *dinv32 = mm->c_dinv.as<float>();
    const uint8_t* mask = mm->mfix.as<uint8_t>();
    const double* dinv = mm->mdinv.as<double>();
    const unsigned gv = grid_for(n);
    const ChebPoly poly = chebyshev(lambda, mech_cheb_ratio(mm->nv));
    const float w = (float)poly.w;
    const int n_steps = (int)poly.steps.size();
    // z = M^-1 r from z = w D^-1 r; returns the buffer that holds it
    auto precondition = [&](cudaStream_t st) -> const float* {
        for (int k = 0; k < n_steps; ++k)
            step(st, MechCheb{zb[k & 1], zb[(k & 1) ^ 1], k == 0 ? zb[0] : d, d, r32, dinv32, r, poly.steps[k].first,
                              poly.steps[k].second, k + 1 == n_steps ? acc : nullptr});
        return zb[n_steps & 1];
    };
    struct Key {
        const void* ptr[15];
        double lambda;
    } key;
    std::memset(&key, 0, sizeof(key));
    const void* ptrs[15] = {r,   p,   q,     acc,   x, mask,         dinv,    mm->mmat.p, mm->g_col.p,
                            r32, zb[0], zb[1], d, mm->mmat32.p, mm->cm.p};
    std::memcpy(key.ptr, ptrs, sizeof(ptrs));
    double ref = 0.0;
    bool broke = true;
    int before = 0;
    if (with_poly) {
        RVE_CUDA(cudaMemsetAsync(acc, 0, PCG_SCALARS * 8, s));
        product(s, x, q, 20, nullptr);
        k_mech_residual<<<gv, 256, 0, s>>>(n, b, q, mask, dinv, r, dinv32, 20, acc);
        k_macro_start<<<1, 2, 0, s>>>(acc, 1, 20, rtol * rtol, max_iter, 0.0);
        k_mech_update<true><<<gv, 256, 0, s>>>(n, mask, dinv, x, r, p, q, r32, zb[0], dinv32, w, acc);
        k_mech_first<true><<<gv, 256, 0, s>>>(n, precondition(s), r, dinv, p);
        RVE_CUDA(cudaGetLastError());
        key.lambda = lambda;
        RVE_TRY(macro_loop(mm, 1, &key, sizeof(key), 1, 20, [&](cudaStream_t cap, cudaGraphConditionalHandle h) {
            product(cap, p, q, 20, acc);
            k_mech_update<true><<<gv, 256, 0, cap>>>(n, mask, dinv, x, r, p, q, r32, zb[0], dinv32, w, acc);
            k_mech_pupdate<true><<<gv, 256, 0, cap>>>(n, precondition(cap), r, dinv, p, acc, h);
        }, its, rel, conv, &ref, &broke));
        if (!broke || its[0] >= max_iter) return RVE_OK;
        before = its[0];
    }
    RVE_CUDA(cudaMemsetAsync(acc, 0, PCG_SCALARS * 8, s));
    product(s, x, q, 0, nullptr);
    k_mech_residual<<<gv, 256, 0, s>>>(n, b, q, mask, dinv, r, nullptr, 0, acc);
    k_macro_start<<<1, 2, 0, s>>>(acc, 1, 0, rtol * rtol, max_iter - before, ref);
    k_mech_first<false><<<gv, 256, 0, s>>>(n, nullptr, r, dinv, p);
    RVE_CUDA(cudaGetLastError());
    key.lambda = 0.0;
    RVE_TRY(macro_loop(mm, 2, &key, sizeof(key), 1, 0, [&](cudaStream_t cap, cudaGraphConditionalHandle h) {
        product(cap, p, q, 0, acc);
        k_mech_update<false><<<gv, 256, 0, cap>>>(n, mask, dinv, x, r, p, q, nullptr, nullptr, nullptr, 0.f, acc);
        k_mech_pupdate<false><<<gv, 256, 0, cap>>>(n, nullptr, r, dinv, p, acc, h);
    }, its, rel, conv));
    its[0] += before;
    return RVE_OK;
}

// FP64 Jacobi PCG of the transport pair; per field converged when (r, D^-1 r) <=
// rtol^2 max((b, D^-1 b), (r0, D^-1 r0)) over the free nodes.
template <class Product>
int transport_pcg(rve_macro mm, double2* x, const double2* b, Product product, double dt_key, double rtol,
                  int max_iter, int its[2], double rel[2], bool& conv) {
    cudaStream_t s = mm->ctx->stream;
    double2 *r = mm->r.as<double2>(), *p = mm->p.as<double2>(), *q = mm->q.as<double2>();
    double* acc = mm->acc.as<double>();
    const uint8_t* mask = mm->mask.as<uint8_t>();
    const double2* dinv = mm->t_dinv.as<double2>();
    const int64_t nv = mm->nv;
    const unsigned gv = grid_for(nv);
    RVE_CUDA(cudaMemsetAsync(acc, 0, PCG_SCALARS * 8, s));
    product(s, x, q, nullptr);
    k_transport_residual<<<gv, 256, 0, s>>>(nv, b, q, mask, dinv, r, p, acc);
    k_macro_start<<<1, 2, 0, s>>>(acc, 2, 0, rtol * rtol, max_iter, 0.0);
    RVE_CUDA(cudaGetLastError());
    struct Key {
        const void* ptr[9];
        double dt, tensors[13];
    } key;
    std::memset(&key, 0, sizeof(key));
    const void* ptrs[9] = {r, p, q, acc, x, mask, dinv, mm->t_mat.p, mm->g_col.p};
    std::memcpy(key.ptr, ptrs, sizeof(ptrs));
    if (mm->element_form) {   // (numbers that the element form's product captures)
        key.dt = dt_key;
        std::memcpy(key.tensors, mm->KT, sizeof(mm->KT));
        std::memcpy(key.tensors + 6, mm->Dc, sizeof(mm->Dc));
        key.tensors[12] = mm->rho_cp;
    }
    return macro_loop(mm, 0, &key, sizeof(key), 2, 0, [&](cudaStream_t cap, cudaGraphConditionalHandle h) {
        product(cap, p, q, acc);
        k_transport_update<<<gv, 256, 0, cap>>>(nv, mask, dinv, x, r, p, q, acc);
        k_transport_pupdate<<<gv, 256, 0, cap>>>(nv, dinv, r, p, acc, h);
    }, its, rel, conv);
}

}  // namespace
}  // namespace rve

using namespace rve;

extern "C" {

int rve_macro_create(rve_ctx c, const double* xyz, int64_t nv, const int32_t* tets, int64_t nt, rve_macro* out) {
    RVE_TRY(check_ctx(c));
    if (!xyz || !tets || !out || nv < 4 || nt < 1) {
        set_error("rve_macro_create: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    rve_macro m = new rve_macro_s();
    m->ctx = c;
    m->nv = nv;
    m->nt = nt;
    m->tets_h.assign(tets, tets + nt * 4);
    std::vector<double> geo((size_t)nt * 13);
    for (int64_t e = 0; e < nt; ++e) {
        const double* X[4];
        for (int a = 0; a < 4; ++a) {
            const int32_t v = tets[e * 4 + a];
            if (v < 0 || v >= nv) {
                delete m;
                set_error("rve_macro_create: vertex index out of range");
                return RVE_ERR_BAD_MESH;
            }
            X[a] = xyz + (int64_t)v * 3;
        }
        double J[3][3];   // rows: edges from vertex 0
        for (int r = 0; r < 3; ++r)
            for (int k = 0; k < 3; ++k) J[r][k] = X[r + 1][k] - X[0][k];
        const double det = J[0][0] * (J[1][1] * J[2][2] - J[1][2] * J[2][1]) -
                           J[0][1] * (J[1][0] * J[2][2] - J[1][2] * J[2][0]) +
                           J[0][2] * (J[1][0] * J[2][1] - J[1][1] * J[2][0]);
        if (!(det > 0)) {
            delete m;
            set_error("rve_macro_create: non-positive tetrahedron volume");
            return RVE_ERR_BAD_MESH;
        }
        // inverse of J: grad lambda_{r+1} is row r of inv(J)^T, i.e. column r of inv(J)
        double inv[3][3];
        inv[0][0] = (J[1][1] * J[2][2] - J[1][2] * J[2][1]) / det;
        inv[0][1] = (J[0][2] * J[2][1] - J[0][1] * J[2][2]) / det;
        inv[0][2] = (J[0][1] * J[1][2] - J[0][2] * J[1][1]) / det;
        inv[1][0] = (J[1][2] * J[2][0] - J[1][0] * J[2][2]) / det;
        inv[1][1] = (J[0][0] * J[2][2] - J[0][2] * J[2][0]) / det;
        inv[1][2] = (J[0][2] * J[1][0] - J[0][0] * J[1][2]) / det;
        inv[2][0] = (J[1][0] * J[2][1] - J[1][1] * J[2][0]) / det;
        inv[2][1] = (J[0][1] * J[2][0] - J[0][0] * J[2][1]) / det;
        inv[2][2] = (J[0][0] * J[1][1] - J[0][1] * J[1][0]) / det;
        double g[4][3];
        for (int r = 0; r < 3; ++r)
            for (int k = 0; k < 3; ++k) g[r + 1][k] = inv[k][r];
        for (int k = 0; k < 3; ++k) g[0][k] = -(g[1][k] + g[2][k] + g[3][k]);
        geo[(size_t)e * 13] = det / 6.0;
        for (int a = 0; a < 4; ++a)
            for (int k = 0; k < 3; ++k) geo[(size_t)e * 13 + 1 + a * 3 + k] = g[a][k];
    }
    cudaStream_t s = c->stream;
    int rc = upload(m->tets, tets, (size_t)nt * 4, s);
    if (rc == RVE_OK) rc = upload(m->geo, geo.data(), geo.size(), s);
    const size_t n2 = (size_t)nv * 2;
    for (DevBuf* bfr : {&m->x, &m->b, &m->r, &m->p, &m->q})
        if (rc == RVE_OK) rc = bfr->ensure(n2 * 8);
    if (rc == RVE_OK) rc = m->acc.ensure(PCG_SCALARS * 8);
    if (rc == RVE_OK) rc = m->gp.ensure((size_t)nt * 4 * 4 * 8);
    if (rc == RVE_OK) rc = m->W.ensure((size_t)nt * 4 * 8);
    if (rc == RVE_OK) rc = m->flags.ensure(16);
    if (rc == RVE_OK && cudaStreamSynchronize(s) != cudaSuccess) {
        set_error("rve_macro_create: upload failed");
        rc = RVE_ERR_CUDA;
    }
    if (rc != RVE_OK) {
        delete m;
        return rc;
    }
    *out = m;
    return RVE_OK;
}

int rve_macro_free(rve_ctx c, rve_macro m) {
    RVE_TRY(check_ctx(c));
    if (m) cudaStreamSynchronize(c->stream);
    delete m;
    return RVE_OK;
}

int rve_macro_set_transport(rve_ctx c, rve_macro m, const double K_T[9], double rho_cp, const double D_c[9]) {
    RVE_TRY(check_ctx(c));
    if (!m || !K_T || !D_c || !(rho_cp > 0)) {
        set_error("rve_macro_set_transport: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    if (!sym_pos_def(K_T) || !sym_pos_def(D_c)) {
        set_error("rve_macro_set_transport: conductivity or diffusivity not symmetric positive definite");
        return RVE_ERR_NOT_SPD;
    }
    to_sym6(K_T, m->KT);
    to_sym6(D_c, m->Dc);
    m->rho_cp = rho_cp;
    m->have_transport = true;
    m->have_stiff = false;
    return RVE_OK;
}

int rve_macro_set_face(rve_ctx c, rve_macro m, const uint8_t* node_mask, double T_C, double c_wt) {
    RVE_TRY(check_ctx(c));
    if (!m || !node_mask) {
        set_error("rve_macro_set_face: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    std::vector<double> hold((size_t)m->nv * 2);
    for (int64_t i = 0; i < m->nv; ++i) {
        hold[(size_t)i * 2] = T_C;
        hold[(size_t)i * 2 + 1] = c_wt;
    }
    return rve_macro_set_held(c, m, node_mask, hold.data());
}

int rve_macro_set_held(rve_ctx c, rve_macro m, const uint8_t* node_mask, const double* values) {
    RVE_TRY(check_ctx(c));
    if (!m || !node_mask || !values) {
        set_error("rve_macro_set_held: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    RVE_TRY(upload(m->mask, node_mask, (size_t)m->nv, c->stream));
    RVE_TRY(upload(m->hold, values, (size_t)m->nv * 2, c->stream));
    RVE_CUDA(cudaStreamSynchronize(c->stream));
    m->have_face = true;
    return RVE_OK;
}

int rve_macro_reset(rve_ctx c, rve_macro m, double T0_C, double c0_wt) {
    RVE_TRY(check_ctx(c));
    if (!m) {
        set_error("rve_macro_reset: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t s = c->stream;
    k_macro_fill<<<grid_for(m->nv), 256, 0, s>>>(m->nv, T0_C, c0_wt, m->x.as<double>());
    launch_fill(m->nt * 4, 1.0, m->W.as<double>(), s);
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_state = true;
    return RVE_OK;
}

// One implicit transport solve over both fields: (C/dt + K) x' = C/dt x with the
// held rows at their values; dt_s = infinity gives the steady problem K x = 0.
// Returns the iterations and final relative residuals per field.
static int transport_solve(rve_macro mm, double dt_s, double rtol, int max_iter, int its[2], double rel[2],
                           bool& conv) {
    cudaStream_t s = mm->ctx->stream;
    double2* x = mm->x.as<double2>();
    double2* b = mm->b.as<double2>();
    const uint8_t* mask = mm->mask.as<uint8_t>();
    const double capT = mm->rho_cp / dt_s, capC = 1.0 / dt_s;
    if (!mm->element_form) {
        const int rc = ensure_transport_matrix(mm, dt_s);
        if (rc == RVE_ERR_OUT_OF_MEMORY)
            RVE_TRY(apply_element_form(mm));
        else
            RVE_TRY(rc);
    }
    // b = C/dt x^n; start from x^n with the held values in place
    auto hold = [&]() {
        k_macro_hold<<<grid_for(mm->nv), 256, 0, s>>>(mm->nv, mask, mm->hold.as<double>(), mm->x.as<double>());
    };
    if (mm->element_form) {
        const int32_t* tets = mm->tets.as<int32_t>();
        const double* geo = mm->geo.as<double>();
        const unsigned ge = grid_for(mm->nt);
        TransportTensors prm;
        std::memcpy(prm.KT, mm->KT, sizeof(prm.KT));
        std::memcpy(prm.Dc, mm->Dc, sizeof(prm.Dc));
        RVE_TRY(mm->t_dinv.ensure((size_t)mm->nv * 16));
        RVE_CUDA(cudaMemsetAsync(mm->t_dinv.p, 0, (size_t)mm->nv * 16, s));
        k_transport_diag<<<ge, 256, 0, s>>>(mm->nt, tets, geo, prm, capT, capC, mm->t_dinv.as<double2>());
        k_invert<<<grid_for(mm->nv * 2), 256, 0, s>>>(mm->nv * 2, mm->t_dinv.as<double>());
        launch_fill(mm->nv * 2, 0.0, mm->b.as<double>(), s);
        k_transport_apply<<<ge, 256, 0, s>>>(mm->nt, tets, geo, prm, capT, capC, 0, x, b);
        hold();
        auto product = [&](cudaStream_t st, const double2* in, double2* out, double* acc) {
            launch_fill(mm->nv * 2, 0.0, reinterpret_cast<double*>(out), st);
            k_transport_apply<<<ge, 256, 0, st>>>(mm->nt, tets, geo, prm, capT, capC, 1, in, out);
            if (acc)
                k_macro_dot<2><<<grid_for(mm->nv), 256, 0, st>>>(mm->nv * 2, reinterpret_cast<const double*>(in),
                                                                 reinterpret_cast<const double*>(out), acc);
        };
        return transport_pcg(mm, x, b, product, dt_s, rtol, max_iter, its, rel, conv);
    }
    const int64_t ns = mm->n_slices;
    const int64_t* base = mm->g_base.as<int64_t>();
    const int32_t* col = mm->g_col.as<int32_t>();
    const double2* mat = mm->t_mat.as<double2>();
    const unsigned gs = (unsigned)((ns + 7) / 8);
    k_transport_rhs<<<gs, 256, 0, s>>>(mm->nv, ns, base, col, mm->t_mass.as<double>(), capT, capC, x, b);
    hold();
    auto product = [&](cudaStream_t st, const double2* in, double2* out, double* acc) {
        k_transport_product<<<gs, 256, 0, st>>>(mm->nv, ns, base, col, mat, in, out, acc);
    };
    return transport_pcg(mm, x, b, product, 0.0, rtol, max_iter, its, rel, conv);
}

int rve_macro_step(rve_ctx c, rve_macro m, double dt_h, const rve_degradation* deg, double rtol, int max_iter,
                   rve_macro_stats* st) {
    NvtxRange nvtx_("macro transport and degradation step");
    RVE_TRY(check_ctx(c));
    if (!m || !(dt_h > 0) || !(rtol > 0) || max_iter < 1) {
        set_error("rve_macro_step: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    if (!m->have_transport || !m->have_face || !m->have_state) {
        set_error("rve_macro_step: set transport, face and initial state first");
        return RVE_ERR_STATE;
    }
    const auto t0 = std::chrono::steady_clock::now();
    rve_degradation dg{-0.001682, 126.0, 1.5, 0};
    if (deg) dg = *deg;
    const double dt_s = dt_h * 3600.0;
    int its[2] = {0, 0};
    double rel[2] = {0, 0};
    bool conv = false;
    RVE_TRY(transport_solve(m, dt_s, rtol, max_iter, its, rel, conv));
    cudaStream_t s = c->stream;
    double* x = m->x.as<double>();
    // Gauss-point states and the degradation update
    RVE_CUDA(cudaMemsetAsync(m->flags.p, 0, 16, s));
    k_macro_gauss<<<grid_for(m->nt * 4), 256, 0, s>>>(m->nt, m->tets.as<int32_t>(), x, m->W.as<double>(),
                                                      m->gp.as<double>(), dt_h, dg.beta, dg.Tg_C, dg.c_sat_wt, 1,
                                                      m->flags.as<int>(),
                                                      reinterpret_cast<unsigned long long*>(m->flags.as<char>() + 8));
    int bad = 0;
    double herr = 0.0;
    RVE_CUDA(cudaMemcpyAsync(&bad, m->flags.p, 4, cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaMemcpyAsync(&herr, m->flags.as<char>() + 8, 8, cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    RVE_CUDA(cudaGetLastError());
    if (st) {
        st->iterations_T = its[0];
        st->iterations_c = its[1];
        st->rel_residual_T = rel[0];
        st->rel_residual_c = rel[1];
        st->converged = conv ? 1 : 0;
        st->gauss_points_unencodable = bad;
        st->handover_max_err = herr;
        st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    if (!conv) {
        set_error("rve_macro_step: PCG did not reach rtol within max_iter");
        return RVE_ERR_NOT_CONVERGED;
    }
    return RVE_OK;
}

int rve_macro_set_state(rve_ctx c, rve_macro m, const double* T_nodal, const double* c_nodal, const double* W_gp,
                        const rve_degradation* deg) {
    RVE_TRY(check_ctx(c));
    if (!m || !T_nodal || !c_nodal || !W_gp) {
        set_error("rve_macro_set_state: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    const int64_t n = m->nt * 4;
    for (int64_t i = 0; i < n; ++i)
        if (!(W_gp[i] > 0.0 && W_gp[i] <= 1.0)) {
            set_error("rve_macro_set_state: 1 - omega outside (0, 1]");
            return RVE_ERR_INVALID_ARGUMENT;
        }
    std::vector<double> x((size_t)m->nv * 2);
    for (int64_t i = 0; i < m->nv; ++i) {
        if (!std::isfinite(T_nodal[i]) || !std::isfinite(c_nodal[i])) {
            set_error("rve_macro_set_state: non-finite nodal value");
            return RVE_ERR_INVALID_ARGUMENT;
        }
        x[(size_t)i * 2] = T_nodal[i];
        x[(size_t)i * 2 + 1] = c_nodal[i];
    }
    rve_degradation dg{-0.001682, 126.0, 1.5, 0};
    if (deg) dg = *deg;
    cudaStream_t s = c->stream;
    RVE_TRY(upload(m->x, x.data(), x.size(), s));
    RVE_TRY(upload(m->W, W_gp, (size_t)n, s));
    // the Gauss-point T, c and t_eq of the restored state; 1 - omega is not advanced
    RVE_CUDA(cudaMemsetAsync(m->flags.p, 0, 16, s));
    k_macro_gauss<<<grid_for(n), 256, 0, s>>>(m->nt, m->tets.as<int32_t>(), m->x.as<double>(), m->W.as<double>(),
                                              m->gp.as<double>(), 0.0, dg.beta, dg.Tg_C, dg.c_sat_wt, 0,
                                              m->flags.as<int>(),
                                              reinterpret_cast<unsigned long long*>(m->flags.as<char>() + 8));
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_state = true;
    return RVE_OK;
}

int rve_macro_gauss_dev(rve_ctx c, rve_macro m, const double** T_gp, const double** c_gp, const double** W_gp,
                        const double** t_eq_gp) {
    RVE_TRY(check_ctx(c));
    if (!m) {
        set_error("rve_macro_gauss_dev: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    const double* g = m->gp.as<double>();
    const int64_t n = m->nt * 4;
    if (T_gp) *T_gp = g;
    if (c_gp) *c_gp = g + n;
    if (W_gp) *W_gp = g + 2 * n;
    if (t_eq_gp) *t_eq_gp = g + 3 * n;
    return RVE_OK;
}

int rve_macro_solve_steady(rve_ctx c, rve_macro m, double rtol, int max_iter, rve_macro_stats* st) {
    NvtxRange nvtx_("macro steady transport solve");
    RVE_TRY(check_ctx(c));
    if (!m || !(rtol > 0) || max_iter < 1) {
        set_error("rve_macro_solve_steady: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    if (!m->have_transport || !m->have_face || !m->have_state) {
        set_error("rve_macro_solve_steady: set transport, held values and initial state first");
        return RVE_ERR_STATE;
    }
    const auto t0 = std::chrono::steady_clock::now();
    int its[2] = {0, 0};
    double rel[2] = {0, 0};
    bool conv = false;
    RVE_TRY(transport_solve(m, HUGE_VAL, rtol, max_iter, its, rel, conv));
    if (st) {
        std::memset(st, 0, sizeof(*st));
        st->iterations_T = its[0];
        st->iterations_c = its[1];
        st->rel_residual_T = rel[0];
        st->rel_residual_c = rel[1];
        st->converged = conv ? 1 : 0;
        st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    if (!conv) {
        set_error("rve_macro_solve_steady: PCG did not reach rtol within max_iter");
        return RVE_ERR_NOT_CONVERGED;
    }
    return RVE_OK;
}

int rve_macro_gradients(rve_ctx c, rve_macro m, int field, double* grad) {
    RVE_TRY(check_ctx(c));
    if (!m || !grad || (field != 0 && field != 1)) {
        set_error("rve_macro_gradients: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t s = c->stream;
    DevBuf g;
    RVE_TRY(g.ensure((size_t)m->nt * 3 * 8));
    k_macro_gradient<<<grid_for(m->nt), 256, 0, s>>>(m->nt, m->tets.as<int32_t>(), m->geo.as<double>(),
                                                     m->x.as<double>(), field, g.as<double>());
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaMemcpyAsync(grad, g.p, (size_t)m->nt * 3 * 8, cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    return RVE_OK;
}

int rve_fibre_directions(rve_ctx c, const double* xyz, int64_t nv, const int32_t* tets, int64_t nt,
                         const int32_t* yarn_of_tet, int n_yarn, const int32_t* yarn_axis, double rtol,
                         double* dir) {
    NvtxRange nvtx_("yarn directions (potential flow)");
    RVE_TRY(check_ctx(c));
    if (!xyz || !tets || !yarn_of_tet || !yarn_axis || !dir || nv < 4 || nt < 1 || n_yarn < 0 || !(rtol > 0)) {
        set_error("rve_fibre_directions: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    for (int y = 0; y < n_yarn; ++y)
        if (yarn_axis[y] < 0 || yarn_axis[y] > 2) {
            set_error("rve_fibre_directions: yarn axis must be 0, 1 or 2");
            return RVE_ERR_INVALID_ARGUMENT;
        }
    for (int y = 0; y < n_yarn; ++y) {
        // the yarn's own tetrahedra, nodes renumbered
        std::vector<int64_t> sel;
        for (int64_t e = 0; e < nt; ++e)
            if (yarn_of_tet[e] == y) sel.push_back(e);
        if (sel.empty()) continue;
        std::vector<int32_t> local(nv, -1), sub_tets(sel.size() * 4);
        std::vector<double> sub_xyz;
        int32_t nn = 0;
        for (size_t i = 0; i < sel.size(); ++i)
            for (int a = 0; a < 4; ++a) {
                const int32_t v = tets[sel[i] * 4 + a];
                if (v < 0 || v >= nv) {
                    set_error("rve_fibre_directions: vertex index out of range");
                    return RVE_ERR_BAD_MESH;
                }
                if (local[v] < 0) {
                    local[v] = nn++;
                    sub_xyz.insert(sub_xyz.end(), xyz + (int64_t)v * 3, xyz + (int64_t)v * 3 + 3);
                }
                sub_tets[i * 4 + a] = local[v];
            }
        // inlet (phi = 0) and outlet (phi = 1): the yarn's ends along its axis
        const int ax = yarn_axis[y];
        double lo = HUGE_VAL, hi = -HUGE_VAL;
        for (int32_t k = 0; k < nn; ++k) {
            lo = std::min(lo, sub_xyz[(size_t)k * 3 + ax]);
            hi = std::max(hi, sub_xyz[(size_t)k * 3 + ax]);
        }
        const double tol = 1e-9 * std::max(1.0, hi - lo);
        std::vector<uint8_t> held(nn, 0);
        std::vector<double> vals((size_t)nn * 2, 0.0);
        for (int32_t k = 0; k < nn; ++k) {
            const double sk = sub_xyz[(size_t)k * 3 + ax];
            if (sk <= lo + tol || sk >= hi - tol) {
                held[k] = 1;
                vals[(size_t)k * 2] = sk >= hi - tol ? 1.0 : 0.0;
            }
        }
        rve_macro m = nullptr;
        RVE_TRY(rve_macro_create(c, sub_xyz.data(), nn, sub_tets.data(), (int64_t)sel.size(), &m));
        static const double eye[9] = {1, 0, 0, 0, 1, 0, 0, 0, 1};
        int rc = rve_macro_set_transport(c, m, eye, 1.0, eye);
        if (rc == RVE_OK) rc = rve_macro_set_held(c, m, held.data(), vals.data());
        if (rc == RVE_OK) rc = rve_macro_reset(c, m, 0.0, 0.0);
        if (rc == RVE_OK) rc = rve_macro_solve_steady(c, m, rtol, 20000, nullptr);
        std::vector<double> g(sel.size() * 3);
        if (rc == RVE_OK) rc = rve_macro_gradients(c, m, 0, g.data());
        rve_macro_free(c, m);
        if (rc != RVE_OK) return rc;
        for (size_t i = 0; i < sel.size(); ++i) {
            const double* gi = &g[i * 3];
            const double nrm = std::sqrt(gi[0] * gi[0] + gi[1] * gi[1] + gi[2] * gi[2]);
            if (nrm > 0)
                for (int k = 0; k < 3; ++k) dir[sel[i] * 3 + k] = gi[k] / nrm;
        }
    }
    return RVE_OK;
}

int rve_macro_get(rve_ctx c, rve_macro m, double* T_nodal, double* c_nodal, double* T_gp, double* c_gp, double* W_gp,
                  double* t_eq_gp) {
    RVE_TRY(check_ctx(c));
    if (!m) {
        set_error("rve_macro_get: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t s = c->stream;
    if (T_nodal || c_nodal) {
        std::vector<double> x((size_t)m->nv * 2);
        RVE_CUDA(cudaMemcpyAsync(x.data(), m->x.p, x.size() * 8, cudaMemcpyDeviceToHost, s));
        RVE_CUDA(cudaStreamSynchronize(s));
        for (int64_t i = 0; i < m->nv; ++i) {
            if (T_nodal) T_nodal[i] = x[(size_t)i * 2];
            if (c_nodal) c_nodal[i] = x[(size_t)i * 2 + 1];
        }
    }
    const int64_t n = m->nt * 4;
    double* outs[4] = {T_gp, c_gp, W_gp, t_eq_gp};
    for (int k = 0; k < 4; ++k)
        if (outs[k]) RVE_CUDA(cudaMemcpyAsync(outs[k], m->gp.as<double>() + k * n, n * 8, cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    return RVE_OK;
}

// ---------------------------------------------------------- macro mechanics

int rve_macro_mech_set_bc(rve_ctx c, rve_macro m, const uint8_t* fixed, const double* values) {
    RVE_TRY(check_ctx(c));
    if (!m || !fixed) {
        set_error("rve_macro_mech_set_bc: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    const size_t n = (size_t)m->nv * 3;
    std::vector<uint8_t> f(n);
    std::vector<double> v(n, 0.0);
    for (size_t i = 0; i < n; ++i) {
        f[i] = fixed[i] ? 1 : 0;
        if (f[i] && values) {
            if (!std::isfinite(values[i])) {
                set_error("rve_macro_mech_set_bc: non-finite prescribed value");
                return RVE_ERR_INVALID_ARGUMENT;
            }
            v[i] = values[i];
        }
    }
    cudaStream_t s = c->stream;
    RVE_TRY(upload(m->mfix, f.data(), n, s));
    RVE_TRY(upload(m->mval, v.data(), n, s));
    if (!m->have_mech_u) {
        RVE_TRY(m->mu.ensure(n * 8));
        RVE_CUDA(cudaMemsetAsync(m->mu.p, 0, n * 8, s));
    }
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_mech_u = true;
    m->have_mech_bc = true;
    return RVE_OK;
}

int rve_macro_mech_set_u(rve_ctx c, rve_macro m, const double* u) {
    RVE_TRY(check_ctx(c));
    if (!m) {
        set_error("rve_macro_mech_set_u: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    const size_t n = (size_t)m->nv * 3;
    cudaStream_t s = c->stream;
    if (u) {
        RVE_TRY(upload(m->mu, u, n, s));
    } else {
        RVE_TRY(m->mu.ensure(n * 8));
        RVE_CUDA(cudaMemsetAsync(m->mu.p, 0, n * 8, s));
    }
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_mech_u = true;
    return RVE_OK;
}

int rve_macro_mech_set_traction(rve_ctx c, rve_macro m, const uint8_t* face_nodes, const double t[3], int add) {
    RVE_TRY(check_ctx(c));
    if (!m || !face_nodes || !t || !std::isfinite(t[0]) || !std::isfinite(t[1]) || !std::isfinite(t[2])) {
        set_error("rve_macro_mech_set_traction: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    const size_t n = (size_t)m->nv * 3;
    std::vector<uint8_t> mk(face_nodes, face_nodes + m->nv);
    for (auto& x : mk) x = x ? 1 : 0;
    cudaStream_t s = c->stream;
    DevBuf fm;
    RVE_TRY(upload(fm, mk.data(), mk.size(), s));
    if (!add || !m->have_mech_load) {
        RVE_TRY(m->mload.ensure(n * 8));
        RVE_CUDA(cudaMemsetAsync(m->mload.p, 0, n * 8, s));
    }
    k_mech_traction<<<grid_for(m->nt), 256, 0, s>>>(m->nt, m->tets.as<int32_t>(), m->geo.as<double>(),
                                                    fm.as<uint8_t>(), t[0], t[1], t[2], m->mload.as<double>());
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_mech_load = true;
    return RVE_OK;
}

int rve_macro_mech_solve(rve_ctx c, rve_macro m, const double* C_gp, int C_on_device, double rtol, int max_iter,
                         rve_macro_mech_stats* st) {
    NvtxRange nvtx_("macro elastic solve");
    RVE_TRY(check_ctx(c));
    if (!m || !C_gp || !(rtol > 0) || max_iter < 1) {
        set_error("rve_macro_mech_solve: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    if (!m->have_mech_bc || !m->have_mech_load) {
        set_error("rve_macro_mech_solve: set the held DOFs and the traction first");
        return RVE_ERR_STATE;
    }
    const auto t0 = std::chrono::steady_clock::now();
    cudaStream_t s = c->stream;
    const int64_t n = m->nv * 3;
    const double* Cg = C_gp;
    if (!C_on_device) {
        RVE_TRY(upload(m->cgp, C_gp, (size_t)m->nt * 4 * 36, s));
        Cg = m->cgp.as<double>();
    }
    for (DevBuf* bfr : {&m->b, &m->r, &m->p, &m->q, &m->mdinv}) RVE_TRY(bfr->ensure((size_t)n * 8));
    RVE_TRY(m->cm.ensure((size_t)m->nt * 36 * 8));
    RVE_TRY(m->msig.ensure((size_t)m->nt * 4 * 6 * 8));
    if (!m->element_form) {
        const int rc = ensure_mech_matrix(m);
        if (rc == RVE_ERR_OUT_OF_MEMORY)
            RVE_TRY(apply_element_form(m));
        else
            RVE_TRY(rc);
    }
    const int32_t* tets = m->tets.as<int32_t>();
    const double* geo = m->geo.as<double>();
    const double* cm = m->cm.as<double>();
    k_mech_material<<<(unsigned)std::min<int64_t>((m->nt * 36 + 255) / 256, (int64_t)sm_count() * 16), 256, 0, s>>>(
        m->nt, Cg, m->cm.as<double>());
    RVE_CUDA(cudaMemsetAsync(m->mdinv.p, 0, (size_t)n * 8, s));   // nodes of no element: z = 0
    double* b = m->b.as<double>();
    double* u = m->mu.as<double>();
    RVE_CUDA(cudaMemcpyAsync(b, m->mload.p, n * 8, cudaMemcpyDeviceToDevice, s));
    k_mech_hold<<<grid_for(n), 256, 0, s>>>(n, m->mfix.as<uint8_t>(), m->mval.as<double>(), u);
    int its[2] = {0, 0};
    double rel[2] = {0, 0};
    bool conv = false;
    if (m->element_form) {
        const unsigned ge = grid_for(m->nt);
        k_mech_diag<<<grid_for(m->nt * 4), 256, 0, s>>>(m->nt, tets, geo, cm, m->mdinv.as<double>());
        k_invert<<<grid_for(n), 256, 0, s>>>(n, m->mdinv.as<double>());
        auto product = [&](cudaStream_t st, const double* in, double* out, int, double* acc) {
            launch_fill(n, 0.0, out, st);
            k_mech_apply<<<ge, 256, 0, st>>>(m->nt, tets, geo, cm, in, out);
            if (acc) k_macro_dot<1><<<grid_for(n), 256, 0, st>>>(n, in, out, acc);
        };
        RVE_TRY(mech_pcg(m, n, u, b, product, [](cudaStream_t, const MechCheb&) {}, rtol, max_iter, its, rel, conv));
    } else {
        const int64_t* base = m->g_base.as<int64_t>();
        const int32_t* col = m->g_col.as<int32_t>();
        k_mech_entries<<<(unsigned)m->n_slices, 256, 0, s>>>(m->nv, base, col, m->g_len.as<int32_t>(),
                                                             m->g_eptr.as<int32_t>(), m->g_inc.as<int32_t>(), tets, geo,
                                                             cm, m->mmat.as<double>(), m->mdinv.as<double>());
        const double* mat = m->mmat.as<double>();
        const unsigned gm = (unsigned)std::min<int64_t>((m->n_slices + 1) / 2, (int64_t)sm_count() * 10);
        auto product = [&](cudaStream_t st, const double* in, double* out, int norm, double* acc) {
            k_mech_product<<<gm, MECH_THREADS, 0, st>>>(m->nv, m->n_slices, base, col, mat, in, out, norm, acc);
        };
        const float* mat32 = m->mmat32.as<float>();
        k_narrow<<<(unsigned)(sm_count() * 16), 256, 0, s>>>(m->n_ell * 288, mat, m->mmat32.as<float>());
        auto step = [&](cudaStream_t st, const MechCheb& c) {
            k_mech_cheb<<<(unsigned)((m->n_slices + 1) / 2), 192, 0, st>>>(m->nv, m->n_slices, base, col, mat32, c);
        };
        RVE_TRY(mech_pcg(m, n, u, b, product, step, rtol, max_iter, its, rel, conv));
    }
    k_mech_stress<<<grid_for(m->nt * 4), 256, 0, s>>>(m->nt, tets, geo, Cg, u, m->msig.as<double>());
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaStreamSynchronize(s));
    m->have_mech_sig = true;
    if (st) {
        st->iterations = its[0];
        st->converged = conv ? 1 : 0;
        st->rel_residual = rel[0];
        st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    }
    if (!conv) {
        set_error("rve_macro_mech_solve: PCG did not reach rtol within max_iter");
        return RVE_ERR_NOT_CONVERGED;
    }
    return RVE_OK;
}

int rve_debug_macro_matrix_limit(rve_ctx c, rve_macro m, int64_t bytes) {
    RVE_TRY(check_ctx(c));
    if (!m || bytes < 0) {
        set_error("rve_debug_macro_matrix_limit: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    RVE_TRY(apply_element_form(m));   // (drops the graph and the matrices)
    m->element_form = false;
    m->mat_limit = (size_t)bytes;
    return RVE_OK;
}

int rve_macro_mech_get(rve_ctx c, rve_macro m, double* u, double* stress_gp, double* load) {
    RVE_TRY(check_ctx(c));
    if (!m) {
        set_error("rve_macro_mech_get: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    if ((u && !m->have_mech_u) || (stress_gp && !m->have_mech_sig) || (load && !m->have_mech_load)) {
        set_error("rve_macro_mech_get: nothing of that kind has been set or solved yet");
        return RVE_ERR_STATE;
    }
    cudaStream_t s = c->stream;
    const size_t n = (size_t)m->nv * 3;
    if (u) RVE_CUDA(cudaMemcpyAsync(u, m->mu.p, n * 8, cudaMemcpyDeviceToHost, s));
    if (load) RVE_CUDA(cudaMemcpyAsync(load, m->mload.p, n * 8, cudaMemcpyDeviceToHost, s));
    if (stress_gp)
        RVE_CUDA(cudaMemcpyAsync(stress_gp, m->msig.p, (size_t)m->nt * 4 * 6 * 8, cudaMemcpyDeviceToHost, s));
    RVE_CUDA(cudaStreamSynchronize(s));
    return RVE_OK;
}

}  // extern "C"
