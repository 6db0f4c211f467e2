// Assembled operator of one field (assembled.cu): block rows of the hierarchic DOF
// nodes, phase by phase, so that one matrix serves every degradation factor.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kernels.h"

namespace rve {

// Entry of the matrix: the NC x NC block (mechanics: 9 values) or the conductivity and
// diffusivity (scalar fields: 2 values), the coupled node's index as the bit pattern
// of an int32 in the next word, padded to a vector load.
template <typename T, int NC>
struct AsmEntry {
    static constexpr int VALUES = NC == 3 ? 9 : 2;
    static constexpr int WORDS = NC == 3 ? (sizeof(T) == 4 ? 12 : 10) : 4;
};

template <typename T>
struct AsmView {
    int64_t n = 0;                    // block rows (scalar DOF nodes)
    const int32_t* order = nullptr;   // [n] node of each row, in order of storage
    const int32_t* ptr = nullptr;     // [n + 1] first entry of each row
    const int32_t* split = nullptr;   // [n] first entry of phase 1 in each row
    const T* ent = nullptr;           // [entries][AsmEntry::WORDS]
    const T* scale = nullptr;         // [ncols][2] factor per column and phase
};

// Sparsity on the device, shared by the fields and precisions of one DOF map.
struct AsmGraph {
    int64_t n = 0, entries = 0;
    int ne = 0;
    const int32_t *order = nullptr, *ptr = nullptr, *split = nullptr, *col = nullptr;
    const int32_t *eptr = nullptr, *inc = nullptr;   // incidences of each node (element * ne + local)
};

// Matrix entries from the FP64 element data (p = 1, 2), in FP64 and / or FP32 (null: not
// wanted); rtab [9 ne^2] is device scratch.
void launch_assemble(int p, int nc, const AsmGraph& g, const int32_t* edofs, const uint8_t* phase,
                     const double* geo64, const double* mat64, double* rtab, double* ent64, float* ent32,
                     cudaStream_t s);

// y = A x for the columns of active groups (active null: all), per-column energies
// x . A x added into energy_acc[slot][col] (null: not wanted), slot < ACC_SLOTS.
template <typename T>
void launch_asm_product(int nc, const AsmView<T>& A, const T* x, T* y, int ncols, const int32_t* active,
                        double* energy_acc, cudaStream_t s);
// y = b - A x for all columns
template <typename T>
void launch_asm_residual(int nc, const AsmView<T>& A, const T* x, const T* b, T* y, int ncols, cudaStream_t s);

// dinv [n_rows][groups]: inverse Jacobi diagonal of the column groups that share one
// (mechanics: the RVEs; scalar fields: conductivity, diffusivity); dinv32 (optional)
// the same times f32 in FP32
void launch_jacobi_inverse(const RowView<double>& rv, int groups, double* dinv, float* dinv32, double f32,
                           cudaStream_t s);

// One step of the Chebyshev iteration for A z = r from z_0 = 0 with the Jacobi diagonal:
//   d_k = c1 d_(k-1) + c2 D^-1 (r - A z_k),  z_(k+1) = z_k + d_k
// in FP32 (Saad, Iterative Methods for Sparse Linear Systems, algorithm 12.1).  With
// rz_acc it is the last one: d is not kept and (r64, z_new) per column is added.
struct ChebArgs {
    const float* d_in = nullptr;
    float* d_out = nullptr;
    const float* dinv = nullptr;   // [n_rows][groups]
    int groups = 0;
    float c1 = 0.f, c2 = 0.f;
    const double* r64 = nullptr;
};
void launch_cheb_step(int nc, const AsmView<float>& A, const float* z, const float* r32, float* z_new,
                      const ChebArgs& ch, int ncols, const int32_t* active, double* rz_acc, cudaStream_t s);

// The vector passes around it in the FP64 PCG (see assembled.cu).
void launch_cheb_update(const RowView<double>& rv, const float* dinv32, double* x, double* r, const double* p,
                        const double* q, float* r32, float* z, float w, ColState cs, bool apply, const Launch& L);
void launch_cheb_beta(ColState cs, int ncols, bool first, cudaGraphConditionalHandle h, int32_t* counter,
                      int max_iter, bool ctl, cudaStream_t s);
void launch_cheb_direction(int64_t n_rows, const float* z, double* p, double* q, ColState cs, bool first,
                           const Launch& L);
// the step behind an element-by-element product (y = A z, cleared): z += d in place
void launch_cheb_vector(int64_t n_rows, int nfield, const float* r32, const ChebArgs& ch, float* z, float* y,
                        const int32_t* active, double* rz_acc, const Launch& L);

// Largest eigenvalue of D^-1 A by power iteration over six columns with the phase scales
// of power_scales ([6][2]): x random, then y = A x and x = D^-1 y / 2 in turn; with out
// [12] (zeroed) instead (x, y) and (x, D x) per column.  x, y [n_rows][6].
void power_scales(int nc, float* scale);
void launch_power_start(int64_t n_rows, float* x, cudaStream_t s);
void launch_power_next(int nc, int64_t n_rows, const double* diag, float* x, const float* y, double* out,
                       cudaStream_t s);

// Cold uniform-traction solves without constraint rows (Solver::traction_start): the unit
// loads of the constraint rows first .. first + n - 1, and the fluctuations from their
// solutions.
void launch_traction_loads(int64_t n_sup, int m, int first, int n, const int64_t* row, const double* coef, int ncols,
                           double* r, cudaStream_t s);
void launch_traction_combine(int64_t n_rows, int nc, int nrve, const double* mu, const int32_t* vertex,
                             const double* xyz, double* x, cudaStream_t s);

}  // namespace rve
