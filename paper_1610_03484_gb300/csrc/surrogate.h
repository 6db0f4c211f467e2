// Launch wrappers of the surrogate kernels (surrogate.cu).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace rve {

// sets the GEMM kernels' shared-memory limit (once per device, before the first launch)
cudaError_t gemm_tc_prepare();
// nonzero once a bounded wait inside the GEMM gave up (sticky for the process)
int gemm_tc_timed_out();
// sets that word (tests) and returns the old one, -1 before gemm_tc_prepare
int gemm_tc_set_timed_out(int v);
// C = A Bt^T on the tensor cores (TMA-fed): problems of the same N and K in one launch,
// each with its own M; an error if a tensor map cannot be encoded
constexpr int GEMM_GROUP = 16;
struct GemmProblem {
    const __nv_bfloat16 *A = nullptr, *Bt = nullptr;
    const float *bias = nullptr, *pre = nullptr;
    __nv_bfloat16* Cb = nullptr;
    float* Cf = nullptr;
    int M = 0;
};
cudaError_t launch_gemm_group(int count, const GemmProblem* probs, int N, int K, int epilogue, cudaStream_t s);
cudaError_t launch_gemm_bf16(int M, int N, int K, const __nv_bfloat16* A, const __nv_bfloat16* Bt,
                             const float* bias, int epilogue, __nv_bfloat16* Cb, float* Cf, cudaStream_t s);
// Fused ensemble inference: all layers of up to mlp_fused_max_members() members per
// 128-row tile with the activations kept on chip; X [M][64] BF16 features, member e's
// W^T of layer l at wt[e] + w_off[l], biases bias[e * 5 + l]; z of member e written
// transposed to zT + e * 64 * ldz ([64][ldz]).  An error if a tensor map cannot be encoded.
int mlp_fused_max_members();
cudaError_t launch_mlp_fused(int M, int members, const __nv_bfloat16* X, const __nv_bfloat16* const* wt,
                             const int64_t* w_off, const float* const* bias, float* zT, int ldz, cudaStream_t s);
constexpr int MAX_MEMBERS = 16;

// jobs of the backward pass: out [cols][rows] = in [rows][cols] transposed, or (out null)
// sum [cols] = column sums of in, or (part given) *sum += the step's loss, part [rows]
constexpr int PREP_JOBS = 64;
struct PrepJob {
    const __nv_bfloat16* in;
    __nv_bfloat16* out;
    float* sum;
    int rows, cols;
    const float* part = nullptr;
};
struct PrepJobs {
    PrepJob job[PREP_JOBS];
};
void launch_backward_prep(const PrepJobs& J, int count, int max_cols, int max_rows, cudaStream_t s);

// part [head_loss_parts]: the loss, a partial sum per warp
struct HeadArgs {
    const float* z[MAX_MEMBERS];
    const int32_t* rows[MAX_MEMBERS];
    __nv_bfloat16* dz[MAX_MEMBERS];
    float* part[MAX_MEMBERS];
};
int head_loss_parts(int M, int noutp);
void launch_head_loss(int members, int M, int noutp, const HeadArgs& A, const float* target, const float* sigma,
                      const uint8_t* diag, cudaStream_t s);

// one layer of one member: weights W [K][N] with the bias [N] behind them, moments m1, m2
// laid out alike, gradients Gt [N][K] (null: zero) and gb [N] (null: weights only)
constexpr int ADAM_JOBS = 40;
struct AdamJob {
    float *W, *m1, *m2;
    const float *Gt, *gb;
    __nv_bfloat16 *Wt, *Wn;
    int K, N, n_valid;
};
struct AdamJobs {
    AdamJob job[ADAM_JOBS];
};
void launch_adam(const AdamJobs& J, int count, float lr, int step, cudaStream_t s);

struct FeatureArgs {
    const int32_t* rows[MAX_MEMBERS];
    __nv_bfloat16* X[MAX_MEMBERS];
};
void launch_features(int members, int n, int M, int kin, const double* feat, const FeatureArgs& A, const float* mean,
                     const float* inv_std, cudaStream_t s);

// member outputs z + e zstride ([64][ldz], transposed) -> ensemble means C [n][36],
// K [n][9], D [n][9] (times the reference scales rc, rk, rd; FP64) and spread [n]
void launch_ensemble(int n, int ldz, int members, const float* z, int64_t zstride, const uint8_t* diag, double rc,
                     double rk, double rd, double* C, double* K, double* D, double* spread, cudaStream_t s);

}  // namespace rve
