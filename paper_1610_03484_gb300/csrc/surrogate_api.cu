// C ABI of the learned surrogate: ensemble MLP training and inference on the
// GPU (surrogate.cu kernels) and the surrogate-plus-fallback batched FE^2 call.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <numeric>
#include <random>
#include <vector>

#include "api_internal.h"
#include "surrogate.h"

namespace rve {
namespace {

constexpr int KIN = 64;      // 8 features padded to one GEMM tile
constexpr int HID = 256;     // hidden width
constexpr int NOUTP = 64;    // 33 outputs padded
constexpr int NOUT = 33;
constexpr int NLAYER = 5;
constexpr int NFEAT = 8;
constexpr int HEADER = 8 + 8 + 33 + 3;   // feature mean, feature std, sigma, reference scales

const int LK[NLAYER] = {KIN, HID, HID, HID, HID};
const int LN[NLAYER] = {HID, HID, HID, HID, NOUTP};

int64_t layer_w_off(int l) {
    int64_t o = 0;
    for (int i = 0; i < l; ++i) o += (int64_t)LK[i] * LN[i] + LN[i];
    return o;
}
int64_t n_params() { return layer_w_off(NLAYER); }

std::vector<uint8_t> diag_mask() {
    std::vector<uint8_t> d(NOUT, 0);
    const int sizes[3] = {6, 3, 3}, offs[3] = {0, 21, 27};
    for (int b = 0; b < 3; ++b) {
        int k = 0;
        for (int i = 0; i < sizes[b]; ++i)
            for (int j = 0; j <= i; ++j) d[offs[b] + k++] = (i == j);
    }
    return d;
}

}  // namespace
}  // namespace rve

using namespace rve;

struct rve_surrogate_s {
    rve_ctx ctx = nullptr;
    int members = 0;
    bool trained = false;
    float feat_mean[8] = {0}, feat_std[8] = {1, 1, 1, 1, 1, 1, 1, 1};
    float sigma[33];
    double ref[3] = {1, 1, 1};
    // per member: FP32 master params, Adam moments, BF16 weights in both layouts
    std::vector<DevBuf> P, M1, M2, Wt, Wn;
    DevBuf d_norm, d_diag;   // feature mean and inverse std [16]; diagonal entries
    DevBuf train_work;       // training buffers of the members trained together (TrainWork)
    size_t work_limit = 0;   // bytes they may take (0: what the device has)
    // inference: the fused kernel (all members' layers per tile, activations on chip)
    // or one GEMM launch per member and layer
    bool fused = true;
    DevBuf H[NLAYER], zall;
};

namespace {

// whether a bounded wait of the GEMMs gave up (call it after a synchronisation)
int wait_status() {
    if (!gemm_tc_timed_out()) return RVE_OK;
    set_error("a bounded wait inside the surrogate GEMM gave up");
    return RVE_ERR_TIMEOUT;
}

// the feature normalisation on the device
int upload_norm(rve_surrogate s) {
    float h[16];
    for (int k = 0; k < 8; ++k) {
        h[k] = s->feat_mean[k];
        h[8 + k] = 1.f / s->feat_std[k];
    }
    return upload(s->d_norm, h, 16, s->ctx->stream);
}

AdamJob adam_job(rve_surrogate s, int e, int l) {
    const int64_t o = layer_w_off(l);
    AdamJob j;
    j.W = s->P[e].as<float>() + o;
    j.m1 = s->M1[e].as<float>() + o;
    j.m2 = s->M2[e].as<float>() + o;
    j.Gt = nullptr;
    j.gb = nullptr;
    j.Wt = s->Wt[e].as<__nv_bfloat16>() + o;
    j.Wn = s->Wn[e].as<__nv_bfloat16>() + o;
    j.K = LK[l];
    j.N = LN[l];
    j.n_valid = LN[l];
    return j;
}

int refresh_bf16(rve_surrogate s, int e) {
    // rebuild BF16 copies from the FP32 master parameters via a zero-lr Adam pass
    AdamJobs J;
    for (int l = 0; l < NLAYER; ++l) J.job[l] = adam_job(s, e, l);
    launch_adam(J, NLAYER, 0.f, 1, s->ctx->stream);
    return RVE_OK;
}

// Training buffers of nm members for batches of M rows, carved out of one allocation:
// per member and layer the input H [M][K] and output gradient G [M][N] with their
// transposes, the pre-activations Z, the gradients, and the network's output.
struct TrainWork {
    __nv_bfloat16 *H[MAX_MEMBERS][NLAYER], *Ht[MAX_MEMBERS][NLAYER], *G[MAX_MEMBERS][NLAYER], *Gt[MAX_MEMBERS][NLAYER];
    float *Z[MAX_MEMBERS][NLAYER], *gradT[MAX_MEMBERS][NLAYER], *gradb[MAX_MEMBERS][NLAYER], *zout[MAX_MEMBERS];
    float* lpart[MAX_MEMBERS];   // partial sums of the loss
};

int train_work(rve_surrogate s, int nm, int M, TrainWork& w) {
    size_t off = 0;
    char* base = nullptr;
    auto take = [&](size_t bytes) {
        char* q = base + off;
        off += (bytes + 255) / 256 * 256;
        return q;
    };
    for (int pass = 0; pass < 2; ++pass) {
        off = 0;
        for (int e = 0; e < nm; ++e) {
            for (int l = 0; l < NLAYER; ++l) {
                w.H[e][l] = reinterpret_cast<__nv_bfloat16*>(take((size_t)M * LK[l] * 2));
                w.Ht[e][l] = reinterpret_cast<__nv_bfloat16*>(take((size_t)M * LK[l] * 2));
                w.G[e][l] = reinterpret_cast<__nv_bfloat16*>(take((size_t)M * LN[l] * 2));
                w.Gt[e][l] = reinterpret_cast<__nv_bfloat16*>(take((size_t)M * LN[l] * 2));
                w.Z[e][l] = reinterpret_cast<float*>(take((size_t)M * LN[l] * 4));
                w.gradT[e][l] = reinterpret_cast<float*>(take((size_t)LK[l] * LN[l] * 4));
                w.gradb[e][l] = reinterpret_cast<float*>(take((size_t)LN[l] * 4));
            }
            w.zout[e] = reinterpret_cast<float*>(take((size_t)M * NOUTP * 4));
            w.lpart[e] = reinterpret_cast<float*>(take((size_t)head_loss_parts(M, NOUTP) * 4));
        }
        if (pass == 0) {
            if (s->work_limit > 0 && nm > 1 && off > s->work_limit) {
                set_error("training buffers above their limit");
                return RVE_ERR_OUT_OF_MEMORY;
            }
            RVE_TRY(s->train_work.ensure(off));
            base = s->train_work.as<char>();
        }
    }
    return RVE_OK;
}

// launches of one problem list, at most GEMM_GROUP each
int gemm_all(std::vector<GemmProblem>& v, int N, int K, int epilogue, rve_ctx c) {
    for (size_t i = 0; i < v.size(); i += GEMM_GROUP) {
        RVE_CUDA(launch_gemm_group((int)std::min<size_t>(GEMM_GROUP, v.size() - i), &v[i], N, K, epilogue, c->stream));
        c->launches++;
    }
    v.clear();
    return RVE_OK;
}

// One minibatch of M rows for the members first .. first + nm - 1 in lockstep, every
// launch covering all of them (a member's GEMMs alone are 8 tiles on 152 SMs): row r of
// member first + e is row rows[e][r] of the data (r without lists).  Leaves the gradients
// in w and adds the loss of member first + e to loss[e].
int forward_backward(rve_surrogate s, int first, int nm, int M, const TrainWork& w, const double* feat,
                     const float* target, const float* sigma, const int32_t* const* rows, float* const* loss) {
    rve_ctx c = s->ctx;
    cudaStream_t st = c->stream;
    FeatureArgs fa;
    for (int e = 0; e < nm; ++e) {
        fa.rows[e] = rows ? rows[e] : nullptr;
        fa.X[e] = w.H[e][0];
    }
    const float* norm = s->d_norm.as<float>();
    launch_features(nm, M, M, KIN, feat, fa, norm, norm + 8, st);
    std::vector<GemmProblem> v;
    for (int l = 0; l < NLAYER; ++l) {
        const int64_t o = layer_w_off(l);
        for (int e = 0; e < nm; ++e) {
            GemmProblem p;
            p.A = w.H[e][l];
            p.Bt = s->Wt[first + e].as<__nv_bfloat16>() + o;
            p.bias = s->P[first + e].as<float>() + o + (int64_t)LK[l] * LN[l];
            p.M = M;
            if (l < NLAYER - 1) {
                p.Cb = w.H[e][l + 1];
                p.Cf = w.Z[e][l];
            } else {
                p.Cf = w.zout[e];
            }
            v.push_back(p);
        }
        RVE_TRY(gemm_all(v, LN[l], LK[l], l < NLAYER - 1 ? 1 : 2, c));
    }
    HeadArgs ha;
    for (int e = 0; e < nm; ++e) {
        ha.z[e] = w.zout[e];
        ha.rows[e] = rows ? rows[e] : nullptr;
        ha.dz[e] = w.G[e][NLAYER - 1];
        ha.part[e] = w.lpart[e];
    }
    launch_head_loss(nm, M, NOUTP, ha, target, sigma, s->d_diag.as<uint8_t>(), st);
    c->launches += 2;
    // dH_l = G_l W_l^T, through the silu of layer l - 1
    for (int l = NLAYER - 1; l > 0; --l) {
        for (int e = 0; e < nm; ++e) {
            GemmProblem p;
            p.A = w.G[e][l];
            p.Bt = s->Wn[first + e].as<__nv_bfloat16>() + layer_w_off(l);
            p.pre = w.Z[e][l - 1];
            p.Cb = w.G[e][l - 1];
            p.M = M;
            v.push_back(p);
        }
        RVE_TRY(gemm_all(v, LK[l], LN[l], 5, c));
    }
    // transposes, bias gradients and the loss, then dW^T [N][K] = G^T H
    PrepJobs J;
    int nj = 0;
    auto flush = [&]() {
        if (nj) {
            launch_backward_prep(J, nj, HID, M, st);
            c->launches++;
        }
        nj = 0;
    };
    for (int e = 0; e < nm; ++e) {
        if (nj + 1 > PREP_JOBS) flush();
        J.job[nj++] = PrepJob{nullptr, nullptr, loss[e], head_loss_parts(M, NOUTP), 0, w.lpart[e]};
        for (int l = 0; l < NLAYER; ++l) {
            if (nj + 3 > PREP_JOBS) flush();
            J.job[nj++] = PrepJob{w.G[e][l], w.Gt[e][l], nullptr, M, LN[l]};
            J.job[nj++] = PrepJob{w.H[e][l], w.Ht[e][l], nullptr, M, LK[l]};
            J.job[nj++] = PrepJob{w.G[e][l], nullptr, w.gradb[e][l], M, LN[l]};
        }
    }
    flush();
    for (int wide = 0; wide < 2; ++wide) {   // layer 0 has 64 inputs, the others 256
        for (int e = 0; e < nm; ++e)
            for (int l = wide; l < (wide ? NLAYER : 1); ++l) {
                GemmProblem p;
                p.A = w.Gt[e][l];
                p.Bt = w.Ht[e][l];
                p.Cf = w.gradT[e][l];
                p.M = LN[l];
                v.push_back(p);
            }
        RVE_TRY(gemm_all(v, wide ? HID : KIN, M, 0, c));
    }
    return RVE_OK;
}

// Adam for the members first .. first + nm - 1
void adam_step(rve_surrogate s, int first, int nm, const TrainWork& w, float lr, int step) {
    AdamJobs J;
    int nj = 0;
    for (int e = 0; e < nm; ++e)
        for (int l = 0; l < NLAYER; ++l) {
            AdamJob j = adam_job(s, first + e, l);
            j.Gt = w.gradT[e][l];
            j.gb = w.gradb[e][l];
            if (l == NLAYER - 1) j.n_valid = NOUT;
            J.job[nj++] = j;
            if (nj == ADAM_JOBS || (e == nm - 1 && l == NLAYER - 1)) {
                launch_adam(J, nj, lr, step, s->ctx->stream);
                s->ctx->launches++;
                nj = 0;
            }
        }
}

}  // namespace

extern "C" {

int rve_surrogate_create(rve_ctx c, int members, uint64_t seed, rve_surrogate* out) {
    RVE_TRY(check_ctx(c));
    if (!out || members < 1 || members > 16) {
        set_error("rve_surrogate_create: members must be 1..16");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    RVE_CUDA(gemm_tc_prepare());
    auto* s = new rve_surrogate_s();
    s->ctx = c;
    s->members = members;
    for (int i = 0; i < NOUT; ++i) s->sigma[i] = 1.f;
    s->P.resize(members);
    s->M1.resize(members);
    s->M2.resize(members);
    s->Wt.resize(members);
    s->Wn.resize(members);
    const int64_t np = n_params();
    cudaStream_t st = c->stream;
    for (int e = 0; e < members; ++e) {
        std::mt19937_64 rng(seed * 1000003ull + (uint64_t)e);
        std::vector<float> h(np, 0.f);
        for (int l = 0; l < NLAYER; ++l) {
            const int64_t o = layer_w_off(l);
            const int kin = l == 0 ? NFEAT : LK[l];   // padded inputs stay zero
            const float lim = std::sqrt(6.f / kin);
            std::uniform_real_distribution<float> U(-lim, lim);
            for (int k = 0; k < LK[l]; ++k)
                for (int n = 0; n < LN[l]; ++n)
                    h[o + (int64_t)k * LN[l] + n] = (k < kin && (l < NLAYER - 1 || n < NOUT)) ? U(rng) : 0.f;
        }
        int rc = upload(s->P[e], h.data(), h.size(), st);
        if (rc == RVE_OK) rc = s->M1[e].ensure(np * 4);
        if (rc == RVE_OK) rc = s->M2[e].ensure(np * 4);
        if (rc == RVE_OK) rc = s->Wt[e].ensure(np * 2);
        if (rc == RVE_OK) rc = s->Wn[e].ensure(np * 2);
        if (rc != RVE_OK) {
            delete s;
            return rc;
        }
        cudaMemsetAsync(s->M1[e].p, 0, np * 4, st);
        cudaMemsetAsync(s->M2[e].p, 0, np * 4, st);
        rc = refresh_bf16(s, e);
        if (rc != RVE_OK) {
            delete s;
            return rc;
        }
    }
    auto dm = diag_mask();
    if (upload(s->d_diag, dm.data(), dm.size(), st) != RVE_OK) {
        delete s;
        return RVE_ERR_OUT_OF_MEMORY;
    }
    *out = s;
    return RVE_OK;
}

int rve_surrogate_free(rve_ctx c, rve_surrogate s) {
    if (!s) return RVE_OK;
    if (c) cudaSetDevice(c->device);
    cudaStreamSynchronize(s->ctx->stream);
    delete s;
    return RVE_OK;
}

int rve_gauss_point_features(rve_ctx c, rve_mesh m, int64_t G, const double* T_C, const double* c_wt,
                             const double* t_h, double* feat) {
    RVE_TRY(check_ctx(c));
    if (!m || G < 0 || (G > 0 && (!T_C || !c_wt || !t_h || !feat))) return RVE_ERR_INVALID_ARGUMENT;
    if (!m->have_materials) return RVE_ERR_STATE;
    if (G == 0) return RVE_OK;
    std::vector<double> w(G);
    RVE_TRY(rve_degradation_factor(c, G, T_C, c_wt, t_h, &m->deg, w.data()));
    const MaterialConsts& mc = m->mc;
    for (int64_t g = 0; g < G; ++g) {
        const double wy = m->deg.apply_to_yarn ? w[g] : 1.0;
        const double f[8] = {T_C[g], c_wt[g], std::log10(std::max(t_h[g], 1e-30)), mc.Em * w[g],
                             mc.E1 * wy, mc.E2 * wy, mc.G12 * wy, mc.km};
        std::memcpy(feat + 8 * g, f, sizeof(f));
    }
    return RVE_OK;
}

int rve_surrogate_train(rve_ctx c, rve_surrogate s, int64_t n, const double* feat, const double* Ct,
                        const double* Kt, const double* Dt, int epochs, int batch, double lr,
                        uint64_t seed, double* loss_history) {
    NvtxRange nvtx_("surrogate training: %lld points, %d members", (long long)n, s ? s->members : 0);
    RVE_TRY(check_ctx(c));
    if (!s || n < 64 || !feat || !Ct || !Kt || !Dt || epochs < 1 || batch < 64 || batch % 64 || !(lr > 0)) {
        set_error("rve_surrogate_train: invalid argument (n >= 64, batch a multiple of 64)");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t st = c->stream;
    // ---- normalisation from the data
    double mean[8] = {0}, var[8] = {0};
    for (int64_t i = 0; i < n; ++i)
        for (int k = 0; k < 8; ++k) mean[k] += feat[8 * i + k] / n;
    for (int64_t i = 0; i < n; ++i)
        for (int k = 0; k < 8; ++k) var[k] += (feat[8 * i + k] - mean[k]) * (feat[8 * i + k] - mean[k]) / n;
    for (int k = 0; k < 8; ++k) {
        s->feat_mean[k] = (float)mean[k];
        s->feat_std[k] = var[k] > 1e-30 * (mean[k] * mean[k] + 1e-30) ? (float)std::sqrt(var[k]) : 1.f;
    }
    double tr[3] = {0, 0, 0};
    for (int64_t i = 0; i < n; ++i) {
        for (int a = 0; a < 6; ++a) tr[0] += Ct[36 * i + 7 * a] / (6.0 * n);
        for (int a = 0; a < 3; ++a) {
            tr[1] += Kt[9 * i + 4 * a] / (3.0 * n);
            tr[2] += Dt[9 * i + 4 * a] / (3.0 * n);
        }
    }
    for (int b = 0; b < 3; ++b) s->ref[b] = tr[b];
    // targets: Cholesky factors of the normalised tensors, row-major lower triangles
    std::vector<float> tgt((size_t)n * NOUT);
    for (int64_t i = 0; i < n; ++i) {
        const double* src[3] = {Ct + 36 * i, Kt + 9 * i, Dt + 9 * i};
        const int sizes[3] = {6, 3, 3}, offs[3] = {0, 21, 27};
        for (int b = 0; b < 3; ++b) {
            const int nn = sizes[b];
            double A[6][6], L[6][6] = {};
            for (int r = 0; r < nn; ++r)
                for (int q = 0; q < nn; ++q) A[r][q] = 0.5 * (src[b][r * nn + q] + src[b][q * nn + r]) / s->ref[b];
            for (int j = 0; j < nn; ++j) {
                double d = A[j][j];
                for (int k = 0; k < j; ++k) d -= L[j][k] * L[j][k];
                if (!(d > 0)) {
                    set_error("rve_surrogate_train: a training tensor is not positive definite");
                    return RVE_ERR_NOT_SPD;
                }
                L[j][j] = std::sqrt(d);
                for (int r = j + 1; r < nn; ++r) {
                    double t = A[r][j];
                    for (int k = 0; k < j; ++k) t -= L[r][k] * L[j][k];
                    L[r][j] = t / L[j][j];
                }
            }
            int k = 0;
            for (int r = 0; r < nn; ++r)
                for (int q = 0; q <= r; ++q) tgt[i * NOUT + offs[b] + k++] = (float)L[r][q];
        }
    }
    // The factors of tensors normalised by their mean trace are O(1); an equal
    // scale for every entry makes the loss the squared error relative to the
    // tensor's own size (what the accuracy target is stated in).
    for (int o = 0; o < NOUT; ++o) s->sigma[o] = 1.f;
    // ---- device data: features and targets once, the row order of every epoch
    const int M = batch, nm = s->members;
    // The members train together; where their buffers (13 KB a row of the batch and member) do
    // not fit, in groups one after the other, which changes nothing but the time: each member
    // has its own row order and weights.
    TrainWork w;
    int group = nm;
    for (;;) {
        const int rc = train_work(s, group, M, w);
        if (rc == RVE_OK) break;
        if (rc != RVE_ERR_OUT_OF_MEMORY || group == 1) return rc;
        cudaGetLastError();
        group = (group + 1) / 2;
    }
    DevBuf dfeat, dtgt, dsig, dperm, dloss;
    RVE_TRY(upload_norm(s));
    RVE_TRY(upload(dfeat, feat, (size_t)n * 8, st));
    RVE_TRY(upload(dtgt, tgt.data(), tgt.size(), st));
    RVE_TRY(upload(dsig, s->sigma, NOUT, st));
    RVE_TRY(dperm.ensure((size_t)group * n * 4));
    RVE_TRY(dloss.ensure((size_t)epochs * nm * 4));
    RVE_CUDA(cudaMemsetAsync(dloss.p, 0, (size_t)epochs * nm * 4, st));
    const int64_t steps_per_epoch = n / M;
    std::vector<std::vector<int64_t>> perm(group);
    std::vector<int32_t> order((size_t)group * n);
    for (int first = 0; first < nm; first += group) {
        const int k = std::min(group, nm - first);
        std::vector<std::mt19937_64> rng;
        for (int e = 0; e < k; ++e) {
            rng.emplace_back(seed * 7919ull + (uint64_t)(first + e));
            perm[e].resize(n);
            std::iota(perm[e].begin(), perm[e].end(), 0);
        }
        int step = 0;
        for (int ep = 0; ep < epochs; ++ep) {
            for (int e = 0; e < k; ++e) {
                std::shuffle(perm[e].begin(), perm[e].end(), rng[e]);
                for (int64_t i = 0; i < n; ++i) order[(size_t)e * n + i] = (int32_t)perm[e][i];
            }
            // (a copy from pageable memory has left the vector when the call returns)
            RVE_CUDA(cudaMemcpyAsync(dperm.p, order.data(), (size_t)k * n * 4, cudaMemcpyHostToDevice, st));
            for (int64_t b = 0; b < steps_per_epoch; ++b) {
                const int32_t* rows[MAX_MEMBERS];
                float* loss[MAX_MEMBERS];
                for (int e = 0; e < k; ++e) {
                    rows[e] = dperm.as<int32_t>() + (size_t)e * n + b * M;
                    loss[e] = dloss.as<float>() + (size_t)ep * nm + first + e;
                }
                RVE_TRY(forward_backward(s, first, k, M, w, dfeat.as<double>(), dtgt.as<float>(), dsig.as<float>(),
                                         rows, loss));
                ++step;
                // cosine decay of the learning rate over all steps
                const double total = (double)epochs * steps_per_epoch;
                const double lr_t = lr * (0.02 + 0.98 * 0.5 * (1.0 + std::cos(M_PI * (step - 1) / total)));
                adam_step(s, first, k, w, (float)lr_t, step);
            }
        }
    }
    std::vector<float> lsum((size_t)epochs * nm);
    RVE_CUDA(cudaMemcpyAsync(lsum.data(), dloss.p, lsum.size() * 4, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaStreamSynchronize(st));
    std::vector<double> hist(epochs, 0.0);
    for (int e = 0; e < nm; ++e)
        for (int ep = 0; ep < epochs; ++ep) hist[ep] += lsum[(size_t)ep * nm + e] / steps_per_epoch / nm;
    RVE_CUDA(cudaGetLastError());
    if (loss_history) std::memcpy(loss_history, hist.data(), sizeof(double) * epochs);
    s->trained = true;
    return wait_status();
}

int rve_surrogate_gradients(rve_ctx c, rve_surrogate s, int member, int n, const double* feat,
                            const float* target_factors, float* grads, double* loss) {
    RVE_TRY(check_ctx(c));
    if (!s || member < 0 || member >= s->members || n < 1 || n % 64 || !feat || !target_factors || !grads) {
        set_error("rve_surrogate_gradients: invalid argument (n a positive multiple of 64)");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    cudaStream_t st = c->stream;
    TrainWork w;
    RVE_TRY(train_work(s, 1, n, w));
    DevBuf df, dt, dsig, dloss;
    RVE_TRY(upload_norm(s));
    RVE_TRY(upload(df, feat, (size_t)n * 8, st));
    RVE_TRY(upload(dt, target_factors, (size_t)n * NOUT, st));
    RVE_TRY(upload(dsig, s->sigma, NOUT, st));
    RVE_TRY(dloss.ensure(4));
    RVE_CUDA(cudaMemsetAsync(dloss.p, 0, 4, st));
    float* dl[1] = {dloss.as<float>()};
    RVE_TRY(forward_backward(s, member, 1, n, w, df.as<double>(), dt.as<float>(), dsig.as<float>(), nullptr, dl));
    std::vector<float> gT, gb;
    for (int q = 0; q < NLAYER; ++q) {
        const int K = LK[q], N = LN[q], nvalid = q == NLAYER - 1 ? NOUT : N;
        const int64_t o = layer_w_off(q);
        gT.resize((size_t)N * K);
        gb.resize(N);
        RVE_CUDA(cudaMemcpyAsync(gT.data(), w.gradT[0][q], gT.size() * 4, cudaMemcpyDeviceToHost, st));
        RVE_CUDA(cudaMemcpyAsync(gb.data(), w.gradb[0][q], gb.size() * 4, cudaMemcpyDeviceToHost, st));
        RVE_CUDA(cudaStreamSynchronize(st));
        for (int k = 0; k < K; ++k)
            for (int j = 0; j < N; ++j) grads[o + (int64_t)k * N + j] = j < nvalid ? gT[(size_t)j * K + k] : 0.f;
        for (int j = 0; j < N; ++j) grads[o + (int64_t)K * N + j] = j < nvalid ? gb[j] : 0.f;
    }
    float l = 0;
    RVE_CUDA(cudaMemcpyAsync(&l, dloss.p, 4, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaStreamSynchronize(st));
    if (loss) *loss = l;
    return wait_status();
}

// Ensemble prediction on device features: member tensors, mean and spread.
static int predict_dev(rve_surrogate s, int64_t n, const double* feat_dev, double* C_dev, double* K_dev,
                       double* D_dev, double* spread_dev) {
    NvtxRange nvtx_("surrogate inference: %lld points, %d members", (long long)n, s->members);
    cudaStream_t st = s->ctx->stream;
    const int64_t chunk = 65536, rows = std::min<int64_t>(chunk, (n + 63) / 64 * 64);
    const bool use_fused = s->fused && s->members <= mlp_fused_max_members();
    for (int l = 0; l < (use_fused ? 1 : NLAYER); ++l) RVE_TRY(s->H[l].ensure((size_t)rows * LK[l] * 2));
    RVE_TRY(s->zall.ensure((size_t)s->members * 64 * rows * 4));
    std::vector<const __nv_bfloat16*> wt;
    std::vector<const float*> bias;
    int64_t w_off[NLAYER];
    for (int l = 0; l < NLAYER; ++l) w_off[l] = layer_w_off(l);
    for (int e = 0; e < s->members; ++e) {
        wt.push_back(s->Wt[e].as<__nv_bfloat16>());
        for (int l = 0; l < NLAYER; ++l) bias.push_back(s->P[e].as<float>() + w_off[l] + (int64_t)LK[l] * LN[l]);
    }
    RVE_TRY(upload_norm(s));
    const float* norm = s->d_norm.as<float>();
    FeatureArgs fa;
    fa.rows[0] = nullptr;
    fa.X[0] = s->H[0].as<__nv_bfloat16>();
    for (int64_t off = 0; off < n; off += chunk) {
        const int nn = (int)std::min<int64_t>(chunk, n - off);
        const int M = ((nn + 63) / 64) * 64;
        launch_features(1, nn, M, KIN, feat_dev + off * 8, fa, norm, norm + 8, st);
        if (use_fused) {
            RVE_CUDA(launch_mlp_fused(M, s->members, s->H[0].as<__nv_bfloat16>(), wt.data(), w_off,
                                      bias.data(), s->zall.as<float>(), M, st));
            s->ctx->launches += 1;
        } else {
            for (int e = 0; e < s->members; ++e)
                for (int l = 0; l < NLAYER; ++l) {
                    const bool last = l == NLAYER - 1;
                    RVE_CUDA(launch_gemm_bf16(M, LN[l], LK[l], s->H[l].as<__nv_bfloat16>(), wt[e] + w_off[l],
                                              bias[e * NLAYER + l], last ? 4 : 1,
                                              last ? nullptr : s->H[l + 1].as<__nv_bfloat16>(),
                                              last ? s->zall.as<float>() + (size_t)e * 64 * M : nullptr, st));
                    s->ctx->launches += 1;
                }
        }
        launch_ensemble(nn, M, s->members, s->zall.as<float>(), (int64_t)64 * M, s->d_diag.as<uint8_t>(), s->ref[0],
                        s->ref[1], s->ref[2], C_dev + off * 36, K_dev + off * 9, D_dev + off * 9, spread_dev + off, st);
        s->ctx->launches += 2;
    }
    RVE_CUDA(cudaGetLastError());
    RVE_CUDA(cudaStreamSynchronize(st));   // the outputs are complete when the call returns
    return wait_status();
}

int rve_surrogate_predict(rve_ctx c, rve_surrogate s, int64_t n, const double* feat, double* C, double* K,
                          double* D, double* spread) {
    RVE_TRY(check_ctx(c));
    if (!s || n < 0 || (n > 0 && (!feat || !C || !K || !D || !spread))) return RVE_ERR_INVALID_ARGUMENT;
    if (!s->trained) {
        set_error("surrogate has not been trained or loaded");
        return RVE_ERR_STATE;
    }
    if (n == 0) return RVE_OK;
    cudaStream_t st = c->stream;
    DevBuf df, dC, dK, dD, dsp;
    RVE_TRY(upload(df, feat, (size_t)n * 8, st));
    RVE_TRY(dC.ensure((size_t)n * 36 * 8));
    RVE_TRY(dK.ensure((size_t)n * 9 * 8));
    RVE_TRY(dD.ensure((size_t)n * 9 * 8));
    RVE_TRY(dsp.ensure((size_t)n * 8));
    RVE_TRY(predict_dev(s, n, df.as<double>(), dC.as<double>(), dK.as<double>(), dD.as<double>(),
                        dsp.as<double>()));
    RVE_CUDA(cudaMemcpyAsync(C, dC.p, (size_t)n * 36 * 8, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaMemcpyAsync(K, dK.p, (size_t)n * 9 * 8, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaMemcpyAsync(D, dD.p, (size_t)n * 9 * 8, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaMemcpyAsync(spread, dsp.p, (size_t)n * 8, cudaMemcpyDeviceToHost, st));
    RVE_CUDA(cudaStreamSynchronize(st));
    return RVE_OK;
}

int rve_surrogate_set_fused(rve_ctx c, rve_surrogate s, int fused) {
    RVE_TRY(check_ctx(c));
    if (!s) return RVE_ERR_INVALID_ARGUMENT;
    s->fused = fused != 0;
    return RVE_OK;
}

int rve_surrogate_predict_dev(rve_ctx c, rve_surrogate s, int64_t n, const double* feat_dev, double* C_dev,
                              double* K_dev, double* D_dev, double* spread_dev) {
    RVE_TRY(check_ctx(c));
    if (!s || n < 0 || (n > 0 && (!feat_dev || !C_dev || !K_dev || !D_dev || !spread_dev)))
        return RVE_ERR_INVALID_ARGUMENT;
    if (!s->trained) {
        set_error("surrogate has not been trained or loaded");
        return RVE_ERR_STATE;
    }
    if (n == 0) return RVE_OK;
    RVE_TRY(predict_dev(s, n, feat_dev, C_dev, K_dev, D_dev, spread_dev));
    RVE_CUDA(cudaGetLastError());
    return RVE_OK;
}

int rve_debug_surrogate_work_limit(rve_ctx c, rve_surrogate s, int64_t bytes) {
    RVE_TRY(check_ctx(c));
    if (!s || bytes < 0) return RVE_ERR_INVALID_ARGUMENT;
    s->work_limit = (size_t)bytes;
    return RVE_OK;
}

int rve_debug_gemm_timeout(int set) { return gemm_tc_set_timed_out(set != 0 ? 1 : 0); }

int rve_surrogate_get_params(rve_ctx c, rve_surrogate s, float* buf, int64_t* len) {
    RVE_TRY(check_ctx(c));
    if (!s || !len) return RVE_ERR_INVALID_ARGUMENT;
    const int64_t np = n_params();
    const int64_t need = HEADER + (int64_t)s->members * np;
    if (!buf) {
        *len = need;
        return RVE_OK;
    }
    if (*len < need) return RVE_ERR_INVALID_ARGUMENT;
    std::memcpy(buf, s->feat_mean, 32);
    std::memcpy(buf + 8, s->feat_std, 32);
    std::memcpy(buf + 16, s->sigma, 33 * 4);
    for (int b = 0; b < 3; ++b) buf[49 + b] = (float)s->ref[b];
    for (int e = 0; e < s->members; ++e)
        RVE_CUDA(cudaMemcpyAsync(buf + HEADER + e * np, s->P[e].p, np * 4, cudaMemcpyDeviceToHost, c->stream));
    RVE_CUDA(cudaStreamSynchronize(c->stream));
    *len = need;
    return RVE_OK;
}

int rve_surrogate_set_params(rve_ctx c, rve_surrogate s, const float* buf, int64_t len) {
    RVE_TRY(check_ctx(c));
    const int64_t np = n_params();
    if (!s || !buf || len != HEADER + (int64_t)s->members * np) {
        set_error("rve_surrogate_set_params: length does not match the ensemble size");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    std::memcpy(s->feat_mean, buf, 32);
    std::memcpy(s->feat_std, buf + 8, 32);
    std::memcpy(s->sigma, buf + 16, 33 * 4);
    for (int b = 0; b < 3; ++b) s->ref[b] = buf[49 + b];
    for (int e = 0; e < s->members; ++e) {
        RVE_CUDA(cudaMemcpyAsync(s->P[e].p, buf + HEADER + e * np, np * 4, cudaMemcpyHostToDevice, c->stream));
        RVE_TRY(refresh_bf16(s, e));
    }
    RVE_CUDA(cudaStreamSynchronize(c->stream));
    s->trained = true;
    return RVE_OK;
}

int macro_update_gauss_points_surrogate(rve_ctx c, const rve_mesh* meshes, const rve_surrogate* surrogates,
                                        int n_meshes, double tau, int64_t G, const double* T_C,
                                        const double* c_wt, const double* t_h, const int32_t* mesh_id,
                                        double* C, double* K, double* D, int32_t* status, uint8_t* fallback,
                                        rve_stats* st) {
    RVE_TRY(check_ctx(c));
    if (!meshes || !surrogates || n_meshes <= 0 || G < 0 || !(tau >= 0) ||
        (G > 0 && (!T_C || !c_wt || !t_h || !mesh_id || !C || !K || !D || !status || !fallback))) {
        set_error("macro_update_gauss_points_surrogate: invalid argument");
        return RVE_ERR_INVALID_ARGUMENT;
    }
    auto t0 = std::chrono::steady_clock::now();
    const int64_t l0 = c->launches;
    if (st) {
        std::memset(st, 0, sizeof(*st));
        st->converged = 1;
    }
    cudaStream_t s = c->stream;
    std::vector<std::vector<int64_t>> groups(n_meshes);
    for (int64_t g = 0; g < G; ++g) {
        if (mesh_id[g] < 0 || mesh_id[g] >= n_meshes) return RVE_ERR_INVALID_ARGUMENT;
        groups[mesh_id[g]].push_back(g);
    }
    std::vector<int64_t> fb_idx;
    std::vector<int32_t> fb_mesh;
    for (int mi = 0; mi < n_meshes; ++mi) {
        auto& grp = groups[mi];
        if (grp.empty()) continue;
        rve_surrogate sg = surrogates[mi];
        if (!sg || !sg->trained) {
            for (auto g : grp) {
                fb_idx.push_back(g);
                fb_mesh.push_back(mi);
            }
            continue;
        }
        const int64_t n = (int64_t)grp.size();
        std::vector<double> T(n), cc(n), tt(n), feat((size_t)n * 8);
        for (int64_t i = 0; i < n; ++i) {
            T[i] = T_C[grp[i]];
            cc[i] = c_wt[grp[i]];
            tt[i] = t_h[grp[i]];
        }
        RVE_TRY(rve_gauss_point_features(c, meshes[mi], n, T.data(), cc.data(), tt.data(), feat.data()));
        std::vector<double> Cp((size_t)n * 36), Kp((size_t)n * 9), Dp((size_t)n * 9), spr(n);
        RVE_TRY(rve_surrogate_predict(c, sg, n, feat.data(), Cp.data(), Kp.data(), Dp.data(), spr.data()));
        for (int64_t i = 0; i < n; ++i) {
            const int64_t g = grp[i];
            if (!(spr[i] <= tau)) {
                fb_idx.push_back(g);
                fb_mesh.push_back(mi);
                continue;
            }
            std::memcpy(C + 36 * g, &Cp[36 * i], 36 * 8);
            std::memcpy(K + 9 * g, &Kp[9 * i], 9 * 8);
            std::memcpy(D + 9 * g, &Dp[9 * i], 9 * 8);
            status[g] = RVE_OK;
            fallback[g] = 0;
        }
    }
    int rc = RVE_OK;
    if (!fb_idx.empty()) {
        const int64_t nf = (int64_t)fb_idx.size();
        std::vector<double> T(nf), cc(nf), tt(nf), Cf((size_t)nf * 36), Kf((size_t)nf * 9), Df((size_t)nf * 9);
        std::vector<int32_t> sf(nf);
        for (int64_t i = 0; i < nf; ++i) {
            T[i] = T_C[fb_idx[i]];
            cc[i] = c_wt[fb_idx[i]];
            tt[i] = t_h[fb_idx[i]];
        }
        rve_stats fs;
        rc = macro_update_gauss_points(c, meshes, n_meshes, nf, T.data(), cc.data(), tt.data(), fb_mesh.data(),
                                       Cf.data(), Kf.data(), Df.data(), sf.data(), RVE_MODE_PCG, &fs);
        if (rc != RVE_OK && rc != RVE_ERR_NOT_CONVERGED && rc != RVE_ERR_NUMERIC) return rc;
        for (int64_t i = 0; i < nf; ++i) {
            const int64_t g = fb_idx[i];
            std::memcpy(C + 36 * g, &Cf[36 * i], 36 * 8);
            std::memcpy(K + 9 * g, &Kf[9 * i], 9 * 8);
            std::memcpy(D + 9 * g, &Df[9 * i], 9 * 8);
            status[g] = sf[i];
            fallback[g] = 1;
        }
        if (st) {
            *st = fs;
        }
    }
    if (st) {
        st->seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        st->kernel_launches = c->launches - l0;
    }
    RVE_TRY(wait_status());
    return rc;
}

}  // extern "C"
