// Learned warm start: a three-layer message-passing network on the pattern of
// C that predicts a starting factor R0 (unit rows) for the Burer-Monteiro
// solve, trained on the factors the solver returns.  The paper starts from a
// random factor; this network is an addition of this library.
//
// Network (definition shared with the CPU oracle of the tests; F = 16 input
// features, H = 32 hidden, r_out outputs, w_ij = C_ij for i != j,
// s_i = sum_j |w_ij|):
//   x_i  = [1, log(1+deg_i)/4, sum_j w_ij / s_i, C_ii / s_i, 12 SplitMix64 normals]
//   m_i  = sum_j (w_ij / s_i) h_j ;  h_i <- relu(W_s h_i + W_n m_i + b)   (3 layers)
//   o_i  = W_o h_i + b_o ;  r_hat_i = o_i / ||o_i||
//   loss = mean over edges i<j of (r_hat_i . r_hat_j - X*_ij)^2
// Activations are stored in bf16 (or float for checking) with float
// arithmetic; weights are float masters, rounded to bf16 for the forward pass
// in bf16 mode; gradients, Adam moments and every reduction are float/double.
// Weight gradients are summed per block in a fixed order and folded over the
// blocks in a fixed order (deterministic).
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/lorads.h"
#include "common.cuh"
#include "gnn_kernels.cuh"

using namespace lorads;
using namespace lorads::gnn;

namespace {

int64_t param_count(int r_out) {
    int64_t p = 0;
    int f = kF;
    for (int l = 0; l < kLayers; ++l) {
        p += 2LL * kH * f + kH;
        f = kH;
    }
    return p + (int64_t)r_out * kH + r_out;
}

int64_t layer_offset(int l) {
    int64_t p = 0;
    int f = kF;
    for (int q = 0; q < l; ++q) {
        p += 2LL * kH * f + kH;
        f = kH;
    }
    return p;
}

}  // namespace

// ====================================================================== object
struct lorads_gnn {
    int r_out = 0, rs = 0;       // outputs, and their row width (a multiple of 4)
    int act = LORADS_BF16;
    int64_t P = 0;
    cudaStream_t stream = nullptr;
    int num_sms = 0, nb = 0;
    std::string err;
    float* theta = nullptr;
    float* grad = nullptr;
    float* m1 = nullptr;
    float* m2 = nullptr;
    float* gpart = nullptr;
    int64_t step = 0;
    // per-node workspace (grown on demand)
    int64_t cap = 0, cap_back = 0;   // nodes of the forward arrays, and of the training step's
    void* x = nullptr;           // n x F  (activation type)
    void* h[kLayers] = {};       // n x H
    void* m[kLayers] = {};       // n x F_in
    float* inv_s = nullptr;
    float* rhat = nullptr;       // n x rs
    float* onrm = nullptr;
    float* d_o = nullptr;        // n x rs: gradient in the outputs before their normalisation
    float* dh[2] = {};           // n x H: W_s^T du and
    float* dm[2] = {};           // n x H: W_n^T du of the layer above, two in turn
    double* lpart = nullptr;     // loss partials
};

namespace {

#define GCK(call)                                                                          \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            cudaGetLastError();                                                            \
            g->err = std::string(#call) + ": " + cudaGetErrorString(e_);                   \
            return e_ == cudaErrorMemoryAllocation ? LORADS_ERR_OOM : LORADS_ERR_CUDA;     \
        }                                                                                  \
    } while (0)

void gfree(void* p) {
    if (p) cudaFree(p);
}

void free_back(lorads_gnn* g) {
    gfree(g->rhat); gfree(g->onrm); gfree(g->d_o);
    g->rhat = g->onrm = g->d_o = nullptr;
    for (int q = 0; q < 2; ++q) {
        gfree(g->dh[q]);
        gfree(g->dm[q]);
        g->dh[q] = g->dm[q] = nullptr;
    }
    for (int l = 0; l < kLayers; ++l) {
        gfree(g->m[l]);
        g->m[l] = nullptr;
    }
    g->cap_back = 0;
}

void free_ws(lorads_gnn* g) {
    free_back(g);
    gfree(g->x); gfree(g->inv_s);
    g->x = nullptr;
    g->inv_s = nullptr;
    for (int l = 0; l < kLayers; ++l) {
        gfree(g->h[l]);
        g->h[l] = nullptr;
    }
    g->cap = 0;
}

// Node arrays for n nodes; `train`: also what the backward pass keeps and writes.
lorads_status ensure_ws(lorads_gnn* g, int64_t n, bool train) {
    const size_t ea = g->act == LORADS_BF16 ? 2 : 4;
    if (n > g->cap) {
        free_ws(g);
        GCK(cudaMalloc(&g->x, (size_t)n * kF * ea));
        for (int l = 0; l < kLayers; ++l) GCK(cudaMalloc(&g->h[l], (size_t)n * kH * ea));
        GCK(cudaMalloc(&g->inv_s, (size_t)n * 4));
        g->cap = n;
    }
    if (train && n > g->cap_back) {
        free_back(g);
        for (int l = 0; l < kLayers; ++l) GCK(cudaMalloc(&g->m[l], (size_t)n * kH * ea));
        GCK(cudaMalloc(&g->rhat, (size_t)n * g->rs * 4));
        GCK(cudaMalloc(&g->onrm, (size_t)n * 4));
        GCK(cudaMalloc(&g->d_o, (size_t)n * g->rs * 4));
        for (int q = 0; q < 2; ++q) {
            GCK(cudaMalloc(&g->dh[q], (size_t)n * kH * 4));
            GCK(cudaMalloc(&g->dm[q], (size_t)n * kH * 4));
        }
        g->cap_back = n;
    }
    return LORADS_OK;
}

int grid_for(const lorads_gnn* g, int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    return (int)std::min<int64_t>(b, (int64_t)g->num_sms * 8);
}

// Forward pass: features, three layers, output rows.  R != null: predict (the FP64 rows
// alone); else everything the backward pass reads is kept.
template <typename TA>
void forward(lorads_gnn* g, int64_t n, const int64_t* rp, const int32_t* ci, const double* cv, uint64_t seed,
             double* R, int ld) {
    cudaStream_t s = g->stream;
    TA* x = static_cast<TA*>(g->x);
    TA *h1 = static_cast<TA*>(g->h[0]), *h2 = static_cast<TA*>(g->h[1]), *h3 = static_cast<TA*>(g->h[2]);
    const bool keep = R == nullptr;
    auto m = [&](int l) { return keep ? static_cast<TA*>(g->m[l]) : nullptr; };
    const int grid = grid_for(g, n, kFwdTile * kFwdThreads / 32);
    k_prep<TA><<<grid_for(g, n, kThreadsG), kThreadsG, 0, s>>>(n, rp, ci, cv, seed, x, g->inv_s);
    k_layer<TA, kF, false><<<grid, kFwdThreads, 0, s>>>(n, rp, ci, cv, g->inv_s, x, g->theta + layer_offset(0), m(0), h1,
                                                      nullptr, 0, nullptr, 0, nullptr, nullptr, 0);
    k_layer<TA, kH, false><<<grid, kFwdThreads, 0, s>>>(n, rp, ci, cv, g->inv_s, h1, g->theta + layer_offset(1), m(1), h2,
                                                      nullptr, 0, nullptr, 0, nullptr, nullptr, 0);
    k_layer<TA, kH, true><<<grid, kFwdThreads, 0, s>>>(n, rp, ci, cv, g->inv_s, h2, g->theta + layer_offset(2), m(2),
                                                     keep ? h3 : nullptr, g->theta + layer_offset(kLayers), g->r_out,
                                                     keep ? g->rhat : nullptr, g->rs, keep ? g->onrm : nullptr, R, ld);
}

// Backward pass from do; returns the blocks of partial sums to fold.
template <typename TA>
int backward(lorads_gnn* g, int64_t n, const int64_t* rp, const int32_t* ci, const double* cv) {
    cudaStream_t s = g->stream;
    // blocks: every block with the same number of tiles (or one less), one resident wave
    const int64_t tiles = (n + kBackTile - 1) / kBackTile, rounds = (tiles + g->nb - 1) / g->nb;
    const int nb = (int)((tiles + rounds - 1) / rounds);
    const float* th_o = g->theta + layer_offset(kLayers);
    const TA* in[kLayers] = {static_cast<const TA*>(g->x), static_cast<const TA*>(g->h[0]),
                             static_cast<const TA*>(g->h[1])};
    auto h = [&](int l) { return static_cast<const TA*>(g->h[l]); };
    auto m = [&](int l) { return static_cast<const TA*>(g->m[l]); };
    k_back<TA, kH, true><<<nb, kThreadsG, 0, s>>>(n, rp, ci, cv, g->inv_s, in[2], m(2), h(2), g->d_o, g->rs, g->r_out,
                                                  th_o, nullptr, nullptr, g->theta + layer_offset(2), g->dh[0],
                                                  g->dm[0], g->gpart, g->P, layer_offset(2), layer_offset(kLayers));
    k_back<TA, kH, false><<<nb, kThreadsG, 0, s>>>(n, rp, ci, cv, g->inv_s, in[1], m(1), h(1), nullptr, 0, 0, nullptr,
                                                   g->dh[0], g->dm[0], g->theta + layer_offset(1), g->dh[1], g->dm[1],
                                                   g->gpart, g->P, layer_offset(1), 0);
    k_back<TA, kF, false><<<nb, kThreadsG, 0, s>>>(n, rp, ci, cv, g->inv_s, in[0], m(0), h(0), nullptr, 0, 0, nullptr,
                                                   g->dh[1], g->dm[1], g->theta + layer_offset(0), nullptr, nullptr,
                                                   g->gpart, g->P, layer_offset(0), 0);
    return nb;
}

lorads_status check(lorads_gnn* g, const char* what) {
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g->err = std::string(what) + ": " + cudaGetErrorString(e);
        return LORADS_ERR_CUDA;
    }
    return LORADS_OK;
}

lorads_status check_graph(lorads_gnn* g, int64_t n, const void* rp, const void* ci, const void* cv) {
    if (n < 1 || n > INT32_MAX) {
        g->err = "n must be in [1, 2^31)";
        return LORADS_ERR_INVALID_ARG;
    }
    if (!rp || !ci || !cv) {
        g->err = "null graph pointer";
        return LORADS_ERR_INVALID_ARG;
    }
    return LORADS_OK;
}

thread_local std::string g_gnn_create_error;

}  // namespace

extern "C" int64_t lorads_gnn_param_count(int32_t r_out) {
    return (r_out < 1 || r_out > kMaxOut) ? -1 : param_count(r_out);
}

extern "C" const char* lorads_gnn_last_error(const lorads_gnn* g) { return g ? g->err.c_str() : "null network"; }

extern "C" const char* lorads_gnn_create_error(void) { return g_gnn_create_error.c_str(); }

extern "C" void lorads_gnn_destroy(lorads_gnn* g) {
    if (!g) return;
    if (g->stream) cudaStreamSynchronize(g->stream);
    free_ws(g);
    gfree(g->theta); gfree(g->grad); gfree(g->m1); gfree(g->m2); gfree(g->gpart); gfree(g->lpart);
    delete g;
}

extern "C" lorads_status lorads_gnn_create(lorads_gnn** out, int32_t r_out, int32_t act_prec, const float* theta0,
                                           void* cuda_stream) {
    if (!out) return LORADS_ERR_INVALID_ARG;
    *out = nullptr;
    if (r_out < 1 || r_out > kMaxOut) {
        g_gnn_create_error = "r_out must be in [1, 32]";
        return LORADS_ERR_INVALID_ARG;
    }
    if (act_prec != LORADS_BF16 && act_prec != LORADS_FP32) {
        g_gnn_create_error = "act_prec must be LORADS_BF16 or LORADS_FP32";
        return LORADS_ERR_INVALID_ARG;
    }
    if (!theta0) {
        g_gnn_create_error = "theta0 (initial parameters) is NULL";
        return LORADS_ERR_INVALID_ARG;
    }
    lorads_gnn* g = new (std::nothrow) lorads_gnn();
    if (!g) return LORADS_ERR_OOM;
    g->r_out = r_out;
    g->rs = (r_out + 3) / 4 * 4;
    g->act = act_prec;
    g->P = param_count(r_out);
    g->stream = static_cast<cudaStream_t>(cuda_stream);
    auto fail = [&](lorads_status s) {
        g_gnn_create_error = g->err;
        lorads_gnn_destroy(g);
        return s;
    };
#define GCREATE(call)                                                                      \
    do {                                                                                   \
        cudaError_t e_ = (call);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            cudaGetLastError();                                                            \
            g->err = std::string(#call) + ": " + cudaGetErrorString(e_);                   \
            return fail(e_ == cudaErrorMemoryAllocation ? LORADS_ERR_OOM : LORADS_ERR_CUDA); \
        }                                                                                  \
    } while (0)
    int dev = 0;
    GCREATE(cudaGetDevice(&dev));
    GCREATE(cudaDeviceGetAttribute(&g->num_sms, cudaDevAttrMultiProcessorCount, dev));
    g->nb = g->num_sms * kBackBlocks;
    const size_t pb = (size_t)g->P * sizeof(float);
    GCREATE(cudaMalloc(&g->theta, pb));
    GCREATE(cudaMalloc(&g->grad, pb));
    GCREATE(cudaMalloc(&g->m1, pb));
    GCREATE(cudaMalloc(&g->m2, pb));
    GCREATE(cudaMalloc(&g->gpart, pb * g->nb));
    GCREATE(cudaMalloc(&g->lpart, sizeof(double) * g->num_sms * 8));
    // on the caller's stream, which need not wait for the default one
    GCREATE(cudaMemcpyAsync(g->theta, theta0, pb, cudaMemcpyHostToDevice, g->stream));
    GCREATE(cudaMemsetAsync(g->m1, 0, pb, g->stream));
    GCREATE(cudaMemsetAsync(g->m2, 0, pb, g->stream));
    GCREATE(cudaMemsetAsync(g->grad, 0, pb, g->stream));
    GCREATE(cudaStreamSynchronize(g->stream));
#undef GCREATE
    *out = g;
    return LORADS_OK;
}

extern "C" lorads_status lorads_gnn_get_params(lorads_gnn* g, float* theta_host, int64_t count) {
    if (!g || !theta_host || count < g->P) return LORADS_ERR_INVALID_ARG;
    GCK(cudaStreamSynchronize(g->stream));
    GCK(cudaMemcpy(theta_host, g->theta, g->P * sizeof(float), cudaMemcpyDeviceToHost));
    return LORADS_OK;
}

extern "C" lorads_status lorads_gnn_set_params(lorads_gnn* g, const float* theta_host, int64_t count) {
    if (!g || !theta_host || count < g->P) return LORADS_ERR_INVALID_ARG;
    GCK(cudaMemcpyAsync(g->theta, theta_host, g->P * sizeof(float), cudaMemcpyHostToDevice, g->stream));
    GCK(cudaMemsetAsync(g->m1, 0, g->P * sizeof(float), g->stream));
    GCK(cudaMemsetAsync(g->m2, 0, g->P * sizeof(float), g->stream));
    GCK(cudaStreamSynchronize(g->stream));
    g->step = 0;
    return LORADS_OK;
}

extern "C" lorads_status lorads_gnn_predict(lorads_gnn* g, int64_t n, const int64_t* c_rowptr,
                                            const int32_t* c_colind, const double* c_val, uint64_t feature_seed,
                                            int32_t ld, double* R_out) {
    if (!g) return LORADS_ERR_INVALID_ARG;
    lorads_status s = check_graph(g, n, c_rowptr, c_colind, c_val);
    if (s != LORADS_OK) return s;
    if (!R_out || ld < g->r_out) {
        g->err = "R_out must be a device n x ld FP64 array with ld >= r_out";
        return LORADS_ERR_INVALID_ARG;
    }
    if ((s = ensure_ws(g, n, false)) != LORADS_OK) return s;
    if (g->act == LORADS_BF16) forward<__nv_bfloat16>(g, n, c_rowptr, c_colind, c_val, feature_seed, R_out, ld);
    else forward<float>(g, n, c_rowptr, c_colind, c_val, feature_seed, R_out, ld);
    return check(g, "gnn forward");
}

extern "C" lorads_status lorads_gnn_edge_targets(int64_t n, const int64_t* c_rowptr, const int32_t* c_colind,
                                                 const double* R, int32_t r, int32_t ld, float* targets,
                                                 void* cuda_stream) {
    if (n < 1 || !c_rowptr || !c_colind || !R || !targets || r < 1 || ld < r) return LORADS_ERR_INVALID_ARG;
    const int grid = (int)std::min<int64_t>((n + 255) / 256, 4096);
    k_targets<<<grid, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(n, c_rowptr, c_colind, R, r, ld,
                                                                               targets);
    return cudaGetLastError() == cudaSuccess ? LORADS_OK : LORADS_ERR_CUDA;
}

extern "C" lorads_status lorads_gnn_train_step(lorads_gnn* g, int64_t n, const int64_t* c_rowptr,
                                               const int32_t* c_colind, const double* c_val, uint64_t feature_seed,
                                               const float* targets, int64_t n_edges, float lr, double* loss_out,
                                               float* grad_out) {
    if (!g) return LORADS_ERR_INVALID_ARG;
    lorads_status s = check_graph(g, n, c_rowptr, c_colind, c_val);
    if (s != LORADS_OK) return s;
    if (!targets || n_edges < 1 || !(lr >= 0.0f)) {
        g->err = "targets must be given, n_edges >= 1 and lr >= 0";
        return LORADS_ERR_INVALID_ARG;
    }
    if ((s = ensure_ws(g, n, true)) != LORADS_OK) return s;
    const bool bf = g->act == LORADS_BF16;
    if (bf) forward<__nv_bfloat16>(g, n, c_rowptr, c_colind, c_val, feature_seed, nullptr, 0);
    else forward<float>(g, n, c_rowptr, c_colind, c_val, feature_seed, nullptr, 0);
    const int nbl = grid_for(g, n * 8, kThreadsG);
    k_loss<<<nbl, kThreadsG, 0, g->stream>>>(n, c_rowptr, c_colind, g->rhat, g->rs, g->onrm, targets,
                                             (float)(2.0 / (double)n_edges), g->d_o, g->lpart);
    const int nb = bf ? backward<__nv_bfloat16>(g, n, c_rowptr, c_colind, c_val)
                      : backward<float>(g, n, c_rowptr, c_colind, c_val);
    const float b1 = 0.9f, b2 = 0.999f;
    if (lr > 0.0f) g->step += 1;
    const float c1 = 1.0f - std::pow(b1, (float)g->step), c2 = 1.0f - std::pow(b2, (float)g->step);
    k_fold_adam<<<(int)((g->P + 31) / 32), 32 * kFoldSlices, 0, g->stream>>>(g->gpart, nb, g->P, g->grad, grad_out, g->theta,
                                                                      g->m1, g->m2, lr, b1, b2, 1e-8f, c1, c2);
    if ((s = check(g, "gnn train step")) != LORADS_OK) return s;
    if (loss_out) {
        std::vector<double> lp(nbl);
        GCK(cudaMemcpyAsync(lp.data(), g->lpart, nbl * sizeof(double), cudaMemcpyDeviceToHost, g->stream));
        GCK(cudaStreamSynchronize(g->stream));
        double L = 0.0;
        for (double v : lp) L += v;
        *loss_out = L / (double)n_edges;
    }
    return LORADS_OK;
}
