// Kernels of the learned warm start (gnn.cu): node features, fused message-passing
// layers, the loss, and the fused backward pass.
#pragma once

#include <math.h>
#include <type_traits>
#include "common.cuh"
#include "cons.cuh"
#include "control_dev.cuh"

namespace lorads {
namespace gnn {

constexpr int kF = 16;            // input features
constexpr int kStruct = 4;        // structural features
constexpr int kH = 32;            // hidden width
constexpr int kLayers = 3;
constexpr int kMaxOut = 32;       // r_out <= 32
constexpr uint64_t kFeatureStream = 0x474E4E;
constexpr int kThreadsG = 256;
constexpr int kFwdNodes = 2;                // nodes a thread of the forward layers computes
constexpr int kFwdTile = 4 * kFwdNodes;     // nodes of a warp's tile
constexpr int kFwdBlocks = 8;               // resident blocks per SM of the forward layers
constexpr int kFwdThreads = 128;
constexpr int kBackTile = 32;     // nodes per tile of the backward layers
constexpr int kBackBlocks = 4;    // resident blocks per SM of the backward layers
constexpr int kFoldSlices = 16;

__device__ __forceinline__ float bf16_round(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

template <typename TA> constexpr bool is_bf16() { return std::is_same<TA, __nv_bfloat16>::value; }
template <typename TA> __device__ __forceinline__ float weight(float w) {
    return is_bf16<TA>() ? bf16_round(w) : w;
}
template <typename TA> __device__ __forceinline__ TA to_act(float v) { return TA(v); }
template <> __device__ __forceinline__ __nv_bfloat16 to_act<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
// value an activation has once stored
template <typename TA> __device__ __forceinline__ float stored(float v) { return is_bf16<TA>() ? bf16_round(v) : v; }

// float to double by moving the fields (the conversion runs on the FP64 pipe, 64 times
// slower); subnormals, infinities and NaN take the conversion.
__device__ __forceinline__ double widen(float f) {
    const uint32_t b = __float_as_uint(f);
    const uint32_t e = (b >> 23) & 255u;
    if ((b << 1) == 0u) return __hiloint2double((int)b, 0);
    if (e == 0u || e == 255u) return (double)f;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20))), (int)(b << 29));
}

// ------------------------------------------------------------------ features
// FP64 normal, out of line: its code is large and, for bf16 features, seldom run.
__device__ __noinline__ float normal_slow(uint64_t base, int64_t e) { return (float)normal_at(base, e); }

// (float)normal_at(base, e) rounded to bf16, without FP64 where its float evaluation
// decides the rounding (Ziv's rounding test): the float value below is within 16 ulp of
// the exact one, and rounding to bf16 is the same for every float within 16 ulp unless a
// tie lies among them (1 value in 2,000), or the cosine is so near its zero that the
// argument's own rounding in normal_at shows (1 in 10^5): *sure says that neither is so.  The
// error in units of 2^-24: an argument rounded once from an integer (1, times 1.44 through
// the logarithm), logf or log1pf (1 ulp: 2), the root (half of these, and 1), the angle (1)
// and sinpif or cospif (2 ulp: 4), the product (1): below 10 units, at most 10 ulp.
// The features of 1e6 nodes: 1.72 ms in FP64, 0.21 ms so (of which the FP64 sums of the weights and their reciprocal take 0.08).
__device__ __forceinline__ __nv_bfloat16 normal_bf16(uint64_t base, int64_t e, bool* sure) {
    const uint64_t golden = 0x9E3779B97F4A7C15ull;
    const uint64_t a = (splitmix_out(base + (uint64_t)(2 * e + 1) * golden) >> 11) + 1;      // u1 2^53
    const uint64_t c = splitmix_out(base + (uint64_t)(2 * e + 2) * golden) >> 11;            // u2 2^53
    const uint64_t one = 1ull << 53;
    const float inv53 = 1.1102230246251565e-16f;
    const float l = a > one / 2 ? -2.f * log1pf(-((float)(one - a) * inv53)) : -2.f * logf((float)a * inv53);
    // cos(2 pi u2): quadrant q and the angle (pi/2) t / 2^51 inside it, by its near axis
    const uint32_t q = (uint32_t)(c >> 51);
    const uint64_t t = c & ((1ull << 51) - 1);
    const bool odd = (q & 1u) != 0;                              // cos in even quadrants, sin in odd ones
    const bool far = t > (1ull << 50);
    const uint64_t w = far ? (1ull << 51) - t : t;
    const float x = (float)w * (0.5f / 2251799813685248.f);      // half turns, at most 1/4
    const bool use_sin = odd != far;
    float v = use_sin ? sinpif(x) : cospif(x);
    if (q == 1u || q == 2u) v = -v;
    const float r = sqrtf(l) * v;
    const uint32_t low = __float_as_uint(r) & 0xffffu;
    const bool near_tie = low - (0x8000u - 16u) <= 32u;
    *sure = !(near_tie || a == one || (use_sin && w < (1ull << 34)));
    return __float2bfloat16_rn(r);
}

// A warp takes 32 nodes: lane = node for the structural features, then the nodes' normals
// over all lanes.  The normals that normal_bf16 leaves undecided are listed and done in FP64
// by the block together at the end (a warp that stopped for each of its own spent a fifth of
// its FP64 time on one lane's work).  log(1 + deg) of the degrees below
// kDegTable comes from a table filled by the block (the same FP64 call, once per degree
// instead of once per node); the features go through shared memory and are stored in whole
// lines.
constexpr int kDegTable = 64;
__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 a, __nv_bfloat16 b) {
    return (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
}
template <typename TA>
__global__ void __launch_bounds__(kThreadsG)
k_prep(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci, const double* __restrict__ cv,
       uint64_t seed, TA* __restrict__ x, float* __restrict__ inv_s) {
    constexpr int PW = 4 / (int)sizeof(TA), W = kF / PW;         // features a word, words a node
    constexpr int WS = kStruct / PW, WN = W - WS;                // structural words, words of normals
    constexpr int kList = 256;
    __shared__ float s_log[kDegTable];
    __shared__ int64_t s_list[kList];
    __shared__ int s_listed;
    __shared__ uint32_t s_x[kThreadsG / 32][32][W + 1];
    if (threadIdx.x < kDegTable) s_log[threadIdx.x] = (float)(log1p((double)threadIdx.x) / 4.0);
    if (threadIdx.x == 0) s_listed = 0;
    __syncthreads();
    const uint64_t golden = 0x9E3779B97F4A7C15ull;
    const uint64_t base = seed ^ (kFeatureStream * golden);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nwarps = (int64_t)gridDim.x * (kThreadsG / 32);
    for (int64_t w0 = (blockIdx.x * (int64_t)(kThreadsG / 32) + warp) * 32; w0 < n; w0 += nwarps * 32) {
        const int nodes = n - w0 < 32 ? (int)(n - w0) : 32;
        if (lane < nodes) {
            const int64_t i = w0 + lane;
            double s = 0, ws = 0, dg = 0;
            int deg = 0;
            const int64_t e1 = rp[i + 1];
            for (int64_t e = rp[i]; e < e1; ++e) {
                const double w = cv[e];
                if (ci[e] == i) {
                    dg += w;
                } else {
                    deg += 1;
                    s += fabs(w);
                    ws += w;
                }
            }
            const double is = s > 0 ? 1.0 / s : 0.0;
            inv_s[i] = (float)is;
            const float f0 = 1.0f, f1 = deg < kDegTable ? s_log[deg] : (float)(log1p((double)deg) / 4.0);
            const float f2 = (float)(ws * is), f3 = (float)(dg * is);
            uint32_t* row = s_x[warp][lane];
            if constexpr (is_bf16<TA>()) {
                row[0] = pack_bf16(to_act<TA>(f0), to_act<TA>(f1));
                row[1] = pack_bf16(to_act<TA>(f2), to_act<TA>(f3));
            } else {
                row[0] = __float_as_uint(f0);
                row[1] = __float_as_uint(f1);
                row[2] = __float_as_uint(f2);
                row[3] = __float_as_uint(f3);
            }
        }
#pragma unroll 1
        for (int q = lane; q < nodes * WN; q += 32) {
            const int u = q / WN, k = q - u * WN;
            const int64_t e = (w0 + u) * (kF - kStruct) + k * PW;
            uint32_t word;
            if constexpr (is_bf16<TA>()) {
                __nv_bfloat16 f[2];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    bool sure;
                    f[h] = normal_bf16(base, e + h, &sure);
                    if (!sure) {
                        const int at = atomicAdd(&s_listed, 1);
                        if (at < kList) s_list[at] = e + h;
                        else f[h] = __float2bfloat16_rn(normal_slow(base, e + h));
                    }
                }
                word = pack_bf16(f[0], f[1]);
            } else {
                word = __float_as_uint(normal_slow(base, e));
            }
            s_x[warp][u][WS + k] = word;
        }
        __syncwarp();
        uint32_t* dst = reinterpret_cast<uint32_t*>(x + w0 * kF);
        for (int e = lane; e < nodes * W; e += 32) dst[e] = s_x[warp][e / W][e % W];
        __syncwarp();
    }
    if constexpr (is_bf16<TA>()) {
        __syncthreads();                             // the words around the listed features are stored
        const int listed = s_listed < kList ? s_listed : kList;
        for (int q = threadIdx.x; q < listed; q += kThreadsG) {
            const int64_t e = s_list[q], i = e / (kF - kStruct);
            x[i * kF + kStruct + (e - i * (kF - kStruct))] = to_act<TA>(normal_slow(base, e));
        }
    }
}

// ------------------------------------------------------------------ aggregation
// Sum over the stored entries (i, j != i) of w_ij in_j (TRANS: w_ij inv_s_j in_j) by a
// group of G = F/4 lanes, four features a lane.  The group loads G entries at a time, one
// a lane (coalesced, one conversion of the double weight for each), and has their rows in
// flight together; the sum runs in the order of the entries.  All lanes of the warp call it.
template <typename TI, int F, bool TRANS>
__device__ __forceinline__ void gather_row(int64_t i, bool act, const int64_t* __restrict__ rp,
                                           const int32_t* __restrict__ ci, const double* __restrict__ cv,
                                           const float* __restrict__ inv_s, const TI* __restrict__ in, float (&acc)[4]) {
    constexpr int G = F / 4;
    const int lane = threadIdx.x & 31, lig = lane % G, base = lane - lig;
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = 0.f;
    const int64_t s1 = act ? __ldg(rp + i + 1) : 0;
    for (int64_t s = act ? __ldg(rp + i) : 0; __any_sync(0xffffffffu, s < s1); s += G) {
        int jo = -1;
        float wo = 0.f;
        if (s + lig < s1) {
            jo = __ldg(ci + s + lig);
            wo = (float)__ldg(cv + s + lig);
            if (jo == i) jo = -1;
            if (TRANS && jo >= 0) wo *= __ldg(inv_s + jo);
        }
        // four rows in flight a lane; the second half of a batch only where a row of the warp
        // reaches it
#pragma unroll
        for (int h = 0; h < G; h += 4) {
            if (h > 0 && !__any_sync(0xffffffffu, s + h < s1)) break;
            int j[4];
            float w[4];
            Unit<TI> x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                j[u] = __shfl_sync(0xffffffffu, jo, base + h + u);
                w[u] = __shfl_sync(0xffffffffu, wo, base + h + u);
                if (j[u] >= 0) x[u].load(in + (int64_t)j[u] * F + 4 * lig);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j[u] >= 0)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[c] = fmaf(w[u], x[u].v[c], acc[c]);
        }
    }
}

// ------------------------------------------------------------------ forward layer
// m = aggregate(in), h = relu(W_s in + W_n m + b) for a warp's tile of kFwdTile = 8 nodes; OUT:
// also o = W_o h + b_o, r_hat = o / ||o||.  m and h are stored only where the caller keeps them
// (the backward pass, the next layer); the tile's rows stay in shared memory between the
// three parts.  A thread owns 4 outputs of kFwdNodes = 2 nodes: per 4 inputs it reads 12 vectors
// of shared memory for 64 multiply-adds, and shared memory is what bounds it (66 to 71% busy; one
// weight and one activation for each multiply-add, with an 8-way bank conflict on the weights,
// took 1.45 ms a layer at n = 1e6 and the aggregation before it 0.18; now 0.23 together, 0.36
// with the output layer; 4 nodes a thread took 0.33 to 0.60 with fewer warps).
// Every sum keeps its order: input by input, W_n m before W_s h.
template <typename TA, int F, bool OUT>
__global__ void __launch_bounds__(kFwdThreads, kFwdBlocks)
k_layer(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci, const double* __restrict__ cv,
        const float* __restrict__ inv_s, const TA* __restrict__ in, const float* __restrict__ theta_l,
        TA* __restrict__ m_out, TA* __restrict__ h_out, const float* __restrict__ theta_o, int r_out,
        float* __restrict__ rhat, int rs, float* __restrict__ onrm, double* __restrict__ R, int ld) {
    constexpr int S = F + 4, SH = kH + 4;            // row strides: 16-byte rows, banks 4 apart
    static_assert(kFwdTile % (128 / F) == 0, "every lane takes part in each gather");
    __shared__ __align__(16) float Ws[F * kH], Wn[F * kH], b[kH];          // [input][output]
    __shared__ __align__(16) float s_h[kFwdThreads / 32][kFwdTile * SH], s_m[kFwdThreads / 32][kFwdTile * SH];
    __shared__ __align__(16) float Wo[OUT ? kH * kMaxOut : 4];
    __shared__ float bo[OUT ? kMaxOut : 1];
    // 16-byte stores of R where its rows allow them
    const bool vec = ld % 2 == 0 && (reinterpret_cast<uintptr_t>(R) & 15u) == 0;
    const int tid = threadIdx.x;
    for (int e = tid; e < kH * F; e += kFwdThreads) {
        const int o = e / F, k = e % F;
        Ws[k * kH + o] = weight<TA>(theta_l[e]);
        Wn[k * kH + o] = weight<TA>(theta_l[kH * F + e]);
    }
    if (tid < kH) b[tid] = weight<TA>(theta_l[2 * kH * F + tid]);
    if constexpr (OUT) {
        for (int e = tid; e < kH * kMaxOut; e += kFwdThreads) {
            const int c = e / kH, k = e % kH;
            Wo[k * kMaxOut + c] = c < r_out ? weight<TA>(theta_o[e]) : 0.f;
        }
        if (tid < kMaxOut) bo[tid] = tid < r_out ? weight<TA>(theta_o[r_out * kH + tid]) : 0.f;
    }
    __syncthreads();
    constexpr int G = F / 4;
    const int lane = tid & 31, warp = tid >> 5, lig = lane % G;
    const int sub = lane & 7, n0 = lane >> 3;        // outputs 4 sub.., nodes n0 + 4 a of the tile (no bank conflict)
    float *hs = s_h[warp], *ms = s_m[warp];
    const int64_t nwarps = (int64_t)gridDim.x * (kFwdThreads / 32);
    for (int64_t t = (int64_t)blockIdx.x * (kFwdThreads / 32) + warp; t * kFwdTile < n; t += nwarps) {
        const int64_t i0 = t * kFwdTile;
#pragma unroll 1
        for (int u = lane / G; u < kFwdTile; u += 32 / G) {
            const int64_t i = i0 + u;
            const bool act = i < n;
            float acc[4];
            gather_row<TA, F, false>(i, act, rp, ci, cv, inv_s, in, acc);
            Unit<TA> own, mo;
            const float sc = act ? __ldg(inv_s + i) : 0.f;
            if (act) own.load(in + i * F + 4 * lig);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                mo.v[c] = stored<TA>(acc[c] * sc);
                if (!act) own.v[c] = 0.f;
            }
            *reinterpret_cast<float4*>(hs + u * S + 4 * lig) = make_float4(own.v[0], own.v[1], own.v[2], own.v[3]);
            *reinterpret_cast<float4*>(ms + u * S + 4 * lig) = make_float4(mo.v[0], mo.v[1], mo.v[2], mo.v[3]);
            if (act && m_out != nullptr) mo.store(m_out + i * F + 4 * lig);
        }
        __syncwarp();
        float u[kFwdNodes][4];
#pragma unroll
        for (int a = 0; a < kFwdNodes; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) u[a][c] = b[4 * sub + c];
#pragma unroll 1
        for (int k0 = 0; k0 < F; k0 += 4) {
            float4 hv[kFwdNodes], mv[kFwdNodes];
#pragma unroll
            for (int a = 0; a < kFwdNodes; ++a) {
                hv[a] = *reinterpret_cast<const float4*>(hs + (n0 + 4 * a) * S + k0);
                mv[a] = *reinterpret_cast<const float4*>(ms + (n0 + 4 * a) * S + k0);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float4 ws = *reinterpret_cast<const float4*>(Ws + (k0 + k) * kH + 4 * sub);
                const float4 wn = *reinterpret_cast<const float4*>(Wn + (k0 + k) * kH + 4 * sub);
#pragma unroll
                for (int a = 0; a < kFwdNodes; ++a) {
                    const float h = k == 0 ? hv[a].x : k == 1 ? hv[a].y : k == 2 ? hv[a].z : hv[a].w;
                    const float m = k == 0 ? mv[a].x : k == 1 ? mv[a].y : k == 2 ? mv[a].z : mv[a].w;
                    u[a][0] = fmaf(ws.x, h, fmaf(wn.x, m, u[a][0]));
                    u[a][1] = fmaf(ws.y, h, fmaf(wn.y, m, u[a][1]));
                    u[a][2] = fmaf(ws.z, h, fmaf(wn.z, m, u[a][2]));
                    u[a][3] = fmaf(ws.w, h, fmaf(wn.w, m, u[a][3]));
                }
            }
        }
        Unit<TA> ho[kFwdNodes];
#pragma unroll
        for (int a = 0; a < kFwdNodes; ++a) {
#pragma unroll
            for (int c = 0; c < 4; ++c) ho[a].v[c] = stored<TA>(fmaxf(u[a][c], 0.0f));
            const int64_t i = i0 + n0 + 4 * a;
            if (i < n && h_out != nullptr) ho[a].store(h_out + i * kH + 4 * sub);
        }
        if constexpr (OUT) {
            __syncwarp();                            // hs has been read
#pragma unroll
            for (int a = 0; a < kFwdNodes; ++a)
                *reinterpret_cast<float4*>(hs + (n0 + 4 * a) * SH + 4 * sub) =
                    make_float4(ho[a].v[0], ho[a].v[1], ho[a].v[2], ho[a].v[3]);
            __syncwarp();
            float o[kFwdNodes][4];
#pragma unroll
            for (int a = 0; a < kFwdNodes; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c) o[a][c] = bo[4 * sub + c];
#pragma unroll 1
            for (int k0 = 0; k0 < kH; k0 += 4) {
                float4 hv[kFwdNodes];
#pragma unroll
                for (int a = 0; a < kFwdNodes; ++a) hv[a] = *reinterpret_cast<const float4*>(hs + (n0 + 4 * a) * SH + k0);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float4 wo = *reinterpret_cast<const float4*>(Wo + (k0 + k) * kMaxOut + 4 * sub);
#pragma unroll
                    for (int a = 0; a < kFwdNodes; ++a) {
                        const float h = k == 0 ? hv[a].x : k == 1 ? hv[a].y : k == 2 ? hv[a].z : hv[a].w;
                        o[a][0] = fmaf(wo.x, h, o[a][0]);
                        o[a][1] = fmaf(wo.y, h, o[a][1]);
                        o[a][2] = fmaf(wo.z, h, o[a][2]);
                        o[a][3] = fmaf(wo.w, h, o[a][3]);
                    }
                }
            }
            // ||o||^2 in the order of the outputs: the lanes of a node's group add their four in turn
            float nn[kFwdNodes];
#pragma unroll
            for (int a = 0; a < kFwdNodes; ++a) nn[a] = 0.f;
            for (int q = 0; 4 * q < r_out; ++q)
#pragma unroll
                for (int a = 0; a < kFwdNodes; ++a) {
                    float t = nn[a];
#pragma unroll
                    for (int c = 0; c < 4; ++c) t = fmaf(o[a][c], o[a][c], t);       // outputs past r_out are 0
                    nn[a] = __shfl_sync(0xffffffffu, t, (lane & 24) + q);
                }
#pragma unroll
            for (int a = 0; a < kFwdNodes; ++a) {
                const int64_t i = i0 + n0 + 4 * a;
                const float nrm = sqrtf(nn[a]);
                const float inv = nrm > 0.f ? 1.0f / nrm : 0.f;
                if (i >= n) continue;
                if (onrm != nullptr && sub == 0) onrm[i] = nrm;
                float v[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) v[c] = 4 * sub + c < r_out ? o[a][c] * inv : 0.f;
                if (rhat != nullptr && 4 * sub < rs)
                    *reinterpret_cast<float4*>(rhat + i * rs + 4 * sub) = make_float4(v[0], v[1], v[2], v[3]);
                if (R != nullptr) {
                    double* row = R + i * ld;
                    if (vec && 4 * sub + 3 < ld) {
                        *reinterpret_cast<double2*>(row + 4 * sub) = make_double2(widen(v[0]), widen(v[1]));
                        *reinterpret_cast<double2*>(row + 4 * sub + 2) = make_double2(widen(v[2]), widen(v[3]));
                    } else {
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            if (4 * sub + c < ld) row[4 * sub + c] = widen(v[c]);
                    }
                    for (int c = kMaxOut + sub; c < ld; c += 8) row[c] = 0.0;
                }
            }
        }
        __syncwarp();                                // the tile has been read
    }
}

// ------------------------------------------------------------------ loss
// Loss over edges i < j, its gradient in r_hat_i, (2 / |E|) sum_j (r_hat_i . r_hat_j - t_ij)
// r_hat_j, and from it the gradient before the normalisation, do = (dr - r_hat (r_hat .
// dr)) / ||o||.  Eight lanes a node, four components a lane (rows padded to rs); eight
// edges at a time, each lane ending with the dot of one (batch_sums).  A warp a node with a
// butterfly an edge took 27 us at n = 3e4, |E| = 6e4 (and 63 us more in the output layer's
// backward pass, which formed do with 32 of 256 threads); now 12 us.
__global__ void __launch_bounds__(kThreadsG)
k_loss(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci, const float* __restrict__ rhat,
       int rs, const float* __restrict__ onrm, const float* __restrict__ target, float two_over_ne,
       float* __restrict__ d_o, double* __restrict__ part) {
    const int lane = threadIdx.x & 31, lig = lane & 7, base = lane - lig;
    const int64_t g = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    const int64_t ng = ((int64_t)gridDim.x * blockDim.x) >> 3;
    const bool col = 4 * lig < rs;
    double loss = 0.0;
    for (int64_t w0 = g - (lane >> 3); w0 < n; w0 += ng) {        // the warp's four nodes
        const int64_t i = w0 + (lane >> 3);
        const bool act = i < n;
        Unit<float> ri;
        float gr[4] = {0.f, 0.f, 0.f, 0.f};
        if (act && col) ri.load(rhat + i * rs + 4 * lig);
        else ri.v[0] = ri.v[1] = ri.v[2] = ri.v[3] = 0.f;
        const int64_t s1 = act ? __ldg(rp + i + 1) : 0;
        for (int64_t s = act ? __ldg(rp + i) : 0; __any_sync(0xffffffffu, s < s1); s += 8) {
            int jo = -1;
            float t = 0.f;
            if (s + lig < s1) {
                jo = __ldg(ci + s + lig);
                t = __ldg(target + s + lig);
                if (jo == i) jo = -1;
            }
            Unit<float> rj[8];
            float d[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int j = __shfl_sync(0xffffffffu, jo, base + u);
                if (j >= 0 && col) rj[u].load(rhat + (int64_t)j * rs + 4 * lig);
                else rj[u].v[0] = rj[u].v[1] = rj[u].v[2] = rj[u].v[3] = 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u)
                d[u] = fmaf(ri.v[3], rj[u].v[3], fmaf(ri.v[2], rj[u].v[2], fmaf(ri.v[1], rj[u].v[1], ri.v[0] * rj[u].v[0])));
            batch_sums(d, 8, lig);
            const float diff = jo >= 0 ? d[0] - t : 0.f;
            if (jo > i) loss += (double)diff * diff;
            const float cf = two_over_ne * diff;
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const float c = __shfl_sync(0xffffffffu, cf, base + u);
#pragma unroll
                for (int e = 0; e < 4; ++e) gr[e] = fmaf(c, rj[u].v[e], gr[e]);
            }
        }
        float dt = fmaf(ri.v[3], gr[3], fmaf(ri.v[2], gr[2], fmaf(ri.v[1], gr[1], ri.v[0] * gr[0])));
        dt = group_sum(dt, 8);
        if (act && col) {
            const float nr = __ldg(onrm + i);
            const float inv = nr > 0.f ? 1.0f / nr : 0.f;
            Unit<float> dv;
#pragma unroll
            for (int e = 0; e < 4; ++e) dv.v[e] = (gr[e] - ri.v[e] * dt) * inv;
            dv.store(d_o + i * rs + 4 * lig);
        }
    }
    double acc[1] = {loss};
    block_partials<1>(acc, part);
}

// ------------------------------------------------------------------ backward layer
// Layer l for tiles of 32 nodes.  du = [h_out > 0] dh_out, where dh_out is W_o^T do for the
// last layer (OUT, with dW_o = sum do h^T and db_o = sum do) and dh_self + A^T dm of the
// layer above for the others; then W_s^T du and W_n^T du for the layer below (not LAST) and
// the block's partial sums of dW_s = sum du h_in^T, dW_n = sum du m^T, db = sum du.
// A thread owns 4 consecutive weights of each matrix and 4 inputs of one node: one scalar
// and two vectors of shared memory for 8 multiply-adds.
template <typename TA, int F, bool OUT>
__global__ void __launch_bounds__(kThreadsG, kBackBlocks)
k_back(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci, const double* __restrict__ cv,
       const float* __restrict__ inv_s, const TA* __restrict__ hin, const TA* __restrict__ min_,
       const TA* __restrict__ hout, const float* __restrict__ d_o, int rs, int r_out,
       const float* __restrict__ theta_o, const float* __restrict__ dh_self, const float* __restrict__ dm_up,
       const float* __restrict__ theta_l, float* __restrict__ dh_in, float* __restrict__ dm,
       float* __restrict__ gpart, int64_t pstride, int64_t poff, int64_t poff_o) {
    constexpr int S = F + 4, SH = kH + 4, V = F / 8;  // V weights of a row per thread
    __shared__ __align__(16) float Ws[kH * F], Wn[kH * F];                 // [output][input]
    __shared__ __align__(16) float Wo[OUT ? kMaxOut * kH : 4];
    __shared__ __align__(16) float s_du[kBackTile * SH], s_hin[kBackTile * S], s_min[kBackTile * S];
    __shared__ __align__(16) float s_do[OUT ? kBackTile * SH : 4], s_h[OUT ? kBackTile * SH : 4];
    const int tid = threadIdx.x, row = tid >> 3, sub = tid & 7;
    for (int e = tid; e < kH * F; e += kThreadsG) {
        Ws[e] = weight<TA>(theta_l[e]);
        Wn[e] = weight<TA>(theta_l[kH * F + e]);
    }
    if constexpr (OUT)
        for (int e = tid; e < kMaxOut * kH; e += kThreadsG) Wo[e] = e < r_out * kH ? weight<TA>(theta_o[e]) : 0.f;
    float gs[V], gn[V], gb = 0.f, go[4] = {0.f, 0.f, 0.f, 0.f}, gbo = 0.f;
#pragma unroll
    for (int c = 0; c < V; ++c) gs[c] = gn[c] = 0.f;
    const int64_t ntiles = (n + kBackTile - 1) / kBackTile;
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t i = t * kBackTile + row;       // the thread's node
        const bool act = i < n;
        __syncthreads();                             // weights are there; the last tile has been read
        float du[4] = {0.f, 0.f, 0.f, 0.f};
        Unit<TA> ho;
        if (act) ho.load(hout + i * kH + 4 * sub);
        else ho.v[0] = ho.v[1] = ho.v[2] = ho.v[3] = 0.f;
        if constexpr (OUT) {
            Unit<float> dv;
            if (act && 4 * sub < rs) dv.load(d_o + i * rs + 4 * sub);
            else dv.v[0] = dv.v[1] = dv.v[2] = dv.v[3] = 0.f;
            *reinterpret_cast<float4*>(s_do + row * SH + 4 * sub) = make_float4(dv.v[0], dv.v[1], dv.v[2], dv.v[3]);
            *reinterpret_cast<float4*>(s_h + row * SH + 4 * sub) = make_float4(ho.v[0], ho.v[1], ho.v[2], ho.v[3]);
        } else {
            gather_row<float, kH, true>(i, act, rp, ci, cv, inv_s, dm_up, du);
            if (act) {
                Unit<float> ds;
                ds.load(dh_self + i * kH + 4 * sub);
#pragma unroll
                for (int c = 0; c < 4; ++c) du[c] += ds.v[c];
            }
        }
        for (int e = tid; e < kBackTile * (F / 4); e += kThreadsG) {
            const int u = e / (F / 4), k = 4 * (e % (F / 4));
            const int64_t iu = t * kBackTile + u;
            Unit<TA> a, m;
            if (iu < n) {
                a.load(hin + iu * F + k);
                m.load(min_ + iu * F + k);
            } else {
#pragma unroll
                for (int c = 0; c < 4; ++c) a.v[c] = m.v[c] = 0.f;
            }
            *reinterpret_cast<float4*>(s_hin + u * S + k) = make_float4(a.v[0], a.v[1], a.v[2], a.v[3]);
            *reinterpret_cast<float4*>(s_min + u * S + k) = make_float4(m.v[0], m.v[1], m.v[2], m.v[3]);
        }
        if constexpr (OUT) {
            __syncthreads();
            for (int c = 0; c < r_out; ++c) {
                const float dc = s_do[row * SH + c];
                const float4 w = *reinterpret_cast<const float4*>(Wo + c * kH + 4 * sub);
                du[0] = fmaf(w.x, dc, du[0]);
                du[1] = fmaf(w.y, dc, du[1]);
                du[2] = fmaf(w.z, dc, du[2]);
                du[3] = fmaf(w.w, dc, du[3]);
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (!(ho.v[c] > 0.f)) du[c] = 0.f;
        *reinterpret_cast<float4*>(s_du + row * SH + 4 * sub) = make_float4(du[0], du[1], du[2], du[3]);
        __syncthreads();
        if (dh_in != nullptr) {                      // for the layer below: inputs V sub.. of the thread's node
            float a[V], m[V];
#pragma unroll
            for (int c = 0; c < V; ++c) a[c] = m[c] = 0.f;
#pragma unroll 8
            for (int o = 0; o < kH; ++o) {
                const float d = s_du[row * SH + o];
#pragma unroll
                for (int c = 0; c < V; ++c) {
                    a[c] = fmaf(Ws[o * F + V * sub + c], d, a[c]);
                    m[c] = fmaf(Wn[o * F + V * sub + c], d, m[c]);
                }
            }
            if (act) {
#pragma unroll
                for (int c = 0; c < V; ++c) {
                    dh_in[i * F + V * sub + c] = a[c];
                    dm[i * F + V * sub + c] = m[c];
                }
            }
        }
        // weight gradients: output `row`, inputs V sub.. of the tile's nodes
#pragma unroll 8
        for (int u = 0; u < kBackTile; ++u) {
            const float d = s_du[u * SH + row];
#pragma unroll
            for (int c = 0; c < V; ++c) {
                gs[c] = fmaf(d, s_hin[u * S + V * sub + c], gs[c]);
                gn[c] = fmaf(d, s_min[u * S + V * sub + c], gn[c]);
            }
            if (sub == 0) gb += d;
            if constexpr (OUT) {
                const float dc = s_do[u * SH + row];
                const float4 h = *reinterpret_cast<const float4*>(s_h + u * SH + 4 * sub);
                go[0] = fmaf(dc, h.x, go[0]);
                go[1] = fmaf(dc, h.y, go[1]);
                go[2] = fmaf(dc, h.z, go[2]);
                go[3] = fmaf(dc, h.w, go[3]);
                if (sub == 0) gbo += dc;
            }
        }
    }
    float* gp = gpart + blockIdx.x * pstride;
#pragma unroll
    for (int c = 0; c < V; ++c) {
        gp[poff + row * F + V * sub + c] = gs[c];
        gp[poff + kH * F + row * F + V * sub + c] = gn[c];
    }
    if (sub == 0) gp[poff + 2 * kH * F + row] = gb;
    if constexpr (OUT) {
        if (row < r_out) {
#pragma unroll
            for (int c = 0; c < 4; ++c) gp[poff_o + row * kH + 4 * sub + c] = go[c];
            if (sub == 0) gp[poff_o + r_out * kH + row] = gbo;
        }
    }
}

// ------------------------------------------------------------------ gradient and Adam
// grad[p] = sum over the blocks of gpart[b][p] (fixed order, double accumulation: sixteen
// threads take every sixteenth block), the caller's copy of it, and Adam (Kingma & Ba 2015)
// on the float master weights when lr > 0.  One thread a parameter over all blocks took
// 46 us (27 blocks, a serial chain of 304 loads); now 21 us for 469 blocks.
__global__ void __launch_bounds__(32 * kFoldSlices)
k_fold_adam(const float* __restrict__ gpart, int nb, int64_t P, float* __restrict__ grad, float* __restrict__ grad_out,
            float* __restrict__ theta, float* __restrict__ m1, float* __restrict__ m2, float lr, float b1, float b2,
            float eps, float c1, float c2) {
    __shared__ double s[kFoldSlices][32];
    const int x = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int64_t p = blockIdx.x * 32LL + x;
    double t = 0.0;
    if (p < P)
        for (int b = q; b < nb; b += 8 * kFoldSlices) {
            float v[8];                              // in flight together
#pragma unroll
            for (int k = 0; k < 8; ++k) v[k] = b + k * kFoldSlices < nb ? gpart[(int64_t)(b + k * kFoldSlices) * P + p] : 0.f;
#pragma unroll
            for (int k = 0; k < 8; ++k) t += widen(v[k]);
        }
    s[q][x] = t;
    __syncthreads();
    if (q != 0 || p >= P) return;
    for (int k = 1; k < kFoldSlices; ++k) t += s[k][x];
    const float g = (float)t;
    grad[p] = g;
    if (grad_out != nullptr) grad_out[p] = g;
    if (!(lr > 0.f)) return;
    const float a = b1 * m1[p] + (1.f - b1) * g;
    const float b = b2 * m2[p] + (1.f - b2) * g * g;
    m1[p] = a;
    m2[p] = b;
    theta[p] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
}

// X*_ij = r_i . r_j on every stored entry of C (0 on the diagonal)
__global__ void k_targets(int64_t n, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                          const double* __restrict__ R, int r, int ld, float* __restrict__ t) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        for (int64_t e = rp[i]; e < rp[i + 1]; ++e) {
            const int j = ci[e];
            double d = 0.0;
            if (j != i)
                for (int c = 0; c < r; ++c) d += R[i * ld + c] * R[(int64_t)j * ld + c];
            t[e] = (float)d;
        }
    }
}

}  // namespace gnn
}  // namespace lorads
