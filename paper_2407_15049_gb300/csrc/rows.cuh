// Problem arrays and row helpers shared by the streaming kernels: gating, arithmetic
// types of the storage types, the warp-uniform row loop, vector loads and stores of rows.
#pragma once

#include <type_traits>
#include "common.cuh"

namespace lorads {

// ------------------------------------------------------------------ problem arrays
struct ProbDev {
    int64_t n, m;
    // C: full symmetric CSR
    const int64_t* c_rowptr;
    const int32_t* c_col;
    const double* c_val;
    const float* c_val32;
    const dfloat* c_valdf;
    // diagonal constraints by row: constraint index (-1: none) and coefficient
    const int32_t* dk;
    const double* da;
    const float* da32;          // float and double-float mirrors of da and b for the
    const dfloat* da_df;        // FP32-unit paths (no per-row FP64 there)
    const dfloat* b_df;
    // off-diagonal constraints as a symmetric pattern: slot -> (column, constraint, coef)
    const int64_t* a_rowptr;
    const int32_t* a_col;
    const int32_t* a_k;
    const double* a_a;
    // constraint list, fused diagonal constraints first: triplets (row <= col, coef) in
    // list order and the constraint of each list position.  k_ptr (general form,
    // constraints with several triplets): position q owns triplets k_ptr[q]..k_ptr[q+1]-1;
    // null: position q is triplet q.
    const int32_t* k_row;
    const int32_t* k_col;
    const double* k_a;
    const int32_t* k_id;
    const int64_t* k_ptr;
    int64_t m_diag, m_off;
    const double* b;
    // double-float mirrors of the constraint coefficients (list order and pattern
    // order) for the FP32-unit paths; may be null for FP64 callers
    const dfloat* k_adf;
    const dfloat* a_adf;
};

// ------------------------------------------------------------------ gating
// Kernels of the captured iteration graph check the control block first and
// return at once when the current phase does not need them.
enum { PH_ALWAYS = 0, PH_INNER = 1, PH_STEP = 2, PH_OUTER = 3 };

__device__ __forceinline__ bool gated_off(const Ctrl* g, int ph) {
    if (g == nullptr || ph == PH_ALWAYS) return false;
    if (g->solve_done | g->pause) return true;
    if (ph == PH_OUTER) return g->phase != PHASE_OUTER;
    if (g->phase != PHASE_INNER) return true;
    if (ph == PH_STEP) return g->step_ok == 0;
    return false;
}

template <typename T>
using arith_t = typename Arith<T>::type;
template <typename T>
using A_of_t = arith_t<T>;

// precision rank of an arithmetic type: float < double-float < double
template <typename T> struct PrecRank;
template <> struct PrecRank<float> { static constexpr int v = 0; };
template <> struct PrecRank<dfloat> { static constexpr int v = 1; };
template <> struct PrecRank<double> { static constexpr int v = 2; };

template <int R> struct RankType;
template <> struct RankType<0> { using type = float; };
template <> struct RankType<1> { using type = dfloat; };
template <> struct RankType<2> { using type = double; };

// wider of the arithmetic types of two storage types
template <typename A, typename B>
using wide_t = typename RankType<(PrecRank<arith_t<A>>::v > PrecRank<arith_t<B>>::v ? PrecRank<arith_t<A>>::v
                                                                                   : PrecRank<arith_t<B>>::v)>::type;

// partial-sum type: double on the all-FP64 path, double-float otherwise (no FP64 pipe)
template <typename A, typename B>
using part_t = std::conditional_t<std::is_same_v<arith_t<A>, double> && std::is_same_v<arith_t<B>, double>,
                                  double, dfloat>;

// value type of C entries multiplied against rows of type TX
template <typename TX>
using cval_t = arith_t<TX>;

template <typename TV> __device__ __forceinline__ const TV* cvals(const ProbDev& p);
template <> __device__ __forceinline__ const double* cvals<double>(const ProbDev& p) { return p.c_val; }
template <> __device__ __forceinline__ const float* cvals<float>(const ProbDev& p) { return p.c_val32; }
template <> __device__ __forceinline__ const dfloat* cvals<dfloat>(const ProbDev& p) { return p.c_valdf; }

// per-row scalar type of the row-update math: double on the FP64 path,
// otherwise the arithmetic type of R (double-float or float)
template <typename TR, typename TD>
using rowscalar_t = std::conditional_t<std::is_same_v<arith_t<TR>, double> && std::is_same_v<arith_t<TD>, double>,
                                       double, arith_t<TR>>;

template <typename S> __device__ __forceinline__ S ld_scalar(const double* d, const dfloat* df, int64_t k);
template <> __device__ __forceinline__ double ld_scalar<double>(const double* d, const dfloat*, int64_t k) {
    return __ldg(d + k);
}
template <> __device__ __forceinline__ dfloat ld_scalar<dfloat>(const double*, const dfloat* df, int64_t k) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(df + k));
    return dfloat(v.x, v.y);
}
template <> __device__ __forceinline__ float ld_scalar<float>(const double*, const dfloat* df, int64_t k) {
    return __ldg(reinterpret_cast<const float*>(df + k));     // hi part
}

// The multipliers y and y~ (double, or double-float): written during a solve, so loaded without
// the read-only path (the persistent kernels read them after other blocks wrote them).
template <typename S> __device__ __forceinline__ S ld_multiplier(const double* y, const dfloat* ydf, int64_t k) {
    if constexpr (std::is_same_v<S, double>) {
        return y[k];
    } else {
        if (ydf == nullptr) return S(y[k]);
        if constexpr (std::is_same_v<S, dfloat>) {
            const float2 v = *reinterpret_cast<const float2*>(ydf + k);
            return dfloat(v.x, v.y);
        } else {
            return ydf[k].hi;
        }
    }
}

// type of the per-row z cache (and of the line-search row terms): double on the
// FP64 path, otherwise the arithmetic type of the direction D
template <typename TD, typename TR>
using zrow_t = std::conditional_t<std::is_same_v<part_t<TD, TR>, double>, double, arith_t<TD>>;

// read-only scalar loads
__device__ __forceinline__ double ldv(const double* p) { return __ldg(p); }
__device__ __forceinline__ float ldv(const float* p) { return __ldg(p); }
__device__ __forceinline__ dfloat ldv(const dfloat* p) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(p));
    return dfloat(v.x, v.y);
}

// Warp-uniform row loop: each warp owns 32/L consecutive rows per trip, so the
// group shuffles below always see the full warp.  Packed groups (`dense`): L may
// be any width up to 32 (one unit per lane, L = units per row); the warp holds
// floor(32/L) rows and its last 32 mod L lanes take no row (`live` false), e.g.
// ld = 24: 5 rows of 6 lanes instead of 4 rows of 8 lanes with 2 idle each.
struct RowLoop {
    int L, lig, gw, rows_per_warp, base_lane;
    bool live;
    int64_t first, stride;
    __device__ __forceinline__ RowLoop(int L_, VGrid vg, bool dense = false) : L(L_) {
        const int lane = threadIdx.x & 31;
        if (dense) {
            gw = lane / L;
            lig = lane - gw * L;
            rows_per_warp = 32 / L;
            live = gw < rows_per_warp;
        } else {
            lig = threadIdx.x & (L - 1);
            gw = lane / L;
            rows_per_warp = 32 / L;
            live = true;
        }
        base_lane = live ? gw * L : 0;
        const int64_t warp = (vg.bid * (int64_t)blockDim.x + threadIdx.x) >> 5;
        const int64_t nwarps = ((int64_t)vg.nblk * blockDim.x) >> 5;
        first = warp * rows_per_warp;
        stride = nwarps * rows_per_warp;
    }
};

// Sum over the L lanes of a packed group, taken in lane order by every lane (the
// same bits in each lane of the group); all 32 lanes take part in the shuffles.
__device__ __forceinline__ float shfl_idx(float v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ double shfl_idx(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ dfloat shfl_idx(dfloat v, int src) {
    return dfloat(__shfl_sync(0xffffffffu, v.hi, src), __shfl_sync(0xffffffffu, v.lo, src));
}
template <typename V>
__device__ __forceinline__ V group_sum_packed(V v, int L, int base_lane) {
    V t = shfl_idx(v, base_lane);
    for (int k = 1; k < L; ++k) t += shfl_idx(v, base_lane + k);
    return t;
}

// Row helpers: lane `lig` of a group of L handles units c*L + lig < Q.
// Units past Q are zero on load and skipped on store.
template <typename T, int CPL>
__device__ __forceinline__ void load_row(Unit<T> (&u)[CPL], const T* base, int64_t row, int ld, int L, int Q, int lig) {
    const T* p = base + row * (int64_t)ld + lig * 4;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        if (c * L + lig < Q) u[c].load(p + c * L * 4);
        else
#pragma unroll
            for (int e = 0; e < 4; ++e) u[c].v[e] = 0;
    }
}

template <typename T, int CPL>
__device__ __forceinline__ void load_row_stream(Unit<T> (&u)[CPL], const T* base, int64_t row, int ld, int L, int Q,
                                                int lig) {
    const T* p = base + row * (int64_t)ld + lig * 4;
#pragma unroll
    for (int c = 0; c < CPL; ++c) {
        if (c * L + lig < Q) u[c].load_stream(p + c * L * 4);
        else
#pragma unroll
            for (int e = 0; e < 4; ++e) u[c].v[e] = 0;
    }
}

// Epilogues of the SpMM over C (see k_spmm_c_body).
enum { EPI_NONE = 0, EPI_LS = 1, EPI_OBJ = 2 };

// L2 prefetch (no register, no wait) of one address of global memory.
__device__ __forceinline__ void prefetch_l2(const void* a) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(a));
}

// L2 prefetch of the units of `row` that lane `lig` loads: issued one row
// iteration ahead, it turns the dependent loads of that iteration into L2 hits.
template <typename T, int CPL>
__device__ __forceinline__ void prefetch_row(const T* base, int64_t row, int ld, int L, int Q, int lig) {
    const T* p = base + row * (int64_t)ld + lig * 4;
#pragma unroll
    for (int c = 0; c < CPL; ++c)
        if (c * L + lig < Q) prefetch_l2(p + c * L * 4);
}

template <typename T, int CPL>
__device__ __forceinline__ void store_row(const Unit<T> (&u)[CPL], T* base, int64_t row, int ld, int L, int Q, int lig) {
    T* p = base + row * (int64_t)ld + lig * 4;
#pragma unroll
    for (int c = 0; c < CPL; ++c)
        if (c * L + lig < Q) u[c].store_stream(p + c * L * 4);
}

template <typename A, typename T1, typename T2, int CPL>
__device__ __forceinline__ A dot_units(const Unit<T1> (&x)[CPL], const Unit<T2> (&y)[CPL]) {
    A s = A(0);
#pragma unroll
    for (int c = 0; c < CPL; ++c)
#pragma unroll
        for (int e = 0; e < 4; ++e) s = fma(A(x[c].v[e]), A(y[c].v[e]), s);
    return s;
}

// Value an element has once stored as T (bf16 rounds; every other type keeps it).
template <typename T, typename A>
__device__ __forceinline__ A as_stored(A v) {
    if constexpr (std::is_same_v<T, __nv_bfloat16>) return A(__bfloat162float(__float2bfloat16_rn(float(v))));
    else return v;
}

}  // namespace lorads
