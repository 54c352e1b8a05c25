// The constraint pass: dots of gathered row pairs, one for each constraint of the
// ordered list, and the scalars of the method that follow from them.
#pragma once

#include "rows.cuh"

namespace lorads {

// ================================================================== constraint pass
// One group of L lanes per constraint t in [k0, k1) of the ordered list
// (diagonal constraints first).  With f = 1 (i == j) or 2 (i < j):
//   CONS_EVAL: out[k] = a (u_i.v_j + [i!=j] u_j.v_i)                  = <A_k, U V^T>
//   CONS_LS  : z = f a r_i.r_j - b, y~ = y - rho z, q1 = f a (r_i.d_j + d_i.r_j),
//              q2 = f a d_i.d_j; partials of y~q1, y~q2, q1^2, q1q2, q2^2
//   CONS_YTIL: out[k] = y~ ;  partial |z|^2
//   CONS_YUPD: y[k] <- y~ (and its double-float mirror);  partials |z|^2, b^T y_new
//   CONS_ZZ  : partial |z|^2
enum { CONS_EVAL = 0, CONS_LS = 1, CONS_YTIL = 2, CONS_YUPD = 3, CONS_ZZ = 4 };

// General form of the constraint pass: list position q is one constraint whose
// triplets t (i <= j, a) are summed with the weights of the triplet convention:
//   <A_k, U V^T> = sum_t a (u_i.v_j + [i != j] u_j.v_i),
// and, with f = 1 (i == j) or 2, z = sum_t f a r_i.r_j - b_k, q1 = sum_t f a
// (r_i.d_j + d_i.r_j) / (1 + [i == j]) ... written per triplet as in the single-triplet
// path, then the same per-constraint formulas.  Each lane accumulates its share of
// every triplet's dots; the group sum follows the triplet loop (no shuffle inside
// the loop, whose trip count differs between the groups of a warp).
template <typename TU, typename TV, int CPL, int MODE>
__device__ __forceinline__ void
k_cons_general(ProbDev p, int64_t k0, int64_t k1, const TU* __restrict__ U, const TV* __restrict__ V, int ld, int L,
               int Q, double* y, void* __restrict__ out, void* zk, dfloat* ydf, const Ctrl* ctrl, double rho_arg,
               double* __restrict__ part, VGrid vg) {
    constexpr int NQ = MODE == CONS_LS ? PL_N : PC_N;
    using PA = part_t<TU, TV>;
    PA accq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accq[q] = PA(0);
    const double rho = ctrl ? ctrl->rho : rho_arg;
    const bool same = (const void*)U == (const void*)V;
    using AU = wide_t<TU, TU>;
    using AW = wide_t<TU, TV>;
    using AV = wide_t<TV, TV>;
    using CS = std::conditional_t<std::is_same_v<PA, double>, double, dfloat>;
    const CS rho_c = CS(rho);
    CS* zkc = static_cast<CS*>(zk);
    RowLoop rl(L, vg);
    const int64_t cnt = k1 - k0;
    for (int64_t base = rl.first; base < cnt; base += rl.stride) {
        const int64_t q = k0 + base + rl.gw;
        const bool act = q < k1;
        // per-lane weighted dots: z part (f a u_i.u_j), q1 part, q2 part / EVAL value
        AU s_z = AU(0);
        AW s_1 = AW(0);
        AV s_2 = AV(0);
        if (act) {
            const int64_t t0 = __ldg(p.k_ptr + q), t1 = __ldg(p.k_ptr + q + 1);
            for (int64_t t = t0; t < t1; ++t) {
                const int i = __ldg(p.k_row + t), j = __ldg(p.k_col + t);
                const bool dg = i == j;
                const double a = __ldg(p.k_a + t);
                const double fa = dg ? a : 2.0 * a;
                Unit<TU> ui[CPL], uj[CPL];
                load_row<TU, CPL>(ui, U, i, ld, L, Q, rl.lig);
                if (!dg) load_row<TU, CPL>(uj, U, j, ld, L, Q, rl.lig);
                if constexpr (MODE == CONS_EVAL) {
                    if (same) {
                        s_z = s_z + AU(fa) * (dg ? dot_units<AU>(ui, ui) : dot_units<AU>(ui, uj));
                    } else {
                        Unit<TV> vi[CPL], vj[CPL];
                        load_row<TV, CPL>(vi, V, i, ld, L, Q, rl.lig);
                        if (dg) {
                            s_1 = s_1 + AW(a) * dot_units<AW>(ui, vi);
                        } else {
                            load_row<TV, CPL>(vj, V, j, ld, L, Q, rl.lig);
                            s_1 = s_1 + AW(a) * (dot_units<AW>(ui, vj) + dot_units<AW>(uj, vi));
                        }
                    }
                } else {
                    if (MODE != CONS_LS || zk == nullptr)
                        s_z = s_z + AU(fa) * (dg ? dot_units<AU>(ui, ui) : dot_units<AU>(ui, uj));
                    if constexpr (MODE == CONS_LS) {
                        Unit<TV> vi[CPL], vj[CPL];
                        load_row<TV, CPL>(vi, V, i, ld, L, Q, rl.lig);
                        if (dg) {
                            const AW d = dot_units<AW>(ui, vi);
                            s_1 = s_1 + AW(fa) * (d + d);
                            s_2 = s_2 + AV(fa) * dot_units<AV>(vi, vi);
                        } else {
                            load_row<TV, CPL>(vj, V, j, ld, L, Q, rl.lig);
                            s_1 = s_1 + AW(fa) * (dot_units<AW>(ui, vj) + dot_units<AW>(vi, uj));
                            s_2 = s_2 + AV(fa) * dot_units<AV>(vi, vj);
                        }
                    }
                }
            }
        }
        s_z = group_sum(s_z, L);
        s_1 = group_sum(s_1, L);
        s_2 = group_sum(s_2, L);
        if (act && rl.lig == 0) {
            const int k = __ldg(p.k_id + q);
            if constexpr (MODE == CONS_EVAL) {
                static_cast<double*>(out)[k] = same ? double(s_z) : double(s_1);
            } else {
                CS yk = CS(0.0), bk;
                if constexpr (MODE != CONS_ZZ) {
                    yk = ld_multiplier<CS>(y, ydf, k);
                }
                if constexpr (std::is_same_v<CS, double>) bk = __ldg(p.b + k);
                else bk = p.b_df ? ld_scalar<CS>(p.b, p.b_df, k) : CS(__ldg(p.b + k));
                const CS z = (MODE == CONS_LS && zk != nullptr) ? zkc[k] : CS(s_z) - bk;
                if constexpr (MODE == CONS_LS) {
                    const CS yt = yk - rho_c * z;
                    const CS q1 = CS(s_1);
                    const CS q2 = CS(s_2);
                    accq[PL_YQ1] += PA(yt * q1);
                    accq[PL_YQ2] += PA(yt * q2);
                    accq[PL_Q1Q1] += PA(q1 * q1);
                    accq[PL_Q1Q2] += PA(q1 * q2);
                    accq[PL_Q2Q2] += PA(q2 * q2);
                } else {
                    accq[PC_ZZ] += PA(z * z);
                    if constexpr (MODE == CONS_YTIL) {
                        static_cast<CS*>(out)[k] = yk - rho_c * z;
                        if (zk != nullptr) zkc[k] = z;
                    } else if constexpr (MODE == CONS_YUPD) {
                        const CS yn = yk - rho_c * z;
                        y[k] = double(yn);
                        if constexpr (std::is_same_v<CS, dfloat>) {
                            if (ydf != nullptr) ydf[k] = yn;
                        } else {
                            if (ydf != nullptr) ydf[k] = dfloat(yn);
                        }
                        accq[PC_BY] += PA(bk * yn);
                    }
                }
            }
        }
    }
    if constexpr (MODE != CONS_EVAL) block_partials<NQ>(accq, part, vg.pslot);
}

// Rows of more than 128 elements (several units per lane), and small maps: one constraint at a time.
template <typename TU, typename TV, int CPL, int MODE>
__device__ __forceinline__ void
k_cons_wide(ProbDev p, int64_t k0, int64_t k1, const TU* __restrict__ U, const TV* __restrict__ V, int ld, int L, int Q,
       double* y, void* __restrict__ out, void* zk, dfloat* ydf, const Ctrl* ctrl, double rho_arg,
       double* __restrict__ part, VGrid vg) {
    constexpr int NQ = MODE == CONS_LS ? PL_N : PC_N;
    using PA = part_t<TU, TV>;
    PA accq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accq[q] = PA(0);
    const double rho = ctrl ? ctrl->rho : rho_arg;
    const bool same = (const void*)U == (const void*)V;
    using AU = wide_t<TU, TU>;
    using AW = wide_t<TU, TV>;
    using AV = wide_t<TV, TV>;
    // per-constraint scalars: double on the all-FP64 path, double-float otherwise
    // (GB300's FP64 rate is ~1/64 of FP32; conversions run on the FP64 pipe too).
    // z = A(RR^T)_k - b_k, y~ and the cached z use the same type (zk, out: CS arrays).
    using CS = std::conditional_t<std::is_same_v<PA, double>, double, dfloat>;
    const CS rho_c = CS(rho);
    CS* zkc = static_cast<CS*>(zk);
    // what each mode gathers besides u_i, u_j
    constexpr bool NEED_V = MODE == CONS_EVAL || MODE == CONS_LS;
    RowLoop rl(L, vg);
    const int64_t cnt = k1 - k0;
    for (int64_t base = rl.first; base < cnt; base += rl.stride) {
        const int64_t t = k0 + base + rl.gw;
        const bool act = t < k1;
        const int i = act ? __ldg(p.k_row + t) : 0, j = act ? __ldg(p.k_col + t) : 0;
        const int k = act ? __ldg(p.k_id + t) : 0;
        const bool diag = i == j;
        CS ak = CS(0.0), yk = CS(0.0), zb = CS(0.0);     // coefficient, y_k, and z_k (cached) or b_k
        Unit<TU> ui[CPL], uj[CPL];
        Unit<TV> vi[CPL], vj[CPL];
        if (act) {
            if constexpr (MODE == CONS_EVAL || std::is_same_v<CS, double>) ak = CS(__ldg(p.k_a + t));
            else ak = p.k_adf ? ld_scalar<CS>(p.k_a, p.k_adf, t) : CS(__ldg(p.k_a + t));
            if constexpr (MODE != CONS_EVAL) {
                if constexpr (MODE != CONS_ZZ) yk = ld_multiplier<CS>(y, ydf, k);
                if (MODE == CONS_LS && zk != nullptr) zb = zkc[k];
                else if constexpr (std::is_same_v<CS, double>) zb = __ldg(p.b + k);
                else zb = p.b_df ? ld_scalar<CS>(p.b, p.b_df, k) : CS(__ldg(p.b + k));
            }
            load_row<TU, CPL>(ui, U, i, ld, L, Q, rl.lig);
            if (!diag) load_row<TU, CPL>(uj, U, j, ld, L, Q, rl.lig);
            if constexpr (NEED_V) {
                if (!(MODE == CONS_EVAL && same)) {
                    load_row<TV, CPL>(vi, V, i, ld, L, Q, rl.lig);
                    if (!diag) load_row<TV, CPL>(vj, V, j, ld, L, Q, rl.lig);
                }
            }
        }
        // dots of the gathered rows; partial per lane, then group sums
        AU s_uu = AU(0);                  // u_i.u_j (EVAL with U==V, and R-only modes)
        AW s_uv = AW(0), s_vu = AW(0);    // u_i.v_j, u_j.v_i
        AV s_vv = AV(0);                  // v_i.v_j
        if (act) {
            if constexpr (MODE == CONS_EVAL) {
                if (same) {
                    s_uu = diag ? dot_units<AU>(ui, ui) : dot_units<AU>(ui, uj);
                } else if (diag) {
                    s_uv = dot_units<AW>(ui, vi);
                } else {
                    s_uv = dot_units<AW>(ui, vj);
                    s_vu = dot_units<AW>(uj, vi);
                }
            } else {
                if (MODE != CONS_LS || zk == nullptr) s_uu = diag ? dot_units<AU>(ui, ui) : dot_units<AU>(ui, uj);
                if constexpr (MODE == CONS_LS) {
                    if (diag) {
                        s_uv = dot_units<AW>(ui, vi);
                        s_vu = s_uv;
                        s_vv = dot_units<AV>(vi, vi);
                    } else {
                        s_uv = dot_units<AW>(ui, vj);
                        s_vu = dot_units<AW>(vi, uj);
                        s_vv = dot_units<AV>(vi, vj);
                    }
                }
            }
        }
        s_uu = group_sum(s_uu, L);
        if constexpr (NEED_V) {
            s_uv = group_sum(s_uv, L);
            s_vu = group_sum(s_vu, L);
            s_vv = group_sum(s_vv, L);
        }
        if (!act || rl.lig != 0) continue;
        if constexpr (MODE == CONS_EVAL) {
            const double a = double(ak);
            const double f = diag ? 1.0 : 2.0;
            double val;
            if (same) val = f * a * double(s_uu);
            else if (diag) val = a * double(s_uv);
            else val = a * (double(s_uv) + double(s_vu));
            static_cast<double*>(out)[k] = val;
        } else {
            const CS fa = diag ? ak : CS(2.0f) * ak;
            const CS z = (MODE == CONS_LS && zk != nullptr) ? zb : fa * CS(s_uu) - zb;
            if constexpr (MODE == CONS_LS) {
                const CS yt = yk - rho_c * z;
                const CS q1 = fa * (CS(s_uv) + CS(s_vu));
                const CS q2 = fa * CS(s_vv);
                accq[PL_YQ1] += PA(yt * q1);
                accq[PL_YQ2] += PA(yt * q2);
                accq[PL_Q1Q1] += PA(q1 * q1);
                accq[PL_Q1Q2] += PA(q1 * q2);
                accq[PL_Q2Q2] += PA(q2 * q2);
            } else {
                accq[PC_ZZ] += PA(z * z);
                if constexpr (MODE == CONS_YTIL) {
                    static_cast<CS*>(out)[k] = yk - rho_c * z;
                    if (zk != nullptr) zkc[k] = z;
                } else if constexpr (MODE == CONS_YUPD) {
                    const CS yn = yk - rho_c * z;
                    y[k] = double(yn);
                    if constexpr (std::is_same_v<CS, dfloat>) {
                        if (ydf != nullptr) ydf[k] = yn;
                    } else {
                        if (ydf != nullptr) ydf[k] = dfloat(yn);
                    }
                    // b_k: zb holds it (z is recomputed in this mode)
                    accq[PC_BY] += PA(zb * yn);
                }
            }
        }
    }
    if constexpr (MODE != CONS_EVAL) block_partials<NQ>(accq, part, vg.pslot);
}

// Per-lane partial dot of gathered rows, by the arithmetic type's own multiply-add; a double-float
// row with a float row by the product of a double word and a float, which drops the terms of the
// zero low parts.
template <typename T1, typename T2>
constexpr bool df_by_float() {
    return std::is_same_v<arith_t<T1>, dfloat> && std::is_same_v<arith_t<T2>, float>;
}
template <typename A, typename T1, typename T2>
__device__ __forceinline__ A dot_lane(const Unit<T1>& x, const Unit<T2>& y) {
    A s = A(0);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        if constexpr (df_by_float<T1, T2>()) s = mul_fp(x.v[e], y.v[e]) + s;
        else if constexpr (df_by_float<T2, T1>()) s = mul_fp(y.v[e], x.v[e]) + s;
        else s = fma(A(x.v[e]), A(y.v[e]), s);
    }
    return s;
}

// Sums of up to kConsBatch values over the L lanes of a group at once: v[u] of every
// lane is a part of value u; afterwards v[0] of lane l (l < min(L, kConsBatch)) is the
// whole of value l.  Each step halves the values a lane carries (4 + 2 + 1 exchanges
// for 8 values where a butterfly for each takes 24); the additions are those of
// group_sum, in its order.
constexpr int kConsBatch = 8;
template <typename V>
__device__ __forceinline__ void batch_sums(V (&v)[kConsBatch], int L, int lig) {
    if (L >= 32)
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] += shfl_xor(v[u], 16);
    if (L >= 16)
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] += shfl_xor(v[u], 8);
    if (L >= 8) {
        const bool up = (lig & 4) != 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const V send = up ? v[u] : v[u + 4];
            const V keep = up ? v[u + 4] : v[u];
            v[u] = keep + shfl_xor(send, 4);
        }
    }
    if (L >= 4) {
        const bool up = (lig & 2) != 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const V send = up ? v[u] : v[u + 2];
            const V keep = up ? v[u + 2] : v[u];
            v[u] = keep + shfl_xor(send, 2);
        }
    }
    if (L >= 2) {
        const bool up = (lig & 1) != 0;
        const V send = up ? v[0] : v[1];
        const V keep = up ? v[1] : v[0];
        v[0] = keep + shfl_xor(send, 1);
    }
}

// Constraints in flight per group: their rows are loaded before any of their dots.
template <typename TU, typename TV, int MODE>
constexpr int cons_in_flight() {
    constexpr bool both = MODE == CONS_EVAL || MODE == CONS_LS;
    if (std::is_same_v<arith_t<TU>, double>) return both ? 1 : 2;
    return std::is_same_v<arith_t<TU>, float> ? 4 : (both ? 2 : 4);
}

// Rows of one unit per lane (up to 128 elements).  A group takes B = min(L, 8)
// consecutive constraints: lane u of the group owns constraint u, loads its indices,
// coefficient, multiplier and right-hand side (coalesced over the warp) and, once the
// group has formed the B dots and summed them together (batch_sums), does its scalar
// arithmetic.  One constraint at a time the scalar part (FP64 on the FP64 path and in
// CONS_EVAL, double-float otherwise) ran with one lane of the group at work and cost as
// much as the dots, and each dot took its own butterfly: the pass was bound by
// instruction issue, not by its gathers, which come from L2.  Measured: line search in the
// mixed form, 9.9e5 constraints, r = 20: 304 -> 88 us; y~: 207 -> 63 us; the map in FP32,
// 2.7e6 constraints, r = 17: 448 -> 94 us.
// ZC: z comes from the cache (CONS_LS).
template <typename TU, typename TV, int MODE, bool ZC>
__device__ __forceinline__ void
k_cons_batch(ProbDev p, int64_t k0, int64_t k1, const TU* __restrict__ U, const TV* __restrict__ V, int ld, int L,
             int Q, double* y, void* __restrict__ out, void* zk, dfloat* ydf, double rho,
             double* __restrict__ part, VGrid vg) {
    constexpr int NQ = MODE == CONS_LS ? PL_N : PC_N;
    using PA = part_t<TU, TV>;
    PA accq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accq[q] = PA(0);
    const bool same = (const void*)U == (const void*)V;
    using AU = wide_t<TU, TU>;
    using AW = wide_t<TU, TV>;
    using AV = wide_t<TV, TV>;
    // per-constraint scalars: double on the all-FP64 path, double-float otherwise
    // (GB300's FP64 rate is ~1/64 of FP32; conversions run on the FP64 pipe too).
    // z = A(RR^T)_k - b_k, y~ and the cached z use the same type (zk, out: CS arrays).
    using CS = std::conditional_t<std::is_same_v<PA, double>, double, dfloat>;
    const CS rho_c = CS(rho);
    CS* zkc = static_cast<CS*>(zk);
    constexpr bool NEED_Z = MODE != CONS_EVAL && !(MODE == CONS_LS && ZC);
    constexpr int UC = cons_in_flight<TU, TV, MODE>();
    const int B = L < kConsBatch ? L : kConsBatch;
    RowLoop rl(L, vg);
    const int64_t cnt = k1 - k0;
    // The lane's own constraint.  In the map its indices are loaded one batch ahead: the rows wait
    // on them and nothing else is in flight meanwhile (2.7e6 constraints, r = 17, float: 109 -> 94
    // us a call).  The other modes load a multiplier and z beside them, and took as long or up to
    // 6% longer with the registers that it takes; in FP64 the dots' arithmetic bounds the map.
    constexpr bool kAhead = MODE == CONS_EVAL && !std::is_same_v<arith_t<TU>, double>;
    const int64_t step = rl.stride * B;
    auto indices = [&](int64_t q, int& i, int& j, int& k) {
        i = -1;
        if (rl.lig < B && q < k1) {
            i = __ldg(p.k_row + q);
            j = __ldg(p.k_col + q);
            k = __ldg(p.k_id + q);
        }
    };
    int ii_nx = -1, jj_nx = -1, kid_nx = 0;
    if constexpr (kAhead) indices(k0 + rl.first * B + rl.gw * B + rl.lig, ii_nx, jj_nx, kid_nx);
    for (int64_t base = rl.first * B; base < cnt; base += step) {
        const int64_t t = k0 + base + rl.gw * B + rl.lig;
        int ii, jj = 0, kid = 0;
        const bool own = rl.lig < B && t < k1;
        if constexpr (kAhead) {
            ii = ii_nx;
            jj = jj_nx;
            kid = kid_nx;
            indices(t + step, ii_nx, jj_nx, kid_nx);
        } else {
            indices(t, ii, jj, kid);
        }
        CS ak = CS(0.0), yk = CS(0.0), zb = CS(0.0);      // coefficient, y_k, and z_k (cached) or b_k
        if (own) {
            if constexpr (std::is_same_v<CS, double>) {
                ak = __ldg(p.k_a + t);
            } else if constexpr (MODE != CONS_EVAL) {
                ak = p.k_adf ? ld_scalar<CS>(p.k_a, p.k_adf, t) : CS(__ldg(p.k_a + t));
            }
            if constexpr (MODE != CONS_EVAL) {
                if constexpr (MODE != CONS_ZZ) {
                    yk = ld_multiplier<CS>(y, ydf, kid);
                }
                if constexpr (MODE == CONS_LS && ZC) zb = zkc[kid];
                else if constexpr (std::is_same_v<CS, double>) zb = __ldg(p.b + kid);
                else zb = p.b_df ? ld_scalar<CS>(p.b, p.b_df, kid) : CS(__ldg(p.b + kid));
            }
        }
        // ---- dots of the group's constraints
        AU s_z[kConsBatch];                  // u_i.u_j (R-only modes, EVAL with U == V)
        // u_i.v_j and u_j.v_i apart: rounded sums of a float dot each, added in CS (in one float
        // chain q1 lost a fifth: rms 1.41e-8 -> 1.68e-8 at r = 20).  In FP64, and with double-float
        // rows and a float direction, CS adds no bits and the lanes' dots are added first: in
        // emulation the rms error of FP64 is the same within its noise, that of the mixed form
        // 3.49e-16 at r = 20 against 3.60e-16 with a sum of each and general products.
        constexpr bool kOneSum = MODE == CONS_LS && (std::is_same_v<AW, double> || df_by_float<TU, TV>());
        AW s_1[kConsBatch], s_1b[kConsBatch];
        AV s_2[kConsBatch];                  // v_i.v_j
#pragma unroll
        for (int u0 = 0; u0 < kConsBatch; u0 += UC) {
            if (u0 >= B) break;
            Unit<TU> ui[UC][1], uj[UC][1];
            Unit<TV> vi[UC][1], vj[UC][1];
            int i[UC], j[UC];
#pragma unroll
            for (int c = 0; c < UC; ++c) {
                i[c] = __shfl_sync(0xffffffffu, ii, rl.base_lane + u0 + c);
                j[c] = __shfl_sync(0xffffffffu, jj, rl.base_lane + u0 + c);
                if (u0 + c >= B) i[c] = -1;
            }
#pragma unroll
            for (int c = 0; c < UC; ++c) {
                const int Qa = i[c] >= 0 ? Q : 0;           // no constraint: zero rows
                const int64_t ri = i[c] >= 0 ? i[c] : 0, rj = i[c] >= 0 ? j[c] : 0;
                load_row<TU, 1>(ui[c], U, ri, ld, L, Qa, rl.lig);
                load_row<TU, 1>(uj[c], U, rj, ld, L, Qa, rl.lig);
                if constexpr (MODE == CONS_LS) {
                    load_row<TV, 1>(vi[c], V, ri, ld, L, Qa, rl.lig);
                    load_row<TV, 1>(vj[c], V, rj, ld, L, Qa, rl.lig);
                } else if constexpr (MODE == CONS_EVAL) {
                    if (!same) {
                        load_row<TV, 1>(vi[c], V, ri, ld, L, Qa, rl.lig);
                        load_row<TV, 1>(vj[c], V, rj, ld, L, Qa, rl.lig);
                    }
                }
            }
#pragma unroll
            for (int c = 0; c < UC; ++c) {
                if (u0 + c >= kConsBatch) continue;
                if constexpr (MODE == CONS_EVAL) {
                    if (same) {
                        s_z[u0 + c] = dot_lane<AU>(ui[c][0], uj[c][0]);
                    } else {
                        s_1[u0 + c] = dot_lane<AW>(ui[c][0], vj[c][0]);
                        s_1b[u0 + c] = dot_lane<AW>(uj[c][0], vi[c][0]);
                    }
                } else {
                    if constexpr (NEED_Z) s_z[u0 + c] = dot_lane<AU>(ui[c][0], uj[c][0]);
                    if constexpr (MODE == CONS_LS) {
                        s_1[u0 + c] = dot_lane<AW>(ui[c][0], vj[c][0]);
                        s_1b[u0 + c] = dot_lane<AW>(vi[c][0], uj[c][0]);
                        if constexpr (kOneSum) s_1[u0 + c] = s_1[u0 + c] + s_1b[u0 + c];
                        s_2[u0 + c] = dot_lane<AV>(vi[c][0], vj[c][0]);
                    }
                }
            }
        }
        if constexpr (MODE == CONS_EVAL) {
            if (same) {
                batch_sums(s_z, L, rl.lig);
            } else {
                batch_sums(s_1, L, rl.lig);
                batch_sums(s_1b, L, rl.lig);
            }
        } else {
            if constexpr (NEED_Z) batch_sums(s_z, L, rl.lig);
            if constexpr (MODE == CONS_LS) {
                batch_sums(s_1, L, rl.lig);
                if constexpr (!kOneSum) batch_sums(s_1b, L, rl.lig);
                batch_sums(s_2, L, rl.lig);
            }
        }
        // ---- the lane's own scalars
        if (!own) continue;
        const bool diag = ii == jj;
        if constexpr (MODE == CONS_EVAL) {
            const double a = __ldg(p.k_a + t);
            double val;
            if (same) val = (diag ? 1.0 : 2.0) * a * double(s_z[0]);
            else if (diag) val = a * double(s_1[0]);
            else val = a * (double(s_1[0]) + double(s_1b[0]));
            static_cast<double*>(out)[kid] = val;
        } else {
            const CS fa = diag ? ak : CS(2.0f) * ak;
            CS z;
            if constexpr (MODE == CONS_LS && ZC) z = zb;
            else z = fa * CS(s_z[0]) - zb;
            if constexpr (MODE == CONS_LS) {
                const CS yt = yk - rho_c * z;
                CS q1;
                if constexpr (kOneSum) q1 = fa * CS(s_1[0]);
                else q1 = fa * (CS(s_1[0]) + CS(s_1b[0]));
                const CS q2 = fa * CS(s_2[0]);
                accq[PL_YQ1] += PA(yt * q1);
                accq[PL_YQ2] += PA(yt * q2);
                accq[PL_Q1Q1] += PA(q1 * q1);
                accq[PL_Q1Q2] += PA(q1 * q2);
                accq[PL_Q2Q2] += PA(q2 * q2);
            } else {
                accq[PC_ZZ] += PA(z * z);
                if constexpr (MODE == CONS_YTIL) {
                    static_cast<CS*>(out)[kid] = yk - rho_c * z;
                    if (zk != nullptr) zkc[kid] = z;
                } else if constexpr (MODE == CONS_YUPD) {
                    const CS yn = yk - rho_c * z;
                    y[kid] = double(yn);
                    if constexpr (std::is_same_v<CS, dfloat>) {
                        if (ydf != nullptr) ydf[kid] = yn;
                    } else {
                        if (ydf != nullptr) ydf[kid] = dfloat(yn);
                    }
                    accq[PC_BY] += PA(zb * yn);
                }
            }
        }
    }
    if constexpr (MODE != CONS_EVAL) block_partials<NQ>(accq, part, vg.pslot);
}


template <typename TU, typename TV, int CPL, int MODE>
__device__ __forceinline__ void
k_cons_body(ProbDev p, int64_t k0, int64_t k1, const TU* __restrict__ U, const TV* __restrict__ V, int ld, int L, int Q,
            double* y, void* __restrict__ out, void* zk, dfloat* ydf, const Ctrl* ctrl, double rho_arg,
            double* __restrict__ part, VGrid vg) {
    if (p.k_ptr != nullptr) {
        k_cons_general<TU, TV, CPL, MODE>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, ctrl, rho_arg, part, vg);
        return;
    }
    const double rho = ctrl ? ctrl->rho : rho_arg;
    if constexpr (CPL == 1 && MODE == CONS_EVAL && std::is_same_v<arith_t<TU>, double>) {
        // A small map in FP64: taken eight at a time the constraints leave seven eighths of its
        // blocks idle, and a group's dots, in flight one at a time, follow each other (1000
        // constraints, r = 24: 20.6 us against 13.3; 2e4: 20.7 against 24.7).  At that number the
        // eighth fills half the chip; below 256 blocks a group takes one constraint.
        if (vg.nblk < 256) {
            k_cons_wide<TU, TV, CPL, MODE>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, ctrl, rho_arg, part, vg);
            return;
        }
    }
    if constexpr (CPL > 1) {
        k_cons_wide<TU, TV, CPL, MODE>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, ctrl, rho_arg, part, vg);
    } else if constexpr (MODE == CONS_LS && !std::is_same_v<arith_t<TU>, dfloat>) {
        // only the standalone line search runs without a cache of z, in FP64, FP32 or BF16
        if (zk != nullptr)
            k_cons_batch<TU, TV, MODE, true>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, rho, part, vg);
        else
            k_cons_batch<TU, TV, MODE, false>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, rho, part, vg);
    } else {
        k_cons_batch<TU, TV, MODE, true>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, rho, part, vg);
    }
}

}  // namespace lorads
