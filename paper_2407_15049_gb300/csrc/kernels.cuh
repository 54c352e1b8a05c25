// Streaming kernels of the LoRADS hot path (templates; instantiated per
// precision in kern_*.cu).  Every kernel is memory-bound by design: rows of the
// n x ld factors are read with 16-byte vector loads by groups of L lanes,
// sparse rows are gathered through L2, and all reductions end in per-block FP64
// partial sums that a single-block control kernel folds in a fixed order.
#pragma once

#include <type_traits>
#include "common.cuh"
#include "rows.cuh"
#include "cons.cuh"

namespace lorads {

// ================================================================== SpMM over C
// out = C X  (+ the diagonal-constraint part -A*(v) X when v != nullptr),
// optional epilogues:
//   EPI_LS : line-search partials at R (= argument R) along D (= X):
//            p1 = 2<CD, R>, p2 = <CD, D>, and for diagonal constraints
//            sum y~ q1, sum y~ q2, sum q1^2, sum q1 q2, sum q2^2
//   EPI_OBJ: <C X, X> (objective with X = R)

// PF (compile-time, so that the default form carries none of the others' code):
// 0 none, 1 the next row's bounds and L2 prefetches, 2 also two rows ahead.
template <typename TX, typename TO, typename TR, int CPL, int EPI, bool DENSE = false, int PF = 0>
__device__ __forceinline__ void
k_spmm_c_body(ProbDev p, const TX* __restrict__ X, TO* __restrict__ out, int ld, int L, int Q,
         const double* __restrict__ v, int write_out,
         const TR* __restrict__ R, const double* __restrict__ y, const void* __restrict__ zrow_v,
         const dfloat* __restrict__ ydf, const Ctrl* ctrl, double rho_arg, double* __restrict__ part, VGrid vg) {
    using A = arith_t<TO>;
    using TV = cval_t<TX>;
    using PA = part_t<TO, TR>;
    // scalar type of the per-row line-search terms: double on the FP64 path, otherwise
    // the arithmetic type of the direction (float, or double-float on the DF64 path)
    using LS = zrow_t<TX, TR>;
    const LS* __restrict__ zrow = static_cast<const LS*>(zrow_v);
    constexpr int NQ = EPI == EPI_LS ? PL_N : (EPI == EPI_OBJ ? PO_N : 1);
    PA accq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accq[q] = PA(0);
    const double rho = ctrl ? ctrl->rho : rho_arg;
    const LS rho_s = LS(rho);
    const TV* __restrict__ cv = cvals<TV>(p);
    static_assert(!DENSE || CPL == 1, "packed row groups hold one unit per lane");
    RowLoop rl(L, vg, DENSE);
    // With pf: the bounds (and constraint index) of this group's next row are loaded one
    // iteration ahead, and that row's entries, own-row streams and scalars are prefetched
    // into L2, so of its dependent load phases only the neighbour gathers wait on HBM.
    const bool own_row = EPI == EPI_LS || EPI == EPI_OBJ || (v != nullptr && p.dk != nullptr);
    // With pf == 2 the bounds run two rows ahead: the stored entries of the row after
    // next are prefetched, so that the next row's column indices are L2 hits one
    // iteration early and each lane can prefetch one neighbour row of D for it.
    int64_t s_nx = -1, e_nx = -1;
    int64_t s_n2 = -1, e_n2 = -1;
    for (int64_t base = rl.first; base < p.n; base += rl.stride) {
        const int64_t i = base + rl.gw;
        const bool act = rl.live && i < p.n;
        const int64_t s_cur = s_nx, e_cur = e_nx;
        s_nx = -1;
        int k_nx = -1;
        int jn = -1;
        if (PF != 0 && rl.live) {
            const int64_t nx = i + rl.stride;
            if (nx < p.n) {
                if (PF == 2 && s_n2 >= 0) {
                    s_nx = s_n2;
                    e_nx = e_n2;
                } else {
                    s_nx = __ldg(p.c_rowptr + nx);
                    e_nx = __ldg(p.c_rowptr + nx + 1);
                }
                if (own_row) prefetch_row<TX, CPL>(X, nx, ld, L, Q, rl.lig);
                if constexpr (EPI == EPI_LS) prefetch_row<TR, CPL>(R, nx, ld, L, Q, rl.lig);
                if (p.dk != nullptr && rl.lig == 0) {
                    k_nx = __ldg(p.dk + nx);
                    prefetch_l2(p.da + nx);
                    if (p.da_df != nullptr) prefetch_l2(p.da_df + nx);
                    if constexpr (EPI == EPI_LS)
                        if (zrow != nullptr) prefetch_l2(zrow + nx);
                }
            }
            if constexpr (PF == 2) {
                const int64_t n2 = nx + rl.stride;
                s_n2 = -1;
                if (n2 < p.n) {
                    s_n2 = __ldg(p.c_rowptr + n2);
                    e_n2 = __ldg(p.c_rowptr + n2 + 1);
                }
                if (s_nx >= 0 && s_nx + rl.lig < e_nx) jn = __ldg(p.c_col + s_nx + rl.lig);
            }
        }
        A acc[CPL][4];
#pragma unroll
        for (int c = 0; c < CPL; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c][e] = A(0);
        if (act) {
            int64_t s = s_cur >= 0 ? s_cur : __ldg(p.c_rowptr + i);
            const int64_t e_ = s_cur >= 0 ? e_cur : __ldg(p.c_rowptr + i + 1);
            // nonzeros in flight per lane: with one unit per lane, all the gathers of a
            // row of up to 8 stored entries are issued together (masked slots load nothing)
            constexpr int UN = CPL == 1 ? 8 : (CPL == 2 ? 4 : 3);
            for (; s < e_; s += UN) {
                if (CPL != 1 && s + UN > e_) break;
                int j[UN];
                A w[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u) {
                    const bool ok = s + u < e_;
                    j[u] = ok ? __ldg(p.c_col + s + u) : -1;
                    w[u] = ok ? A(ldv(cv + s + u)) : A(0);
                }
                Unit<TX> x[UN][CPL];
#pragma unroll
                for (int u = 0; u < UN; ++u) {
                    if (j[u] >= 0) load_row<TX, CPL>(x[u], X, j[u], ld, L, Q, rl.lig);
                    else
#pragma unroll
                        for (int c = 0; c < CPL; ++c)
#pragma unroll
                            for (int e = 0; e < 4; ++e) x[u][c].v[e] = 0;
                }
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (j[u] >= 0)
#pragma unroll
                        for (int c = 0; c < CPL; ++c)
#pragma unroll
                            for (int e = 0; e < 4; ++e) acc[c][e] = fma(w[u], A(x[u][c].v[e]), acc[c][e]);
            }
            for (; s < e_; ++s) {
                const int j0 = __ldg(p.c_col + s);
                const A w0 = A(ldv(cv + s));
                Unit<TX> x0[CPL];
                load_row<TX, CPL>(x0, X, j0, ld, L, Q, rl.lig);
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[c][e] = fma(w0, A(x0[c].v[e]), acc[c][e]);
            }
            if constexpr (PF == 2) {
                // one neighbour row of the next row (its first and last element), and the
                // stored entries of the row after next
                if (jn >= 0) {
                    const TX* rowp = X + (int64_t)jn * ld;
                    prefetch_l2(rowp);
                    prefetch_l2(rowp + ld - 1);
                }
                if (s_n2 >= 0 && rl.lig < 2 && e_n2 > s_n2) {
                    const int64_t q = rl.lig == 0 ? s_n2 : e_n2 - 1;
                    prefetch_l2(p.c_col + q);
                    prefetch_l2(cv + q);
                }
            } else if (s_nx >= 0 && rl.lig < 2 && e_nx > s_nx) {
                // the next row's stored entries (first and last sector) and multiplier terms
                const int64_t q = rl.lig == 0 ? s_nx : e_nx - 1;
                prefetch_l2(p.c_col + q);
                prefetch_l2(cv + q);
            }
            if (k_nx >= 0) {
                if (v != nullptr) prefetch_l2(v + k_nx);
                if constexpr (EPI == EPI_LS) {
                    prefetch_l2(ydf ? static_cast<const void*>(ydf + k_nx) : static_cast<const void*>(y + k_nx));
                    if (zrow == nullptr) prefetch_l2(p.b_df ? static_cast<const void*>(p.b_df + k_nx)
                                                            : static_cast<const void*>(p.b + k_nx));
                }
            }
            if (v != nullptr && p.dk != nullptr) {
                const int k = __ldg(p.dk + i);
                if (k >= 0) {
                    const A w = A(-__ldg(p.da + i) * __ldg(v + k));
                    Unit<TX> xi[CPL];
                    load_row<TX, CPL>(xi, X, i, ld, L, Q, rl.lig);
#pragma unroll
                    for (int c = 0; c < CPL; ++c)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[c][e] = fma(w, A(xi[c].v[e]), acc[c][e]);
                }
            }
            if (write_out) {
                Unit<TO> o[CPL];
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[c].v[e] = acc[c][e];
                store_row<TO, CPL>(o, out, i, ld, L, Q, rl.lig);
            }
        }
        if constexpr (EPI == EPI_OBJ) {
            if (act) {
                Unit<TX> xi[CPL];
                load_row<TX, CPL>(xi, X, i, ld, L, Q, rl.lig);
                A t = A(0);
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) t = fma(acc[c][e], A(xi[c].v[e]), t);
                accq[PO_CRR] += PA(t);
            }
        }
        if constexpr (EPI == EPI_LS) {
            using AW = wide_t<TR, TX>;           // |r|^2 (when not cached) and <CD, R>
            using AD = arith_t<TX>;              // products of D with D and with R
            AW t_p1 = AW(0), t_rr = AW(0);
            AD t_p2 = AD(0), t_rd = AD(0), t_dd = AD(0);
            if (act) {
                Unit<TX> di[CPL];
                Unit<TR> ri[CPL];
                load_row<TX, CPL>(di, X, i, ld, L, Q, rl.lig);
                load_row_stream<TR, CPL>(ri, R, i, ld, L, Q, rl.lig);
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const AD d = AD(di[c].v[e]);
                        const AD rlow = AD(ri[c].v[e]);
                        t_p2 = fma(AD(acc[c][e]), d, t_p2);
                        t_rd = fma(rlow, d, t_rd);
                        t_dd = fma(d, d, t_dd);
                        if (zrow == nullptr) {
                            const AW r = AW(ri[c].v[e]);
                            t_p1 = fma(AW(acc[c][e]), r, t_p1);
                            t_rr = fma(r, r, t_rr);
                        }
                    }
            }
            accq[PL_P2] += t_p2;
            if (zrow == nullptr) accq[PL_P1] += PA(AW(2) * t_p1);
            if (p.dk != nullptr) {
                if constexpr (DENSE) {
                    if (zrow == nullptr) t_rr = group_sum_packed(t_rr, L, rl.base_lane);
                    t_rd = group_sum_packed(t_rd, L, rl.base_lane);
                    t_dd = group_sum_packed(t_dd, L, rl.base_lane);
                } else {
                    if (zrow == nullptr) t_rr = group_sum(t_rr, L);
                    t_rd = group_sum(t_rd, L);
                    t_dd = group_sum(t_dd, L);
                }
                if (act && rl.lig == 0) {
                    const int k = __ldg(p.dk + i);
                    if (k >= 0) {
                        if constexpr (std::is_same_v<LS, double>) {
                            const double a = __ldg(p.da + i);
                            const double z = zrow ? zrow[i] : a * double(t_rr) - __ldg(p.b + k);
                            const double yt = ld_multiplier<double>(y, nullptr, k) - rho * z;
                            const double q1 = 2.0 * a * double(t_rd);
                            const double q2 = a * double(t_dd);
                            accq[PL_YQ1] += PA(yt * q1);
                            accq[PL_YQ2] += PA(yt * q2);
                            accq[PL_Q1Q1] += PA(q1 * q1);
                            accq[PL_Q1Q2] += PA(q1 * q2);
                            accq[PL_Q2Q2] += PA(q2 * q2);
                        } else {
                            // line-search terms in the direction's arithmetic; z from the
                            // row cache, else |r|^2 in double-float
                            const LS a = ld_scalar<LS>(p.da, p.da_df, i);
                            LS z;
                            if (zrow) {
                                z = zrow[i];
                            } else {
                                const dfloat zz = dfloat(t_rr) * ld_scalar<dfloat>(p.da, p.da_df, i) -
                                                  ld_scalar<dfloat>(p.b, p.b_df, k);
                                z = LS(zz);
                            }
                            const LS yv = ld_multiplier<LS>(y, ydf, k);
                            const LS yt = yv - rho_s * z;
                            const LS q1 = LS(2) * a * LS(t_rd);
                            const LS q2 = a * LS(t_dd);
                            accq[PL_YQ1] += PA(yt * q1);
                            accq[PL_YQ2] += PA(yt * q2);
                            accq[PL_Q1Q1] += PA(q1 * q1);
                            accq[PL_Q1Q2] += PA(q1 * q2);
                            accq[PL_Q2Q2] += PA(q2 * q2);
                        }
                    }
                }
            }
        }
    }
    if constexpr (EPI != EPI_NONE) block_partials<NQ>(accq, part, vg.pslot);
}

// ================================================================== SpMM over the
// off-diagonal constraint pattern:  out = beta_acc * out + alpha * A*_off(v) X
// VDF: v holds double-float values and each weight alpha a v_k is formed in the
// output's arithmetic from the double-float coefficient mirror (no FP64
// operation); otherwise v is double and the weight is formed in FP64.  v is y~, which a
// persistent kernel rewrites every iteration: no read-only load.
template <typename TX, typename TO, int CPL, bool VDF>
__device__ __forceinline__ A_of_t<TO> spmm_a_weight(const ProbDev& p, const void* v, double alpha, A_of_t<TO> alpha_a,
                                                   int64_t s) {
    using A = A_of_t<TO>;
    const int k = __ldg(p.a_k + s);
    if constexpr (VDF) {
        return alpha_a * ld_scalar<A>(nullptr, p.a_adf, s) * ld_multiplier<A>(nullptr, static_cast<const dfloat*>(v), k);
    } else {
        return A(alpha * __ldg(p.a_a + s) * ld_multiplier<double>(static_cast<const double*>(v), nullptr, k));
    }
}

// acc += the weighted rows of the slots [s, s1), four slots in flight, each weight formed by
// every lane.  For groups of one and two lanes, which have little to share and, with a slot a
// lane as the wider groups take them, one or two rows in flight (product of 4e5 constraints on 2e4
// rows, v double, us here and with a slot a lane: FP64, ld = 4, 49 and 102, ld = 8, 64 and 91; bf16,
// ld = 4, 33 and 64; 1000 x 60000, FP64, ld = 4: 196 and 500).
template <typename TX, typename TO, int CPL, bool VDF>
__device__ __forceinline__ void
spmm_a_row_narrow(const ProbDev& p, const TX* __restrict__ X, int ld, int L, int Q, const void* __restrict__ v,
                  double alpha, int lig, int64_t s, int64_t s1, A_of_t<TO> (&acc)[CPL][4]) {
    using A = A_of_t<TO>;
    const A alpha_a = A(alpha);
    constexpr int UN = 4;
    for (; s + UN <= s1; s += UN) {
        int j[UN];
        A w[UN];
#pragma unroll
        for (int u = 0; u < UN; ++u) {
            j[u] = __ldg(p.a_col + s + u);
            w[u] = spmm_a_weight<TX, TO, CPL, VDF>(p, v, alpha, alpha_a, s + u);
        }
        Unit<TX> x[UN][CPL];
#pragma unroll
        for (int u = 0; u < UN; ++u) load_row<TX, CPL>(x[u], X, j[u], ld, L, Q, lig);
#pragma unroll
        for (int u = 0; u < UN; ++u)
#pragma unroll
            for (int c = 0; c < CPL; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[c][e] = fma(w[u], A(x[u][c].v[e]), acc[c][e]);
    }
    for (; s < s1; ++s) {
        const int j = __ldg(p.a_col + s);
        const A w = spmm_a_weight<TX, TO, CPL, VDF>(p, v, alpha, alpha_a, s);
        Unit<TX> x[CPL];
        load_row<TX, CPL>(x, X, j, ld, L, Q, lig);
#pragma unroll
        for (int c = 0; c < CPL; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c][e] = fma(w, A(x[c].v[e]), acc[c][e]);
    }
}

// NARROW: groups of one or two lanes (L <= 2), else L >= 4.
template <typename TX, typename TO, int CPL, bool VDF, bool NARROW>
__device__ __forceinline__ void
k_spmm_a_body(ProbDev p, const TX* __restrict__ X, TO* __restrict__ out, int ld, int L, int Q,
         const void* __restrict__ v, double alpha, int accumulate, VGrid vg) {
    using A = arith_t<TO>;
    const A alpha_a = A(alpha);
    RowLoop rl(L, vg);
    // Slots per trip of a group: lane u loads slot u of the batch (coalesced) and forms
    // its weight; the rows are then gathered with the slots broadcast by shuffles.  Forming
    // each weight in every lane of the group made the pass FP64-bound where v is double (two
    // products and a conversion per slot and lane).
    const int B = L < 8 ? L : 8;
    constexpr int UN = CPL == 1 ? (sizeof(TX) == 8 ? 4 : 8) : 2;     // rows in flight per lane
    // bf16 rows: a slot past the end loads a row of zeros under a mask; with a branch around each
    // load they were not in flight together (5.4e6 slots on 1e5 rows, ld = 24: 190 and 109 us; 1000 x
    // 60000, ld = 16: 141 and 95, where four slots in every lane took 116).  The 4- and 8-byte
    // rows keep the branch: FP64 1000 x 60000, ld = 16: 152, 172 under the mask.
    constexpr bool kMasked = sizeof(TX) == 2;
    for (int64_t base = rl.first; base < p.n; base += rl.stride) {
        const int64_t i = base + rl.gw;
        const bool act = i < p.n;
        A acc[CPL][4];
#pragma unroll
        for (int c = 0; c < CPL; ++c)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[c][e] = A(0);
        const int64_t s0 = act ? __ldg(p.a_rowptr + i) : 0, s1 = act ? __ldg(p.a_rowptr + i + 1) : 0;
        if constexpr (NARROW) {
            spmm_a_row_narrow<TX, TO, CPL, VDF>(p, X, ld, L, Q, v, alpha, rl.lig, s0, s1, acc);
        } else {
            // warp-uniform loop: the groups of a warp may hold different numbers of slots
            for (int64_t s = s0; __any_sync(0xffffffffu, s < s1); s += B) {
                const int64_t q = s + rl.lig;
                int jo = -1;
                A wo = A(0);
                if (rl.lig < B && q < s1) {
                    jo = __ldg(p.a_col + q);
                    wo = spmm_a_weight<TX, TO, CPL, VDF>(p, v, alpha, alpha_a, q);
                }
#pragma unroll
                for (int u0 = 0; u0 < 8; u0 += UN) {
                    if (u0 >= B) break;
                    int j[UN];
                    A w[UN];
                    Unit<TX> x[UN][CPL];
#pragma unroll
                    for (int u = 0; u < UN; ++u) {
                        const int src = rl.base_lane + (u0 + u < B ? u0 + u : 0);
                        j[u] = __shfl_sync(0xffffffffu, jo, src);
                        w[u] = shfl_idx(wo, src);
                        if (u0 + u >= B) j[u] = -1;
                    }
#pragma unroll
                    for (int u = 0; u < UN; ++u) {
                        if constexpr (kMasked)
                            load_row<TX, CPL>(x[u], X, j[u] >= 0 ? j[u] : 0, ld, L, j[u] >= 0 ? Q : 0, rl.lig);
                        else if (j[u] >= 0)
                            load_row<TX, CPL>(x[u], X, j[u], ld, L, Q, rl.lig);
                    }
#pragma unroll
                    for (int u = 0; u < UN; ++u)
                        if (j[u] >= 0)
#pragma unroll
                            for (int c = 0; c < CPL; ++c)
#pragma unroll
                                for (int e = 0; e < 4; ++e) acc[c][e] = fma(w[u], A(x[u][c].v[e]), acc[c][e]);
                }
            }
        }
        if (!act) continue;
        Unit<TO> o[CPL];
        if (accumulate) {
            load_row<TO, CPL>(o, out, i, ld, L, Q, rl.lig);
#pragma unroll
            for (int c = 0; c < CPL; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[c].v[e] = arith_t<TO>(o[c].v[e]) + acc[c][e];
        } else {
#pragma unroll
            for (int c = 0; c < CPL; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[c].v[e] = acc[c][e];
        }
        store_row<TO, CPL>(o, out, i, ld, L, Q, rl.lig);
    }
}

// ================================================================== direction
// D = cG G + sum_u (cS_u S_u + cY_u Y_u) over the stored pairs (the two-loop
// recursion of Algorithm 1 carried out on coefficients); partials <G,D>, ||D||^2.
// TDIR: storage of D and of the stored pairs (they may be stored narrower than G;
// <G,D> and ||D||^2 are then taken of the stored direction).
template <typename TD, typename TDIR = TD>
__device__ __forceinline__ void
k_dir_body(int64_t nunits, const TD* __restrict__ G, TDIR* __restrict__ D, const TDIR* __restrict__ hist,
      int64_t slot_stride, const Ctrl* ctrl, double* __restrict__ part, VGrid vg) {
    using A = arith_t<TD>;
    using PA = part_t<TD, TD>;
    PA accq[PD_N] = {PA(0), PA(0)};
    const int mem = ctrl->mem_count;
    const A cG = A(ctrl->cG);
    A cS[kMaxMem], cY[kMaxMem];
    const TDIR* Sp[kMaxMem];
    const TDIR* Yp[kMaxMem];
#pragma unroll
    for (int t = 0; t < kMaxMem; ++t) {
        const int s = ctrl->order[t];
        cS[t] = A(ctrl->cS[s]);
        cY[t] = A(ctrl->cY[s]);
        Sp[t] = hist + (int64_t)(2 * s) * slot_stride;
        Yp[t] = hist + (int64_t)(2 * s + 1) * slot_stride;
    }
    const int64_t stride = (int64_t)vg.nblk * blockDim.x;
    for (int64_t u = vg.bid * (int64_t)blockDim.x + threadIdx.x; u < nunits; u += stride) {
        Unit<TD> g, d;
        g.load_stream(G + u * 4);
#pragma unroll
        for (int e = 0; e < 4; ++e) d.v[e] = cG * A(g.v[e]);
#pragma unroll
        for (int t = 0; t < kMaxMem; ++t) {
            if (t < mem) {
                Unit<TDIR> s, y;
                s.load_stream(Sp[t] + u * 4);
                y.load_stream(Yp[t] + u * 4);
#pragma unroll
                for (int e = 0; e < 4; ++e) d.v[e] = fma(cS[t], A(s.v[e]), fma(cY[t], A(y.v[e]), A(d.v[e])));
            }
        }
        Unit<TDIR> dst;
        A gd = A(0), dd = A(0);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            dst.v[e] = as_stored<TDIR>(A(d.v[e]));
            const A dv = A(dst.v[e]);           // value as stored
            gd += A(g.v[e]) * dv;
            dd += dv * dv;
        }
        dst.store(D + u * 4);
        accq[PD_GD] += gd;
        accq[PD_DD] += dd;
    }
    block_partials<PD_N>(accq, part, vg.pslot);
}

// ================================================================== step (flat)
// R += tau D, CR += tau CD  (used when the gradient needs a separate pattern pass)
template <typename TR, typename TD, typename TDIR = TD>
__device__ __forceinline__ void
k_step_body(int64_t nunits, TR* __restrict__ R, TR* __restrict__ CR, const TDIR* __restrict__ D,
       const TD* __restrict__ CD, const Ctrl* ctrl, VGrid vg) {
    using A = arith_t<TR>;
    const A tau = A(ctrl->tau);
    const int64_t stride = (int64_t)vg.nblk * blockDim.x;
    for (int64_t u = vg.bid * (int64_t)blockDim.x + threadIdx.x; u < nunits; u += stride) {
        Unit<TR> r, cr;
        Unit<TDIR> d;
        Unit<TD> cd;
        r.load_stream(R + u * 4);
        cr.load_stream(CR + u * 4);
        d.load_stream(D + u * 4);
        cd.load_stream(CD + u * 4);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            r.v[e] = fma(tau, A(d.v[e]), A(r.v[e]));
            cr.v[e] = fma(tau, A(cd.v[e]), A(cr.v[e]));
        }
        r.store_stream(R + u * 4);
        cr.store_stream(CR + u * 4);
    }
}

// ================================================================== row update
// Per row i (group of L lanes):
//   STEP : r += tau d, cr += tau cd                         (Algorithm 1 step)
//   grad : g' = 2 (cr - a_i y~_k r - w_i),  y~_k = y_k - rho (a_i |r|^2 - b_k)
//          for the diagonal constraint k of row i, w = A*_off(y~) R (if given)
//   HIST : s_new = tau d, y_new = g' - g   into the new slot, and the dot
//          products that keep the Gram data of the stored pairs current
//          (<s_new,y_new>, ||y_new||^2, <g',y_new>, and per stored pair v:
//          <s_new,y_v>, <s_v,y_new>, <y_new,y_v>)
// partials: ||g'||^2, sum z_k^2 (diagonal constraints), and the Gram dots.
// 3 resident blocks per SM where the registers allow it without real spills
// (one unit per lane, FP32-unit arithmetic), 2 otherwise.
template <typename TR, typename TD, int CPL>
constexpr int update_min_blocks() {
    return (CPL == 1 && !std::is_same_v<arith_t<TR>, double>) ? 3 : 2;
}

// MAXOLD: most stored pairs besides the new one (T - 1 of Algorithm 1) the pass is
// compiled for; the Gram accumulators of the others are compile-time zeros, which
// frees their registers (T = 2: 8 partial sums instead of 14).
template <typename TR, typename TD, int CPL, bool STEP, bool HIST, typename TDIR = TD, bool DENSE = false,
          int MAXOLD = kMaxMem - 1>
__device__ __forceinline__ void
k_update_body(ProbDev p, TR* __restrict__ R, TR* __restrict__ CR, const TDIR* __restrict__ D,
         const TD* __restrict__ CD, TD* __restrict__ G, const TD* __restrict__ W,
         TDIR* __restrict__ hist, int64_t slot_stride, int ld, int L, int Q,
         const double* __restrict__ y, const dfloat* __restrict__ ydf, void* __restrict__ zrow_v,
         const Ctrl* ctrl, double* __restrict__ part, VGrid vg, int pf = 0) {
    using AR = arith_t<TR>;
    using AD = arith_t<TD>;
    using PA = part_t<TR, TD>;
    using RS = rowscalar_t<TR, TD>;             // per-row scalars (no FP64 off the FP64 path)
    using ZS = zrow_t<TD, TR>;
    ZS* __restrict__ zrow = static_cast<ZS*>(zrow_v);
    const RS rho_r = RS(ctrl->rho);
    PA accq[PU_N];
#pragma unroll
    for (int q = 0; q < PU_N; ++q) accq[q] = PA(0);
    const double taud = ctrl->tau;
    const AR tau = AR(taud);
    const AD tau_d = AD(taud);
    int nold = 0;
    TDIR* Snew = nullptr;                       // pairs stored in the direction's type
    TDIR* Ynew = nullptr;
    static_assert(MAXOLD >= 1 && MAXOLD <= kMaxMem - 1, "stored pairs");
    const TDIR* So[MAXOLD];
    const TDIR* Yo[MAXOLD];
    if constexpr (HIST) {
        nold = ctrl->old_count;
        const int ns = ctrl->new_slot;
        Snew = hist + (int64_t)(2 * ns) * slot_stride;
        Ynew = hist + (int64_t)(2 * ns + 1) * slot_stride;
#pragma unroll
        for (int t = 0; t < MAXOLD; ++t) {
            const int s = ctrl->old_slots[t < nold ? t : 0];
            So[t] = hist + (int64_t)(2 * s) * slot_stride;
            Yo[t] = hist + (int64_t)(2 * s + 1) * slot_stride;
        }
    }
    static_assert(!DENSE || CPL == 1, "packed row groups hold one unit per lane");
    RowLoop rl(L, vg, DENSE);
    for (int64_t base = rl.first; base < p.n; base += rl.stride) {
        const int64_t i = base + rl.gw;
        const bool act = rl.live && i < p.n;
        int knx = -1;                            // constraint of the next row, loaded one iteration ahead
        if (pf != 0) {
            // Prefetch the next row of this group into L2: the several dependent load
            // phases of that iteration (R..C D, the old G, each stored pair) then wait
            // on L2 instead of HBM.
            const int64_t nx = i + rl.stride;
            if (rl.live && nx < p.n) {
                prefetch_row<TR, CPL>(R, nx, ld, L, Q, rl.lig);
                prefetch_row<TR, CPL>(CR, nx, ld, L, Q, rl.lig);
                if constexpr (STEP || HIST) prefetch_row<TDIR, CPL>(D, nx, ld, L, Q, rl.lig);
                if constexpr (STEP) prefetch_row<TD, CPL>(CD, nx, ld, L, Q, rl.lig);
                if (W != nullptr) prefetch_row<TD, CPL>(W, nx, ld, L, Q, rl.lig);
                if constexpr (HIST) {
                    prefetch_row<TD, CPL>(G, nx, ld, L, Q, rl.lig);
#pragma unroll
                    for (int t = 0; t < MAXOLD; ++t)
                        if (t < nold) {
                            prefetch_row<TDIR, CPL>(So[t], nx, ld, L, Q, rl.lig);
                            prefetch_row<TDIR, CPL>(Yo[t], nx, ld, L, Q, rl.lig);
                        }
                }
                if (p.dk != nullptr && rl.lig == 0) {
                    knx = __ldg(p.dk + nx);
                    if constexpr (std::is_same_v<RS, double>) prefetch_l2(p.da + nx);
                    else prefetch_l2(p.da_df + nx);
                }
            }
        }
        Unit<TR> r[CPL], cr[CPL];
        Unit<TDIR> d[CPL];
        AR rr = AR(0);
        if (act) {
            load_row_stream<TR, CPL>(r, R, i, ld, L, Q, rl.lig);
            load_row_stream<TR, CPL>(cr, CR, i, ld, L, Q, rl.lig);
            if constexpr (STEP || HIST) load_row_stream<TDIR, CPL>(d, D, i, ld, L, Q, rl.lig);
            if constexpr (STEP) {
                Unit<TD> cd[CPL];
                load_row_stream<TD, CPL>(cd, CD, i, ld, L, Q, rl.lig);
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        r[c].v[e] = step_add<AR, AD>(AR(r[c].v[e]), tau, tau_d, AD(d[c].v[e]));
                        cr[c].v[e] = step_add<AR, AD>(AR(cr[c].v[e]), tau, tau_d, AD(cd[c].v[e]));
                    }
                store_row<TR, CPL>(r, R, i, ld, L, Q, rl.lig);
                store_row<TR, CPL>(cr, CR, i, ld, L, Q, rl.lig);
            }
#pragma unroll
            for (int c = 0; c < CPL; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) rr = sq_add<AR>(rr, AR(r[c].v[e]));
        }
        // diagonal-constraint coefficient a_i y~_k of row i
        AR coef = AR(0);
        if (p.dk != nullptr) {
            if constexpr (DENSE) rr = group_sum_packed(rr, L, rl.base_lane);
            else rr = group_sum(rr, L);
            if (act) {
                const int k = __ldg(p.dk + i);
                if (k >= 0) {
                    const RS a = ld_scalar<RS>(p.da, p.da_df, i);
                    const RS z = a * RS(rr) - ld_scalar<RS>(p.b, p.b_df, k);
                    const RS yv = ld_multiplier<RS>(y, ydf, k);
                    coef = AR(a * (yv - rho_r * z));
                    if (rl.lig == 0) {
                        accq[PU_ZZ] += PA(z * z);
                        if (zrow != nullptr) zrow[i] = ZS(z);
                    }
                }
            }
        }
        if (act) {
            Unit<TD> g[CPL];
            Unit<TD> w[CPL];
            if (W != nullptr) load_row_stream<TD, CPL>(w, W, i, ld, L, Q, rl.lig);
#pragma unroll
            for (int c = 0; c < CPL; ++c)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    if (W != nullptr) {
                        const AR gv = AR(cr[c].v[e]) - coef * AR(r[c].v[e]) - AR(w[c].v[e]);
                        g[c].v[e] = AD(AR(2) * gv);
                    } else {
                        g[c].v[e] = grad_elem<AR, AD>(AR(cr[c].v[e]), coef, AR(r[c].v[e]));
                    }
                }
            if constexpr (HIST) {
                // the new pair as stored (rounded to TDIR): the Gram dots below are those
                // of the stored vectors, which the direction pass reads
                Unit<TD> gold[CPL];
                Unit<TDIR> sn[CPL], yn[CPL];
                load_row_stream<TD, CPL>(gold, G, i, ld, L, Q, rl.lig);
#pragma unroll
                for (int c = 0; c < CPL; ++c)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        sn[c].v[e] = as_stored<TDIR>(tau_d * AD(d[c].v[e]));
                        yn[c].v[e] = as_stored<TDIR>(AD(g[c].v[e]) - AD(gold[c].v[e]));
                    }
                store_row<TDIR, CPL>(sn, Snew, i, ld, L, Q, rl.lig);
                store_row<TDIR, CPL>(yn, Ynew, i, ld, L, Q, rl.lig);
                accq[PU_GYN] += dot_units<AD>(g, yn);
                accq[PU_SYN] += dot_units<AD>(sn, yn);
                accq[PU_YYN] += dot_units<AD>(yn, yn);
#pragma unroll
                for (int t = 0; t < MAXOLD; ++t) {
                    if (t < nold) {
                        Unit<TDIR> so[CPL], yo[CPL];
                        load_row_stream<TDIR, CPL>(so, So[t], i, ld, L, Q, rl.lig);
                        load_row_stream<TDIR, CPL>(yo, Yo[t], i, ld, L, Q, rl.lig);
                        PA* q = accq + PU_FIXED + PU_PER_OLD * t;
                        q[0] += dot_units<AD>(sn, yo);
                        q[1] += dot_units<AD>(so, yn);
                        q[2] += dot_units<AD>(yn, yo);
                    }
                }
            }
            store_row<TD, CPL>(g, G, i, ld, L, Q, rl.lig);
            accq[PU_GG] += dot_units<AD>(g, g);
        }
        if (knx >= 0) {
            // the next row's multiplier and right-hand side
            if constexpr (std::is_same_v<RS, double>) {
                prefetch_l2(y + knx);
                prefetch_l2(p.b + knx);
            } else {
                prefetch_l2(ydf ? static_cast<const void*>(ydf + knx) : static_cast<const void*>(y + knx));
                prefetch_l2(p.b_df + knx);
            }
        }
    }
    block_partials<PU_N>(accq, part, vg.pslot);
}

// ================================================================== kernels
// One launch per body over the hardware grid; a kernel of the captured
// iteration graph first checks the phase flags of the control block.

// Resident blocks per SM the SpMM over C is compiled for: for float rows 4 (64
// registers, no spills) with one unit per lane and 3 (85 registers) with more,
// for bf16 rows 3 (their conversions take more registers), where the pass is
// bound by the latency of its dependent loads; otherwise left to the compiler.
template <typename TX, typename TO, int CPL>
constexpr int spmm_min_blocks() {
    if constexpr (std::is_same_v<TX, float> && std::is_same_v<TO, float>) return CPL == 1 ? 4 : 3;
    else if constexpr (std::is_same_v<TX, __nv_bfloat16> && std::is_same_v<TO, float>) return 3;
    else return 1;
}

template <typename TX, typename TO, typename TR, int CPL, int EPI, bool DENSE = false, int PF = 0>
__global__ void __launch_bounds__(kThreads, (spmm_min_blocks<TX, TO, CPL>()))
k_spmm_c(ProbDev p, const TX* __restrict__ X, TO* __restrict__ out, int ld, int L, int Q,
         const double* __restrict__ v, int write_out,
         const TR* __restrict__ R, const double* __restrict__ y, const void* __restrict__ zrow_v,
         const dfloat* __restrict__ ydf, const Ctrl* ctrl, double rho_arg, double* __restrict__ part,
         const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_spmm_c_body<TX, TO, TR, CPL, EPI, DENSE, PF>(p, X, out, ld, L, Q, v, write_out, R, y, zrow_v, ydf, ctrl, rho_arg,
                                                   part, hw_grid());
}

template <typename TX, typename TO, int CPL, bool VDF, bool NARROW>
__global__ void __launch_bounds__(kThreads)
k_spmm_a(ProbDev p, const TX* __restrict__ X, TO* __restrict__ out, int ld, int L, int Q,
         const void* __restrict__ v, double alpha, int accumulate, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_spmm_a_body<TX, TO, CPL, VDF, NARROW>(p, X, out, ld, L, Q, v, alpha, accumulate, hw_grid());
}

template <typename TU, typename TV, int CPL, int MODE>
__global__ void __launch_bounds__(kThreads, 2)
k_cons(ProbDev p, int64_t k0, int64_t k1, const TU* __restrict__ U, const TV* __restrict__ V, int ld, int L, int Q,
       double* y, void* __restrict__ out, void* zk, dfloat* ydf, const Ctrl* ctrl, double rho_arg,
       double* __restrict__ part, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_cons_body<TU, TV, CPL, MODE>(p, k0, k1, U, V, ld, L, Q, y, out, zk, ydf, ctrl, rho_arg, part, hw_grid());
}

template <typename TD, typename TDIR = TD>
__global__ void __launch_bounds__(kThreads)
k_dir(int64_t nunits, const TD* __restrict__ G, TDIR* __restrict__ D, const TDIR* __restrict__ hist,
      int64_t slot_stride, const Ctrl* ctrl, double* __restrict__ part, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_dir_body<TD, TDIR>(nunits, G, D, hist, slot_stride, ctrl, part, hw_grid());
}

template <typename TR, typename TD, typename TDIR = TD>
__global__ void __launch_bounds__(kThreads)
k_step(int64_t nunits, TR* __restrict__ R, TR* __restrict__ CR, const TDIR* __restrict__ D,
       const TD* __restrict__ CD, const Ctrl* ctrl, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_step_body<TR, TD, TDIR>(nunits, R, CR, D, CD, ctrl, hw_grid());
}

template <typename TR, typename TD, int CPL, bool STEP, bool HIST, typename TDIR = TD>
__global__ void __launch_bounds__(kThreads, (update_min_blocks<TR, TD, CPL>()))
k_update(ProbDev p, TR* __restrict__ R, TR* __restrict__ CR, const TDIR* __restrict__ D,
         const TD* __restrict__ CD, TD* __restrict__ G, const TD* __restrict__ W,
         TDIR* __restrict__ hist, int64_t slot_stride, int ld, int L, int Q,
         const double* __restrict__ y, const dfloat* __restrict__ ydf, void* __restrict__ zrow_v,
         const Ctrl* ctrl, double* __restrict__ part, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    k_update_body<TR, TD, CPL, STEP, HIST, TDIR>(p, R, CR, D, CD, G, W, hist, slot_stride, ld, L, Q, y, ydf, zrow_v, ctrl, part, hw_grid());
}

// The step update with EXTRA more resident blocks per SM (fewer registers per
// thread, some spilled to L1): more rows in flight for the latency-bound pass.
// DENSE: packed row groups of L = Q lanes (RowLoop).  MAXOLD: see k_update_body.
template <typename TR, typename TD, int CPL, int EXTRA, typename TDIR = TD, bool DENSE = false,
          int MAXOLD = kMaxMem - 1>
__global__ void __launch_bounds__(kThreads, (update_min_blocks<TR, TD, CPL>() + EXTRA))
k_update_step_occ(ProbDev p, TR* __restrict__ R, TR* __restrict__ CR, const TDIR* __restrict__ D,
                  const TD* __restrict__ CD, TD* __restrict__ G, const TD* __restrict__ W,
                  TDIR* __restrict__ hist, int64_t slot_stride, int ld, int L, int Q,
                  const double* __restrict__ y, const dfloat* __restrict__ ydf, void* __restrict__ zrow_v,
                  const Ctrl* ctrl, double* __restrict__ part, const Ctrl* gate, int ph, int pf) {
    if (gated_off(gate, ph)) return;
    k_update_body<TR, TD, CPL, true, true, TDIR, DENSE, MAXOLD>(p, R, CR, D, CD, G, W, hist, slot_stride, ld, L, Q, y,
                                                                 ydf, zrow_v, ctrl, part, hw_grid(), pf);
}

}  // namespace lorads
