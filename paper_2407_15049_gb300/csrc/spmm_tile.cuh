// The SpMM over C for rows of one unit per lane (up to 128 elements): a warp owns a tile of
// consecutive rows, its lanes in packed groups of Q = ld/4 (one unit each, floor(32/Q) rows
// at a time, nsub times).
#pragma once

#include "rows.cuh"
#include "cons.cuh"

namespace lorads {

constexpr int kTileLaneRows = 192;        // row sums of a tile: rows x Q partials at most
// Stored entries of a tile held in shared memory.  A tile of 30 rows (n >= 3e5, ld = 20) holds more
// from 4.3 neighbours a row on, and reads them from global memory; the FP64 line search is still
// the faster form there (12 neighbours: 0.47 of k_spmm_c's time).
constexpr int kTileEntries = 160;

// Threads per block: 8-byte forms take twice the shared memory a warp.
template <typename TX, typename TO> constexpr int tile_threads() {
    return sizeof(arith_t<TX>) == 8 || sizeof(arith_t<TO>) == 8 ? 128 : 256;
}
// Resident blocks the kernel is compiled for.
constexpr int kTileBlocks = 4;

// Row groups a warp takes in turn (nsub) and the grid: one resident wave of warps that walk
// the tiles; small problems take tiles of one row group, so that every row has its lanes.
struct TilePlan {
    int nsub, blocks;
};
inline TilePlan tile_plan(int64_t n, int Q, int most_blocks, int threads) {
    const int rpw = 32 / Q, nw = threads / 32;
    int most = 32 / rpw;
    if (most > kTileLaneRows / (rpw * Q)) most = kTileLaneRows / (rpw * Q);
    int64_t nsub = n / ((int64_t)rpw * most_blocks * nw);
    nsub = nsub < 1 ? 1 : (nsub > most ? most : nsub);
    const int64_t tiles = (n + rpw * nsub - 1) / (rpw * nsub);
    const int64_t blocks = (tiles + nw - 1) / nw;
    return TilePlan{(int)nsub, (int)(blocks < most_blocks ? blocks : most_blocks)};
}

// Rows of C: stored entries a row on average, and of the longest row.
struct RowEntries {
    double mean;
    int64_t longest;
};
constexpr int kTileInFlight4 = 5, kTileInFlight8 = 4;      // gathers in flight per lane, 4- and 8-byte rows

// Whether the tile kernel is the faster one for a product over C; k_spmm_c takes the others.
// Both were measured for random graphs of 3 to 20 neighbours a row, lattices of 4 and a dense
// matrix, n = 1e3 to 1e6, rows of 4 to 128 elements (tile against k_spmm_c, us):
//  - FP64 line search: everywhere but on long rows (n = 1e6, ld = 20, 4 neighbours: 545 / 1437;
//    n = 1e3, 500 neighbours, ld = 8: 208 / 193).
//  - FP64 product: where packed groups keep more lanes busy than groups of a power of two (n = 1e6,
//    ld = 20, 4 neighbours: 0.74 of the time; ld = 16: 1.0, on a lattice of 1e5 1.1); rows of one
//    or two units (0.8 to 1.0), rows of up to three entries (C = I, n = 5e4: 0.55 to 0.8); long
//    rows not (40 neighbours: 1.06 to 1.16).
//  - Products in float: on irregular rows a row group waits for the longest of its rows, in rounds
//    of five gathers, where k_spmm_c has eight in flight (float rows, n = 1e5, ld = 24, 4 neighbours:
//    30 / 21, 12 neighbours: 51 / 29; dense: 103 / 41).  The tile is faster where every row
//    takes one round and the streams leave L2 (lattice of 1e6, ld = 20: 98 / 155), and for bf16
//    rows on up to 12 neighbours, where the weights' FP64 in every lane bounds the other (n = 1e6,
//    ld = 20, 4 neighbours: 141 / 217; without a multiplier 128 / 148).
//  - Line search in float: its epilogue gains as in FP64, its gathers lose as above (float rows,
//    n = 1e6, ld = 24: 0.8 of the time at 3 neighbours, 1.14 at 12).
template <typename TX, typename TO>
inline bool tile_pays(int epi, bool weighted, int64_t n, int Q, const RowEntries& c) {
    if (Q > 32) return false;
    int L = 1;
    while (L < Q) L <<= 1;
    const int busy = 32 / Q * Q, busy_pow2 = 32 / L * Q;   // lanes at work: packed groups, groups of L
    const bool packed = busy > busy_pow2, by_half = 2 * busy >= 3 * busy_pow2;
    const double units = (double)n * Q;
    if (std::is_same_v<arith_t<TO>, dfloat>) return true;  // bound by arithmetic (840 / 355 at n = 1e6)
    if (std::is_same_v<arith_t<TO>, double>) {
        if (epi == EPI_LS) return c.mean <= 64;
        if (c.mean > 24) return false;
        if (Q <= 2 || packed || c.mean <= 3.5) return true;
        if (Q >= 16) return units >= 9e5;
        if (Q == 4 && n < 50000) return true;
        return c.mean <= 7.5 && (c.longest > kTileInFlight4 || units >= 1.2e6);
    }
    const bool narrow = sizeof(TX) == 2;                   // bf16 rows
    if (epi == EPI_LS) {
        if (narrow) return c.mean <= (Q == 1 ? 6 : 22);
        return Q >= 2 && c.mean <= (Q >= 16 ? 14 : packed ? 10 : 6);
    }
    if (c.longest <= kTileInFlight4) {                     // each row in one round of gathers
        if (c.mean <= 3.5 && (packed || units <= 1e5 || (narrow && Q > 1))) return true;
        if (narrow) return weighted ? Q >= 2 && units >= 8e5 : Q >= 3 && units >= (packed ? 1.4e6 : 3.5e6);
        return Q >= 3 && (weighted ? units >= 1.5e6 : packed && units >= 3e6);
    }
    if (Q < 3 || units < 3e6) return false;
    if (!narrow) return weighted && by_half && c.mean <= 4.5;
    if (weighted) return c.mean <= (by_half ? 13.5 : packed ? 9.5 : 5.5);
    return packed && c.mean <= (by_half ? 9.5 : 5.5);
}

// 4 or 8 bytes of global memory to shared memory, without a register.
template <int BYTES>
__device__ __forceinline__ void stage_bytes(void* smem, const void* g) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(s), "l"(g), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void stage_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Sum of a row's Q values in shared memory by one lane, as group_sum adds the values of L >= Q lanes:
// at the last exchange the even and the odd lanes meet, at the first l and l + L/2.  The lanes past
// Q hold zeros there and cost nothing here.  In registers over the loaded values for float, whose
// rows of 32 units waited on one dependent access after another in place (ld = 128, n = 2e5: 1.3
// times the row groups' time); in place in FP64, where the registers cost more (n = 1e6, ld = 20: 597
// and 581 us).  The same additions.
template <int L, int OFF, int STEP, typename V>
__device__ __forceinline__ V row_tree_part(const V* s, int Q) {
    if constexpr (STEP >= L) {
        return s[OFF];
    } else {
        V t = row_tree_part<L, OFF, 2 * STEP>(s, Q);
        if (OFF + STEP < Q) t += row_tree_part<L, OFF + STEP, 2 * STEP>(s, Q);
        return t;
    }
}
template <typename V>
__device__ __forceinline__ V row_tree(V* s, int Q) {
    if (Q == 1) return s[0];
    if constexpr (std::is_same_v<V, double>) {
        for (int h = 1 << (31 - __clz(Q - 1)); h > 0; h >>= 1)
            for (int q = 0; q < h && q + h < Q; ++q) s[q] += s[q + h];
        return s[0];
    }
    if (Q <= 2) return row_tree_part<2, 0, 1>(s, Q);
    if (Q <= 4) return row_tree_part<4, 0, 1>(s, Q);
    if (Q <= 8) return row_tree_part<8, 0, 1>(s, Q);
    if (Q <= 16) return row_tree_part<16, 0, 1>(s, Q);
    return row_tree_part<32, 0, 1>(s, Q);
}

// out = C X (- A*_diag(v) X), EPI as in k_spmm_c (kernels.cuh); EPI_LS without a cache of z (the
// line search of a caller's own method).  Why tiles: with one row group at a time every lane of
// the group loaded the row's bounds, entries and multiplier term for itself, the row sums took
// shuffles in every lane, and the scalar terms of the line search ran with one lane of the group
// at work; in FP64 (2 lanes a cycle and SM) they cost as much as the products, and the weight of
// the diagonal constraint, formed by every lane, more than the float row's multiply-adds.  Here
//  - the bounds and per-row scalars of the tile are loaded by lane = row (coalesced), the weight
//    and the line-search scalars formed by lane = row, once per tile;
//  - the stored entries of the next tile are copied to shared memory (cp.async) while this one
//    is computed, so that a row's gathers wait on no index load;
//  - the row sums go through shared memory and are taken by lane = row.
// Element sums keep the order of the stored entries.  Measured: line search in FP64, n = 1e6,
// ld = 20, 5e6 entries: 1437 -> 545 us, 631 before the rows were sorted and a tile's sums
// fused (346 us of FP64 multiply-adds at two lanes a cycle; the FP64 pipe is 89% busy);
// double-float C R with the objective, n = 1e6, ld = 24: 840 -> 360 us; float product with a
// multiplier on a 1000 x 1000 torus, ld = 20: 146 -> 121 us with eight gathers in flight a lane and
// 3 blocks per SM, 89 us with five and 4 (four: 96 us).  The line search of the solve keeps
// k_spmm_c: its scalars are few in float, and the tile form took 318 us (24 resident warps) where
// k_spmm_c takes 218 (n = 1e6, ld = 24).
template <typename TX, typename TO, typename TR, int EPI>
__global__ void __launch_bounds__((tile_threads<TX, TO>()), kTileBlocks)
k_spmm_tile(ProbDev p, const TX* __restrict__ X, TO* __restrict__ out, int ld, int Q, int nsub,
            const double* __restrict__ v, int write_out, const TR* __restrict__ R, const double* __restrict__ y,
            double rho_arg, double* __restrict__ part, const Ctrl* gate, int ph) {
    if (gated_off(gate, ph)) return;
    using A = arith_t<TO>;
    using TV = cval_t<TX>;
    using PA = part_t<TO, TR>;
    using LS = zrow_t<TX, TR>;
    using AW = wide_t<TR, TX>;
    using AD = arith_t<TX>;
    constexpr int NW = tile_threads<TX, TO>() / 32;
    constexpr int UN = sizeof(AD) == 8 ? kTileInFlight8 : kTileInFlight4;    // gathers in flight per lane
    constexpr bool kSums = EPI == EPI_LS;
    // FP64 line search, bound by the FP64 pipe: a row group takes as many steps as the longest of
    // its rows, so the tile's rows are taken in the order of their lengths, and a tile's p1 and p2
    // are summed by the multiply-adds themselves (through one sum for the whole walk, four times the
    // additions to it, the coefficients' error grew from 1.6e-17 to 1.4e-16)
    constexpr bool kFp64Ls = EPI == EPI_LS && std::is_same_v<A, double>;
    __shared__ unsigned char s_row[NW][kFp64Ls ? 32 : 1];
    __shared__ __align__(16) int s_col[NW][2][kTileEntries];
    __shared__ __align__(16) TV s_val[NW][2][kTileEntries];
    __shared__ AD s_rd[NW][kSums ? kTileLaneRows : 1], s_dd[NW][kSums ? kTileLaneRows : 1];
    __shared__ AW s_rr[NW][kSums ? kTileLaneRows : 1];
    const TV* __restrict__ cv = cvals<TV>(p);
    constexpr int NQ = EPI == EPI_LS ? PL_N : (EPI == EPI_OBJ ? PO_N : 1);
    PA accq[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) accq[q] = PA(0);
    const LS rho = LS(rho_arg);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int rpw = 32 / Q, gw = lane / Q, lig = lane - gw * Q;
    const bool live = gw < rpw;
    const int rows = rpw * nsub;
    const int64_t ntiles = (p.n + rows - 1) / rows;
    const int64_t nwarps = (int64_t)gridDim.x * NW;
    int64_t t = (int64_t)blockIdx.x * NW + wib;

    // bounds of the lane's row of tile tt (an empty range past the tile's or the matrix's end)
    auto bounds = [&](int64_t tt, int64_t& s, int64_t& e) {
        s = e = 0;
        if (tt < ntiles) {
            const int64_t r = tt * rows + (lane < rows ? lane : rows);
            s = __ldg(p.c_rowptr + (r < p.n ? r : p.n));
            e = lane < rows && r < p.n ? __ldg(p.c_rowptr + r + 1) : s;
        }
    };
    // entries [first, last) of a tile to buffer `buf` (a longer tile is read from global memory)
    auto stage = [&](int buf, int64_t first, int64_t last) {
        if (last - first <= kTileEntries)
            for (int k = lane; k < (int)(last - first); k += 32) {
                stage_bytes<4>(&s_col[wib][buf][k], p.c_col + first + k);
                stage_bytes<sizeof(TV)>(&s_val[wib][buf][k], cv + first + k);
            }
        stage_commit();
    };
    int64_t s_nx, e_nx, first;           // bounds of the next tile's rows; first entry of this one
    bounds(t, s_nx, e_nx);
    first = __shfl_sync(0xffffffffu, s_nx, 0);
    int64_t end = __shfl_sync(0xffffffffu, e_nx, 31);
    // of the lane's row: its length, and where it starts (in the tile, when that is staged)
    int my_len = (int)(e_nx - s_nx);
    bool in_smem = end - first <= kTileEntries;
    int64_t my_at = in_smem ? s_nx - first : s_nx;
    int buf = 0;
    stage(0, first, end);
    bounds(t + nwarps, s_nx, e_nx);
    for (; t < ntiles; t += nwarps) {
        first = __shfl_sync(0xffffffffu, s_nx, 0);
        end = __shfl_sync(0xffffffffu, e_nx, 31);
        stage(buf ^ 1, first, end);
        const int len_nx = (int)(e_nx - s_nx);
        const bool smem_nx = end - first <= kTileEntries;
        const int64_t at_nx = smem_nx ? s_nx - first : s_nx;
        bounds(t + 2 * nwarps, s_nx, e_nx);
        const int64_t r0 = t * rows;
        // per-row scalars of lane = row
        const int64_t my = r0 + lane;
        const bool own = lane < rows && my < p.n;
        int kc = -1;
        A wv = A(0);
        if (p.dk != nullptr && own) {
            kc = __ldg(p.dk + my);
            if (v != nullptr && kc >= 0) wv = A(-__ldg(p.da + my) * __ldg(v + kc));
        }
        stage_wait<1>();
        __syncwarp();
        if constexpr (kFp64Ls) {
            const int mine = own ? my_len : -1;
            int rank = 0;
#pragma unroll
            for (int q = 0; q < 32; ++q) {
                const int other = __shfl_sync(0xffffffffu, mine, q);
                rank += other > mine || (other == mine && q < lane) ? 1 : 0;
            }
            s_row[wib][rank] = (unsigned char)lane;      // ranks are distinct; lanes without a row come last
            __syncwarp();
        }
        const int* sc = s_col[wib][buf];
        const TV* sv = s_val[wib][buf];
        const bool diag = v != nullptr && p.dk != nullptr;
        double t_p1 = 0.0, t_p2 = 0.0;                     // the tile's, in the FP64 line search
#pragma unroll 1
        for (int sb = 0; sb < nsub; ++sb) {
            int lr = sb * rpw + gw;                        // the group's row of the tile
            if constexpr (kFp64Ls) lr = live ? s_row[wib][lr] : 0;
            const int64_t i = r0 + lr;
            const bool act = live && lr < rows && i < p.n;
            const int src = live ? lr : 0;
            const int len = __shfl_sync(0xffffffffu, my_len, src);
            // the row's entries: in shared memory, or where they are (generic addresses)
            const int64_t at = __shfl_sync(0xffffffffu, my_at, src);
            const int* rc = in_smem ? sc + (int)at : p.c_col + at;
            const TV* rv = in_smem ? sv + (int)at : cv + at;
            A acc[4] = {A(0), A(0), A(0), A(0)};
            Unit<TX> di;
            Unit<TR> ri;
            if (act) {
                if constexpr (EPI != EPI_NONE) di.load(X + i * (int64_t)ld + lig * 4);
                if constexpr (EPI == EPI_LS) ri.load_stream(R + i * (int64_t)ld + lig * 4);
            }
            for (int k = 0; act && k < len; k += UN) {
                int j[UN];
                TV w[UN];
                Unit<TX> x[UN];
#pragma unroll
                for (int u = 0; u < UN; ++u) {
                    const bool ok = k + u < len;
                    j[u] = -1;
                    w[u] = TV(0);
                    if (ok) {
                        j[u] = rc[k + u];
                        w[u] = rv[k + u];
                    }
                }
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (j[u] >= 0) x[u].load(X + (int64_t)j[u] * ld + lig * 4);
#pragma unroll
                for (int u = 0; u < UN; ++u)
                    if (j[u] >= 0)
#pragma unroll
                        for (int e = 0; e < 4; ++e) acc[e] = fma(A(w[u]), A(x[u].v[e]), acc[e]);
            }
            if (diag) {
                const int kr = __shfl_sync(0xffffffffu, kc, src);
                const A w = shfl_idx(wv, src);
                if (act && kr >= 0) {
                    Unit<TX> xi;
                    if constexpr (EPI != EPI_NONE) xi = di;
                    else xi.load(X + i * (int64_t)ld + lig * 4);
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[e] = fma(w, A(xi.v[e]), acc[e]);
                }
            }
            const A(&o)[4] = acc;
            if (write_out && act) {
                Unit<TO> ou;
#pragma unroll
                for (int e = 0; e < 4; ++e) ou.v[e] = o[e];
                ou.store_stream(out + i * (int64_t)ld + lig * 4);
            }
            if constexpr (EPI == EPI_OBJ) {
                if (act) {
                    A d = A(0);
#pragma unroll
                    for (int e = 0; e < 4; ++e) d = fma(o[e], A(di.v[e]), d);
                    accq[PO_CRR] += PA(d);
                }
            }
            if constexpr (EPI == EPI_LS) {
                if (act) {
                    AD p2 = AD(0), rd = AD(0), dd = AD(0);
                    AW p1 = AW(0), rr = AW(0);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const AD d = AD(di.v[e]);
                        if constexpr (kFp64Ls) t_p2 = fma(AD(o[e]), d, t_p2);
                        else p2 = fma(AD(o[e]), d, p2);
                        rd = fma(AD(ri.v[e]), d, rd);
                        dd = fma(d, d, dd);
                        const AW r = AW(ri.v[e]);
                        if constexpr (kFp64Ls) t_p1 = fma(AW(o[e]), r, t_p1);
                        else p1 = fma(AW(o[e]), r, p1);
                        rr = fma(r, r, rr);
                    }
                    if constexpr (!kFp64Ls) accq[PL_P2] += p2;
                    s_rd[wib][lr * Q + lig] = rd;
                    s_dd[wib][lr * Q + lig] = dd;
                    if constexpr (!kFp64Ls) accq[PL_P1] += PA(AW(2) * p1);
                    s_rr[wib][lr * Q + lig] = rr;
                }
            }
        }
        __syncwarp();
        if constexpr (kFp64Ls) {
            accq[PL_P1] += 2.0 * t_p1;
            accq[PL_P2] += t_p2;
        }
        if constexpr (EPI == EPI_LS) {
            if (kc >= 0) {
                // (a chain of up to 32 additions would round more than the groups' tree)
                const AD t_rd = row_tree(s_rd[wib] + lane * Q, Q);
                const AD t_dd = row_tree(s_dd[wib] + lane * Q, Q);
                const AW t_rr = row_tree(s_rr[wib] + lane * Q, Q);
                LS a, z, yv;
                if constexpr (std::is_same_v<LS, double>) {
                    a = __ldg(p.da + my);
                    z = a * double(t_rr) - __ldg(p.b + kc);
                    yv = __ldg(y + kc);
                } else {
                    a = ld_scalar<LS>(p.da, p.da_df, my);
                    z = LS(dfloat(t_rr) * ld_scalar<dfloat>(p.da, p.da_df, my) - ld_scalar<dfloat>(p.b, p.b_df, kc));
                    yv = LS(__ldg(y + kc));
                }
                const LS yt = yv - rho * z;
                const LS q1 = LS(2) * a * LS(t_rd);
                const LS q2 = a * LS(t_dd);
                accq[PL_YQ1] += PA(yt * q1);
                accq[PL_YQ2] += PA(yt * q2);
                accq[PL_Q1Q1] += PA(q1 * q1);
                accq[PL_Q1Q2] += PA(q1 * q2);
                accq[PL_Q2Q2] += PA(q2 * q2);
            }
            __syncwarp();                                  // the sums have been read
        }
        my_len = len_nx;
        my_at = at_nx;
        in_smem = smem_nx;
        buf ^= 1;
    }
    stage_wait<0>();
    if constexpr (EPI != EPI_NONE) block_partials<NQ>(accq, part, (int)blockIdx.x);
}

}  // namespace lorads
