// tree.cuh -- the general stage of the parallel Riccati tree: shapes of more than 32 states,
// the tensor-core stage products, and Algorithm 6 as printed.
//
// One team owns one subproblem (chunk) of one level and walks its stages serially;
// inside a stage the lanes share the small dense products.  All per-chunk state
// (P, Psi, V, v, Q^_w) and the stage's A_t, B_t live in the workspace; Q_t and l_t
// are read from global memory inside the products.
//
//   reduce_chunk  Algorithm 4 (matrix part always; vector part when a
//                 right-hand side is given).  Non-last chunks emit the master
//                 stage (A^ = V_0^T, a^ = v_0, Q^_x = P_0, l^_x = -Psi_0, and the
//                 input part in square-root form B = R^T, Q_w = I with
//                 R^T R = Q^_w = B^); the last chunk of a level is factored with its
//                 known terminal (Algorithms 1-2) and emits the next level's
//                 terminal cost (Q^_x,p = P_0, l^_x,p = -Psi_0); the top chunk
//                 emits nothing.  reduce.cuh has it for at most 32 states.
//   down_chunk_literal  Algorithm 6 as printed (every subproblem solved again).
//
// vec.cuh has the vector passes over stored factors (rhs_chunk, down_chunk),
// resid.cuh the stage assembly and the KKT residual.
#pragma once
#include <stdint.h>
#include <type_traits>

#include "common.h"
#include "f32conv.h"
#include "reduce.cuh"
#include "stage.cuh"
#include "tc.cuh"
#include "vec.cuh"
#include "warp.cuh"
#include "wgemm.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// Shared-memory workspace of one team (every matrix slot holds up to NX x NX;
// columns and vectors 16-byte aligned for the vector loads of wgemm_tn).
template <typename T, int NX>
struct Ws {
    static constexpr int VEC = 16 / (int)sizeof(T);
    static constexpr int ld = pick_ld(NX, VEC);
    static constexpr int slot = NX * ld;
    static constexpr int nv = (NX + VEC - 1) / VEC * VEC;   // a vector's length, rounded to the 16-byte unit
    static constexpr int count = (10 * slot + 8 * nv + 8 + VEC - 1) / VEC * VEC;
    static_assert(ld % VEC == 0 && slot % VEC == 0 && nv % VEC == 0, "16-byte aligned columns and vectors");
    T *P, *V, *Qw, *A, *Tt, *B, *PB, *H, *K, *G;
    T *Psi, *v, *u, *e, *tv, *g, *k, *tmp;
    T* sc;
    MHE_DEV void carve(T* base)
    {
        T* p = base;
        P = p; p += slot; V = p; p += slot; Qw = p; p += slot; A = p; p += slot;
        Tt = p; p += slot; B = p; p += slot; PB = p; p += slot; H = p; p += slot;
        K = p; p += slot; G = p; p += slot;
        Psi = p; p += nv; v = p; p += nv; u = p; p += nv; e = p; p += nv;
        tv = p; p += nv; g = p; p += nv; k = p; p += nv; tmp = p; p += nv;
        sc = p;
    }
};

// A -> s.A, B -> s.B, a -> s.e.  FP32 blocks stored in memory (leaf and master
// stages) move in 16-byte pieces when n is a multiple of four: a column of A or
// B is n contiguous floats, 16-byte aligned (the blocks lie back to back in a
// 256-byte aligned arena).
template <typename T, int NX, int MT, int KIND>
MHE_DEV void load_AB(Ws<T, NX>& s, const StageRef<T>& st)
{
    constexpr int ld = Ws<T, NX>::ld;
    using X = Acc<T, KIND, NX, MT>;
    if constexpr (sizeof(T) == 4 && NX % 4 == 0 && ld % 4 == 0 && KIND != KIND_ARRIVAL) {
        constexpr int CA = NX * NX / 4, CB = NX * MT / 4;
        wcopy<CA + CB>(
            [&](int u) { return u < CA ? ld16g(st.A + 4 * u) : ld16g(st.B + 4 * (u - CA)); },
            [&](int u, const F4& v) {
                const int k = 4 * (u < CA ? u : u - CA);
                st16((u < CA ? s.A : s.B) + k % NX + (k / NX) * ld, v);
            });
    } else {
        wcopy<NX * NX>([&](int idx) { return X::A(st, idx % NX, idx / NX); },
                       [&](int idx, T v) { s.A[idx % NX + (idx / NX) * ld] = v; });
        wcopy<NX * MT>([&](int idx) { return X::B(st, idx % NX, idx / NX); },
                       [&](int idx, T v) { s.B[idx % NX + (idx / NX) * ld] = v; });
    }
    wcopy<NX>([&](int i) { return X::a(st, i); }, [&](int i, T v) { s.e[i] = v; });
}

// Store the R x C column-major block at src (shared memory, leading dimension
// LD) to dst (global, leading dimension R), times sgn; then tail(k) for k < ntail in the
// same step.  FP32 blocks of a multiple of four rows go in 16-byte pieces (every
// column of dst then starts 16-byte aligned, as dst does: the stored blocks are laid out
// back to back in a 256-byte aligned arena), others element by element.
template <typename T, int R, int C, int LD, class TF>
MHE_DEV void store_block(T* dst, const T* src, T sgn, int ntail, TF&& tail)
{
    if constexpr (sizeof(T) == 4 && R % 4 == 0 && LD % 4 == 0) {
        constexpr int NV = R * C / 4;
        wfor(NV + ntail, [&](int u) {
            if (u >= NV) {
                tail(u - NV);
                return;
            }
            const int i = 4 * (u % (R / 4)), j = u / (R / 4);
            float v[4];
            ld16(src + i + j * LD, v);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = sgn * v[q];
            st16(dst + i + j * R, v);
        });
    } else {
        wfor(R * C + ntail, [&](int r) {
            if (r >= R * C) {
                tail(r - R * C);
                return;
            }
            const int i = r % R, j = r / R;
            dst[r] = sgn * src[i + j * LD];
        });
    }
}

// In-place lower Cholesky of the M x M matrix Gm (leading dimension ld of the
// workspace).  Returns true when a pivot fell below piv_rel * G_jj, its
// column's diagonal before elimination (the pivot is then replaced by 1 to stay
// finite).  Lane i owns row i of the lower
// triangle: at column j lane j takes the square root, the lanes below scale
// their entry of column j and update their own row, so no two lanes write the
// same entry and a column costs two barriers.  INV stores 1 / L_jj on the
// diagonal, the form the triangular solves use: a multiply per pivot, where an FP64
// division costs as much as six FP64 products of a warp (407 against 64 cycles).
template <typename T, int NX, int M, bool INV = false>
MHE_DEV bool chol_inplace(Ws<T, NX>& s, T* Gm, double piv_rel)
{
    static_assert(M <= MHE_TEAM && M <= NX, "one lane per row");
    constexpr int ld = Ws<T, NX>::ld;
    if constexpr (M <= 32) {
        // rows in the registers of one warp, columns passed by shuffles
        static_assert(INV, "reciprocal pivots");
        team_chol<T, M>(Gm, ld, piv_rel, s.sc + 1);
        return s.sc[1] != 0;
    }
    wone([&](int) { s.sc[1] = 0; });
    for (int j = 0; j < M; ++j) {
        wone([&](int) {
            T d = Gm[j + j * ld];
            // column j's diagonal before elimination: the pivot plus the squares of row j of L
            T g0 = d;
            for (int k = 0; k < j; ++k) g0 += Gm[j + k * ld] * Gm[j + k * ld];
            if (!(d > (T)(piv_rel * (double)mabs(g0)))) { s.sc[1] = 1; d = 1; }
            const T l = msqrt(d);
            s.sc[2] = l;
            Gm[j + j * ld] = INV ? (T)1 / l : l;
        });
        const T ljj = s.sc[2];
        wlanes([&](int i) {
            if (i <= j || i >= M) return;
            const T lij = Gm[i + j * ld] / ljj;
            Gm[i + j * ld] = lij;
            s.tmp[i] = lij;
        });
        wlanes([&](int i) {
            if (i <= j || i >= M) return;
            const T lij = s.tmp[i];
            for (int c = j + 1; c <= i; ++c) Gm[i + c * ld] -= lij * s.tmp[c];
        });
    }
    return s.sc[1] != 0;
}

template <typename T, int NX, int MT>
MHE_DEV bool chol_G(Ws<T, NX>& s, double piv_rel)
{
    return chol_inplace<T, NX, MT, true>(s, s.G, piv_rel);
}

// ---- blocked triangular solves with the Cholesky factor in s.G (1 / L_jj on its diagonal) ----
// Diagonal blocks of SB rows (the largest divisor of M up to 8): a column's
// solve within a block is a short chain in registers; the coupling between
// blocks is a team product (wgemm), so every lane works and no register array
// grows with M.
constexpr int solve_block(int M)
{
    int b = 1;
    for (int d = 1; d <= 8 && d <= M; ++d)
        if (M % d == 0) b = d;
    return b;
}

template <int I, int N, class F>
MHE_DEV void static_for(F&& f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>());
        static_for<I + 1, N>(f);
    }
}

// X = L^{-1} R (M rows, NC columns): rhs(i, c) gives R, put/get store and read X.
template <typename T, int NX, int M, int NC, class FR, class FG, class FP>
MHE_DEV void lower_solve(const Ws<T, NX>& s, FR&& rhs, FG&& get, FP&& put)
{
    constexpr int ld = Ws<T, NX>::ld, SB = solve_block(M), NB = M / SB;
    static_for<0, NB>([&](auto jb) {
        constexpr int J = decltype(jb)::value, R0 = J * SB;
        if constexpr (J > 0)   // rows R0.. of R minus L[R0.., 0..R0) X[0..R0)
            wgemm<T, SB, NC, R0>([&](int i, int c) { return rhs(R0 + i, c); },
                                 [&](int i, int p) { return -s.G[R0 + i + p * ld]; },
                                 [&](int p, int c) { return get(p, c); },
                                 [&](int i, int c, T v) { put(R0 + i, c, v); });
        wfor(NC, [&](int c) {
            T y[SB];
#pragma unroll
            for (int i = 0; i < SB; ++i) {
                T acc = (J > 0) ? get(R0 + i, c) : rhs(R0 + i, c);
#pragma unroll
                for (int p = 0; p < i; ++p) acc -= s.G[R0 + i + (R0 + p) * ld] * y[p];
                y[i] = acc * s.G[R0 + i + (R0 + i) * ld];
            }
#pragma unroll
            for (int i = 0; i < SB; ++i) put(R0 + i, c, y[i]);
        });
    });
}

// X = L^{-T} R: rhs(i, c) gives R, put/get store and read X.
template <typename T, int NX, int M, int NC, class FR, class FG, class FP>
MHE_DEV void upper_solve(const Ws<T, NX>& s, FR&& rhs, FG&& get, FP&& put)
{
    constexpr int ld = Ws<T, NX>::ld, SB = solve_block(M), NB = M / SB;
    static_for<0, NB>([&](auto kb) {
        constexpr int J = NB - 1 - decltype(kb)::value, R0 = J * SB, R1 = R0 + SB;
        if constexpr (J < NB - 1)   // rows R0.. of R minus L[R1.., R0..]^T X[R1..)
            wgemm<T, SB, NC, M - R1>([&](int i, int c) { return rhs(R0 + i, c); },
                                     [&](int i, int p) { return -s.G[R1 + p + (R0 + i) * ld]; },
                                     [&](int p, int c) { return get(R1 + p, c); },
                                     [&](int i, int c, T v) { put(R0 + i, c, v); });
        wfor(NC, [&](int c) {
            T y[SB];
#pragma unroll
            for (int i = SB - 1; i >= 0; --i) {
                T acc = (J < NB - 1) ? get(R0 + i, c) : rhs(R0 + i, c);
#pragma unroll
                for (int p = i + 1; p < SB; ++p) acc -= s.G[R0 + p + (R0 + i) * ld] * y[p];
                y[i] = acc * s.G[R0 + i + (R0 + i) * ld];
            }
#pragma unroll
            for (int i = 0; i < SB; ++i) put(R0 + i, c, y[i]);
        });
    });
}

// Y = L^{-1} R and (when upper) X = L^{-T} Y for pivots blocks of at most 16
// rows: one right-hand-side column per lane, held in registers through both
// substitutions (the factor read by broadcast from shared memory), so the two
// solves take one team step instead of a barrier per diagonal block.
// rhs(i, c) gives R; putY / putX store Y and X.
template <typename T, int NX, int M, int NC, class FR, class FY, class FX>
MHE_DEV void col_solves(const Ws<T, NX>& s, bool upper, FR&& rhs, FY&& putY, FX&& putX)
{
    static_assert(M <= 16, "a right-hand-side column of at most 16 rows per lane");
    constexpr int ld = Ws<T, NX>::ld;
    wfor(NC, [&](int c) {
        T y[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            T acc = rhs(i, c);
#pragma unroll
            for (int p = 0; p < i; ++p) acc -= s.G[i + p * ld] * y[p];
            y[i] = acc * s.G[i + i * ld];
            putY(i, c, y[i]);
        }
        if (upper) {
#pragma unroll
            for (int i = M - 1; i >= 0; --i) {
                T acc = y[i];
#pragma unroll
                for (int p = i + 1; p < M; ++p) acc -= s.G[p + i * ld] * y[p];
                y[i] = acc * s.G[i + i * ld];
                putX(i, c, y[i]);
            }
        }
    });
}

// ---- the stage products on the tensor cores (tcgen05, kind::tf32) -------------
//
// Tensor state of a team whose stage products run on the tensor cores: TMEM
// base address, the mbarrier the MMAs complete on and the parity of its next
// phase, a 32 KB shared-memory tile outside the workspace, and whether every
// wait so far completed within its limit.
struct TcState {
    uint32_t tbase;
    uint64_t* mbar;
    float* xbuf;
    uint32_t phase;
    int ok;
};

// Accumulator rows from TMEM; after a wait that ran out (the products may still be in
// flight) nothing is read and zeros stand in (the instance already reports the timeout).
// The condition is the same for every thread of the team, as the loads require.
MHE_DEV void tmem_pair(const TcState& t, int row, int c0, int c1, float (&v)[16], float (&w)[16])
{
    if (t.ok) {
        tc::tmem_ld16x2(t.tbase, row, c0, c1, v, w);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = w[i] = 0.f;
    }
}
MHE_DEV void tmem_one(const TcState& t, int row, int c0, float (&v)[16])
{
    if (t.ok) {
        tc::tmem_ld16(t.tbase, row, c0, v);
    } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = 0.f;
    }
}

// the team's wait for the MMAs it committed last; a wait that runs out marks the
// state failed, and no further MMA is issued
MHE_DEV void tc_team_wait(TcState& t)
{
    if (!t.ok) return;
    if (tc::team_wait(t.mbar, t.phase)) t.phase ^= 1u;
    else t.ok = 0;
}

// Both products of Algorithm 1's stage update, with [A | B] the n x (n + m)
// stage matrix and P = P_{t+1} (symmetric):
//   X^T = [A | B]^T P                 (M = 128 >= n + m rows, K = n)
//   [A | B]^T X = [[A^T P A, A^T P B], [B^T P A, B^T P B]]   (M = 128, K = n)
// then F = Q_x + A^T P A -> s.P, H = Q_xw + A^T P B -> s.H, G = Q_w + B^T P B
// -> s.G (full blocks, each entry from its own row of the product).  Every operand
// is split into TF32 hi + lo (lo = x - hi rounded to TF32 again).  The B
// operands are stored [hi; lo] (hi rows, then lo rows), so one MMA of twice the
// N gives hi*hi and hi*lo side by side, and a second adds lo*hi to the hi*lo
// half: hi*hi and the cross terms stay in separate FP32 accumulators, summed
// when read (the small terms in the large accumulator lose bits to its
// alignment, in their own they do not: a one-CTA measurement on GB300 gave a
// max relative error of 2.0e-7 of sum |a b| for K = 64, an FP32 FMA chain
// 1.8e-7, all three products in one accumulator 5.1e-7).  TMEM columns:
// [0, 2n) the two halves of X^T, [2n, 2n + 2(n+m)) those of the second product.
// Operand tiles, canonical K-major (rows of 4 x 16 B core matrices along K = n):
// [A|B]^T hi in the V and Qw slots, lo in the extra tile; [P hi; P lo] in the PB
// and H slots; [X^T hi; X^T lo] in PB..G once the first product is done.  The
// workspace slots used as tiles are free in a stage without V (the serial plan
// and the last chunk of each level).
template <int NX, int MT, int KIND>
MHE_DEV void tc_stage_products(Ws<float, NX>& s, const StageRef<float>& st, TcState& tcs)
{
    using X = Acc<float, KIND, NX, MT>;
    using W = Ws<float, NX>;
    constexpr int ld = W::ld;
    constexpr int NAB = NX + MT;
    constexpr int LBO = 128, SBO = (NX / 4) * 128;
    constexpr int TILE = 128 * NX * 4;   // bytes of a 128-row operand tile
    constexpr int C2 = 2 * NX;            // TMEM column of the second product
    static_assert(MHE_TEAM == 128 && NX > 0, "a tensor-core team is the four warps of one CTA");
    static_assert(NX % 16 == 0 && NAB % 16 == 0 && NAB <= 128, "MMA shapes M = 128, N = 2n and 2(n + m)");
    static_assert(2 * W::slot * 4 >= TILE && TILE <= 32 * 1024, "[A|B]^T tiles fit the V, Qw slots and the extra tile");
    static_assert(4 * W::slot * 4 >= 2 * NAB * NX * 4, "[X^T hi; X^T lo] fits the PB, H, K, G slots");
    static_assert(C2 + 2 * NAB <= 512, "accumulators within the 512 TMEM columns");
    char* ABh = reinterpret_cast<char*>(s.V);
    char* ABl = reinterpret_cast<char*>(tcs.xbuf);
    char* Ph = reinterpret_cast<char*>(s.PB);
    char* Pl = Ph + (NX / 8) * SBO;   // row n of the stacked tile
    char* Xh = reinterpret_cast<char*>(s.PB);
    char* Xl = Xh + (NAB / 8) * SBO;  // row n + m of the stacked tile
    auto split_store = [&](char* hi, char* lo, int off, const float (&x)[4]) {
        float h[4], l[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            h[i] = tc::tf32_hi(x[i]);
            l[i] = tc::tf32_hi(x[i] - h[i]);
        }
        st16(reinterpret_cast<float*>(hi + off), h);
        st16(reinterpret_cast<float*>(lo + off), l);
    };
    // operands: row r of [A|B]^T is column r of A or B, row r of P is its column r;
    // each lane loads four 16-byte pieces, then splits and stores them
    constexpr int UAB = NAB * (NX / 4), UP = NX * (NX / 4);
    static_assert(UAB % (4 * MHE_TEAM) == 0 && UP % (4 * MHE_TEAM) == 0, "whole batches of four pieces per lane");
    tc::lanes_publish([&](int lane) {
#pragma unroll 1
        for (int u0 = 0; u0 < UAB + UP; u0 += 4 * MHE_TEAM) {
            float x[4][4];
            int off[4];
            const bool ab = u0 < UAB;   // the same for every lane of the batch
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int u = u0 + lane + q * MHE_TEAM;
                if (ab) {
                    const int r = u % NAB, kc = u / NAB;
                    ld16((r < NX ? s.A + r * ld : s.B + (r - NX) * ld) + 4 * kc, x[q]);
                    off[q] = tc::kmaj_off(r, 4 * kc, LBO, SBO);
                } else {
                    const int v = u - UAB, r = v % NX, kc = v / NX;
                    ld16(s.P + r * ld + 4 * kc, x[q]);
                    off[q] = tc::kmaj_off(r, 4 * kc, LBO, SBO);
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) split_store(ab ? ABh : Ph, ab ? ABl : Pl, off[q], x[q]);
        }
    });
    wone([&](int) {
        if (!tcs.ok) return;
        tc::fence_after();
        constexpr uint32_t id2 = tc::idesc_tf32(128, 2 * NX), id1 = tc::idesc_tf32(128, NX);
#pragma unroll 1
        for (int k = 0; k < NX / 8; ++k) {
            const uint64_t ah = tc::sdesc(ABh + 256 * k, LBO, SBO), al = tc::sdesc(ABl + 256 * k, LBO, SBO);
            const uint64_t b = tc::sdesc(Ph + 256 * k, LBO, SBO);
            tc::mma_tf32(tcs.tbase, ah, b, id2, k > 0);     // [hi*hi | hi*lo]
            tc::mma_tf32(tcs.tbase + NX, al, b, id1, true); // + lo*hi
        }
        tc::commit(tcs.mbar);
    });
    tc_team_wait(tcs);
    // X^T (TMEM lane r = row r) -> its hi / lo rows
    tc::lanes_publish([&](int r) {
#pragma unroll 1
        for (int c = 0; c < NX; c += 16) {
            float v[16], w[16];
            tmem_pair(tcs, r, c, NX + c, v, w);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += w[i];
            if (r < NAB) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float x[4] = {v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]};
                    split_store(Xh, Xl, tc::kmaj_off(r, c + 4 * q, LBO, SBO), x);
                }
            }
        }
    });
    wone([&](int) {
        if (!tcs.ok) return;
        tc::fence_after();
        constexpr uint32_t id2 = tc::idesc_tf32(128, 2 * NAB), id1 = tc::idesc_tf32(128, NAB);
#pragma unroll 1
        for (int k = 0; k < NX / 8; ++k) {
            const uint64_t ah = tc::sdesc(ABh + 256 * k, LBO, SBO), al = tc::sdesc(ABl + 256 * k, LBO, SBO);
            const uint64_t b = tc::sdesc(Xh + 256 * k, LBO, SBO);
            tc::mma_tf32(tcs.tbase + C2, ah, b, id2, k > 0);
            tc::mma_tf32(tcs.tbase + C2 + NAB, al, b, id1, true);
        }
        tc::commit(tcs.mbar);
    });
    tc_team_wait(tcs);
    // row r of the second product: F and H rows (r < n), G rows (n <= r < n + m),
    // whole rows; the stage Hessian's entries of the next 16 columns are
    // requested before this block's accumulator loads and stores.  F is written
    // in full (the update P = F - Y^T Y that follows reads one triangle and
    // writes P symmetric), G in full (its Cholesky reads the lower triangle).
    wlanes([&](int r) {
        const bool row = r < NAB;   // whole warps
        float qv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, i) : 0.f;
#pragma unroll 1
        for (int c = 0; c < NAB; c += 16) {
            float v[16], w[16];
            tmem_pair(tcs, r, C2 + c, C2 + NAB + c, v, w);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = qv[i] + (v[i] + w[i]);
            if (c + 16 < NAB) {
#pragma unroll
                for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, c + 16 + i) : 0.f;
            }
            // c is a multiple of 16 and n, n + m are too: a block lies in one of P, H or G
            if (r < NX) {
                float* dst = c < NX ? s.P + r + c * ld : s.H + r + (c - NX) * ld;
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i * ld] = v[i];
            } else if (row && c >= NX) {
                float* dst = s.G + (r - NX) + (c - NX) * ld;
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i * ld] = v[i];
            }
        }
        tc::fence_before();
    });
}

// The same two products with BF16 operands (kind::f16, K = 16 per instruction).
// A BF16 value keeps 7 fraction bits, so each operand is split three ways,
// x = hi + mid + lo (each the BF16 rounding of what the previous pieces leave),
// and each product sums the six terms down to 2^-16 relative in three FP32
// accumulators by magnitude: hi*hi; hi*mid + mid*hi; hi*lo + mid*mid + lo*hi.
// The B operands are stored [hi; mid; lo]: per K step, A_hi x [B_hi; B_mid]
// (N = 2k) gives hi*hi | hi*mid, A_hi x B_lo gives hi*lo, A_mid x [B_hi; B_mid]
// adds mid*hi | mid*mid, A_lo x B_hi adds lo*hi.  TMEM columns [0, 3n) hold the
// three parts of X^T, then (after they are read) [0, 3(n+m)) those of the second
// product.  Tiles (16-bit, canonical K-major): [A|B]^T hi and mid in the V, Qw
// slots, lo in the extra tile; [P hi; mid; lo] in PB and H; [X^T hi; mid; lo]
// in PB..G.
template <int NX, int MT, int KIND>
MHE_DEV void tc_stage_products_bf16(Ws<float, NX>& s, const StageRef<float>& st, TcState& tcs)
{
    using X = Acc<float, KIND, NX, MT>;
    using W = Ws<float, NX>;
    constexpr int ld = W::ld;
    constexpr int NAB = NX + MT;
    constexpr int LBO = 128, SBO = (NX / 8) * 128;
    constexpr int TILE = 128 * NX * 2;   // bytes of a 128-row 16-bit operand tile
    static_assert(MHE_TEAM == 128 && NX > 0, "a tensor-core team is the four warps of one CTA");
    static_assert(NX % 16 == 0 && NAB % 16 == 0 && 2 * NAB <= 256, "MMA shapes M = 128, N <= 256");
    static_assert(2 * W::slot * 4 >= 2 * TILE && TILE <= 32 * 1024, "[A|B]^T tiles fit the V, Qw slots and the extra tile");
    static_assert(2 * W::slot * 4 >= 3 * NX * NX * 2 && 4 * W::slot * 4 >= 3 * NAB * NX * 2, "stacked B tiles fit");
    static_assert(3 * NAB <= 512, "accumulators within the 512 TMEM columns");
    char* Ah = reinterpret_cast<char*>(s.V);
    char* Am = Ah + TILE;
    char* Al = reinterpret_cast<char*>(tcs.xbuf);
    char* Pt = reinterpret_cast<char*>(s.PB);   // [P hi; P mid; P lo], NX rows each
    char* Xt = reinterpret_cast<char*>(s.PB);   // [X^T hi; mid; lo], NAB rows each
    // 8 values of one row along K -> three 16-byte rows of core matrices
    auto split_store8 = [&](char* h, char* m, char* l, const float (&x)[8]) {
        unsigned short ph[8], pm[8], pl[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            ph[i] = tc::bf16_bits(x[i]);
            const float r1 = x[i] - tc::bf16_val(ph[i]);
            pm[i] = tc::bf16_bits(r1);
            pl[i] = tc::bf16_bits(r1 - tc::bf16_val(pm[i]));
        }
        auto store = [](char* dst, const unsigned short (&v)[8]) {
            const unsigned w[4] = {v[0] | (unsigned)v[1] << 16, v[2] | (unsigned)v[3] << 16,
                                   v[4] | (unsigned)v[5] << 16, v[6] | (unsigned)v[7] << 16};
            st16u(dst, w);
        };
        store(h, ph);
        store(m, pm);
        store(l, pl);
    };
    constexpr int UAB = NAB * (NX / 8), UP = NX * (NX / 8);   // 8-value pieces
    tc::lanes_publish([&](int lane) {
#pragma unroll 1
        for (int u = lane; u < UAB + UP; u += MHE_TEAM) {
            float x[8];
            if (u < UAB) {
                const int r = u % NAB, kc = u / NAB;
                const float* src = (r < NX ? s.A + r * ld : s.B + (r - NX) * ld) + 8 * kc;
                float a[4], b[4];
                ld16(src, a);
                ld16(src + 4, b);
#pragma unroll
                for (int i = 0; i < 4; ++i) { x[i] = a[i]; x[4 + i] = b[i]; }
                const int off = tc::kmaj_off16(r, 8 * kc, LBO, SBO);
                split_store8(Ah + off, Am + off, Al + off, x);
            } else {
                const int v = u - UAB, r = v % NX, kc = v / NX;
                float a[4], b[4];
                ld16(s.P + r * ld + 8 * kc, a);
                ld16(s.P + r * ld + 8 * kc + 4, b);
#pragma unroll
                for (int i = 0; i < 4; ++i) { x[i] = a[i]; x[4 + i] = b[i]; }
                split_store8(Pt + tc::kmaj_off16(r, 8 * kc, LBO, SBO), Pt + tc::kmaj_off16(NX + r, 8 * kc, LBO, SBO),
                             Pt + tc::kmaj_off16(2 * NX + r, 8 * kc, LBO, SBO), x);
            }
        }
    });
    // issue the four MMAs per K step of one product: A [128 x K] against the stacked
    // B rows [0, 2N) (hi, mid) and [2N, 3N) (lo), into TMEM columns [0, 3N)
    auto issue = [&](const char* Bt, int N, uint32_t idN, uint32_t id2N) {
#pragma unroll 1
        for (int k = 0; k < NX / 16; ++k) {
            const uint64_t ah = tc::sdesc(Ah + 256 * k, LBO, SBO), am = tc::sdesc(Am + 256 * k, LBO, SBO),
                           al = tc::sdesc(Al + 256 * k, LBO, SBO);
            const uint64_t bhm = tc::sdesc(Bt + 256 * k, LBO, SBO);
            const uint64_t blo = tc::sdesc(Bt + (2 * N / 8) * SBO + 256 * k, LBO, SBO);
            tc::mma_bf16(tcs.tbase, ah, bhm, id2N, k > 0);          // hi*hi | hi*mid
            tc::mma_bf16(tcs.tbase + 2 * N, ah, blo, idN, k > 0);   // hi*lo
            tc::mma_bf16(tcs.tbase + N, am, bhm, id2N, true);       // + mid*hi | mid*mid
            tc::mma_bf16(tcs.tbase + 2 * N, al, bhm, idN, true);    // + lo*hi
        }
        tc::commit(tcs.mbar);
    };
    wone([&](int) {
        if (!tcs.ok) return;
        tc::fence_after();
        issue(Pt, NX, tc::idesc_bf16(128, NX), tc::idesc_bf16(128, 2 * NX));
    });
    tc_team_wait(tcs);
    // X^T (TMEM lane r = row r) -> its three stacked rows
    tc::lanes_publish([&](int r) {
#pragma unroll 1
        for (int c = 0; c < NX; c += 16) {
            float v[16], w[16], z[16];
            tmem_pair(tcs, r, c, NX + c, v, w);
            tmem_one(tcs, r, 2 * NX + c, z);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] += w[i] + z[i];
            if (r < NAB) {
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    float x[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) x[i] = v[8 * q + i];
                    split_store8(Xt + tc::kmaj_off16(r, c + 8 * q, LBO, SBO),
                                 Xt + tc::kmaj_off16(NAB + r, c + 8 * q, LBO, SBO),
                                 Xt + tc::kmaj_off16(2 * NAB + r, c + 8 * q, LBO, SBO), x);
                }
            }
        }
    });
    wone([&](int) {
        if (!tcs.ok) return;
        tc::fence_after();
        issue(Xt, NAB, tc::idesc_bf16(128, NAB), tc::idesc_bf16(128, 2 * NAB));
    });
    tc_team_wait(tcs);
    // row r of the second product (see tc_stage_products)
    wlanes([&](int r) {
        const bool row = r < NAB;   // whole warps
        float qv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, i) : 0.f;
#pragma unroll 1
        for (int c = 0; c < NAB; c += 16) {
            float v[16], w[16], z[16];
            tmem_pair(tcs, r, c, NAB + c, v, w);
            tmem_one(tcs, r, 2 * NAB + c, z);
#pragma unroll
            for (int i = 0; i < 16; ++i) v[i] = qv[i] + (v[i] + (w[i] + z[i]));
            if (c + 16 < NAB) {
#pragma unroll
                for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, c + 16 + i) : 0.f;
            }
            if (r < NX) {
                float* dst = c < NX ? s.P + r + c * ld : s.H + r + (c - NX) * ld;
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i * ld] = v[i];
            } else if (row && c >= NX) {
                float* dst = s.G + (r - NX) + (c - NX) * ld;
#pragma unroll
                for (int i = 0; i < 16; ++i) dst[i * ld] = v[i];
            }
        }
        tc::fence_before();
    });
}

// One backward stage of Algorithm 4 (or Algorithms 1-2 when want_v is false).
// On entry s.P = P_{t+1}, s.Psi = Psi_{t+1}, s.V = V_{t+1}, s.v = v_{t+1},
// s.Qw = partial Q^_w.  Stores P_{t+1}, the factor of G_{t+1} (store_factor), K_{t+1}, k_{t+1},
// L_{t+1} (nullptr skips a store).  Returns true on a failed pivot.
template <typename T, int NX, int MT, int KIND, int TC = 0>
MHE_DEV bool reduce_step(Ws<T, NX>& s, const StageRef<T>& st, T* Pout, T* Lgout, T* Kout,
                         T* kout, T* Lout, bool want_v, double piv_rel, TcState* tcs = nullptr)
{
    constexpr int ld = Ws<T, NX>::ld;
    using X = Acc<T, KIND, NX, MT>;
    if (Pout) store_block<T, NX, NX, ld>(Pout, s.P, (T)1, 0, [](int) {});
    load_AB<T, NX, MT, KIND>(s, st);
    bool on_tc = false;
    if constexpr (TC != 0) on_tc = !want_v;
    if (on_tc) {
        // u = Psi - P a, then F, G, H on the tensor cores (P is overwritten by F)
        wgemm_tn<T, NX, 1, NX, ld, 0>([&](int i, int) { return s.Psi[i]; }, s.P, s.e, (T)-1,
                                      [&](int i, int, T v) { s.u[i] = v; });
        if constexpr (TC == 1) tc_stage_products<NX, MT, KIND>(s, st, *tcs);
        if constexpr (TC == 2) tc_stage_products_bf16<NX, MT, KIND>(s, st, *tcs);
    } else {
        // P A -> Tt,  P B -> PB,  u = Psi - P a
        // (P is symmetric: row i of P is column i, read along the inner dimension)
        wgemm_tn<T, NX, NX, NX, ld, ld>([&](int, int) { return (T)0; }, s.P, s.A, (T)1,
                                        [&](int i, int j, T v) { s.Tt[i + j * ld] = v; });
        wgemm_tn<T, NX, MT, NX, ld, ld>([&](int, int) { return (T)0; }, s.P, s.B, (T)1,
                                        [&](int i, int j, T v) { s.PB[i + j * ld] = v; });
        wgemm_tn<T, NX, 1, NX, ld, 0>([&](int i, int) { return s.Psi[i]; }, s.P, s.e, (T)-1,
                                      [&](int i, int, T v) { s.u[i] = v; });
        // F = Q_x + A^T P A -> P (symmetric),  G = Q_w + B^T P B (symmetric),  H = Q_xw + A^T P B
        wgemm_tn<T, NX, NX, NX, ld, ld, true>([&](int i, int j) { return X::qx(st, i, j); }, s.A, s.Tt, (T)1,
                                              [&](int i, int j, T v) { s.P[i + j * ld] = v; s.P[j + i * ld] = v; });
        wgemm_tn<T, MT, MT, NX, ld, ld, true>([&](int i, int j) { return X::qw(st, i, j); }, s.B, s.PB, (T)1,
                                              [&](int i, int j, T v) { s.G[i + j * ld] = v; s.G[j + i * ld] = v; });
        wgemm_tn<T, NX, MT, NX, ld, ld>([&](int i, int j) { return X::qxw(st, i, j); }, s.A, s.PB, (T)1,
                                        [&](int i, int j, T v) { s.H[i + j * ld] = v; });
    }
    // g = B^T u - l_w,  tv = A^T u
    wgemm_tn<T, MT, 1, NX, ld, 0>([&](int j, int) { return -X::lw(st, j); }, s.B, s.u, (T)1,
                                  [&](int j, int, T v) { s.g[j] = v; });
    wgemm_tn<T, NX, 1, NX, ld, 0>([&](int, int) { return (T)0; }, s.A, s.u, (T)1,
                                  [&](int i, int, T v) { s.tv[i] = v; });
    const bool bad = chol_G<T, NX, MT>(s, piv_rel);
    // [Y | y] = Lg^{-1} [H^T | g] (Y in PB, y in tmp);  K = -Lg^{-T} Y (s.K),  k = Lg^{-T} y = G^{-1} g (s.k)
    {
        auto rhsY = [&](int i, int c) -> T { return c < NX ? s.H[c + i * ld] : s.g[i]; };
        auto getY = [&](int i, int c) -> T { return c < NX ? s.PB[i + c * ld] : s.tmp[i]; };
        auto putY = [&](int i, int c, T v) {
            if (c < NX) s.PB[i + c * ld] = v;
            else s.tmp[i] = v;
        };
        auto getX = [&](int i, int c) -> T { return c < NX ? -s.K[i + c * ld] : s.k[i]; };
        auto putX = [&](int i, int c, T v) {
            if (c < NX) s.K[i + c * ld] = -v;
            else s.k[i] = v;
        };
        if constexpr (MT <= 16) {
            col_solves<T, NX, MT, NX + 1>(s, true, rhsY, putY, putX);
        } else {
            lower_solve<T, NX, MT, NX + 1>(s, rhsY, getY, putY);
            upper_solve<T, NX, MT, NX + 1>(s, getY, getX, putX);
        }
        if (Kout)
            store_block<T, MT, NX, ld>(Kout, s.K, (T)1, kout ? MT : 0, [&](int j) { kout[j] = s.k[j]; });
        else if (kout)
            wfor(MT, [&](int j) { kout[j] = s.k[j]; });
    }
    // P -= Y^T Y (symmetric),  Psi = A^T u - l_x + K^T g,  store the factor (no barrier: G keeps until the next stage)
    wgemm_tn<T, NX, NX, MT, ld, ld, true>([&](int i, int j) { return s.P[i + j * ld]; }, s.PB, s.PB, (T)-1,
                                          [&](int i, int j, T v) { s.P[i + j * ld] = v; s.P[j + i * ld] = v; });
    wgemm_tn<T, NX, 1, MT, ld, 0>([&](int i, int) { return s.tv[i] - X::lx(st, i); }, s.K, s.g, (T)1,
                                  [&](int i, int, T v) { s.Psi[i] = v; });
    if (Lgout) store_factor<T, MT, ld>(Lgout, s.G);
    if (!want_v) return bad;
    // e = a + B k
    wgemm<T, NX, 1, MT>([&](int i, int) { return s.e[i]; }, [&](int i, int j) { return s.B[i + j * ld]; },
                        [&](int j, int) { return s.k[j]; }, [&](int i, int, T v) { s.tv[i] = v; });
    // v += V^T e;  BV = B^T V (in H)
    wgemm_tn<T, NX, 1, NX, ld, 0>([&](int i, int) { return s.v[i]; }, s.V, s.tv, (T)1,
                                  [&](int i, int, T v) { s.v[i] = v; });
    wgemm_tn<T, MT, NX, NX, ld, ld>([&](int, int) { return (T)0; }, s.B, s.V, (T)1,
                                    [&](int j, int c, T v) { s.H[j + c * ld] = v; });
    // Z = Lg^{-1} BV (in PB),  L = -Lg^{-T} Z (formed in Tt, stored)
    {
        auto rhsZ = [&](int i, int c) -> T { return s.H[i + c * ld]; };
        auto getZ = [&](int i, int c) -> T { return s.PB[i + c * ld]; };
        auto putZ = [&](int i, int c, T v) { s.PB[i + c * ld] = v; };
        auto getL = [&](int i, int c) -> T { return s.Tt[i + c * ld]; };
        auto putL = [&](int i, int c, T v) { s.Tt[i + c * ld] = v; };
        lower_solve<T, NX, MT, NX>(s, rhsZ, getZ, putZ);
        if (Lout) upper_solve<T, NX, MT, NX>(s, getZ, getL, putL);
        if (Lout) store_block<T, MT, NX, ld>(Lout, s.Tt, (T)-1, 0, [](int) {});
    }
    // V_new = A^T V + K^T BV -> Tt;  Q^_w += Z^T Z (symmetric)
    wgemm_tn<T, NX, NX, NX, ld, ld>([&](int, int) { return (T)0; }, s.A, s.V, (T)1,
                                    [&](int i, int j, T v) { s.Tt[i + j * ld] = v; });
    wgemm_tn<T, NX, NX, MT, ld, ld>([&](int i, int j) { return s.Tt[i + j * ld]; }, s.K, s.H, (T)1,
                                    [&](int i, int j, T v) { s.Tt[i + j * ld] = v; });
    wgemm_tn<T, NX, NX, MT, ld, ld, true>([&](int i, int j) { return s.Qw[i + j * ld]; }, s.PB, s.PB, (T)1,
                                          [&](int i, int j, T v) { s.Qw[i + j * ld] = v; s.Qw[j + i * ld] = v; });
    T* tmp = s.V;
    s.V = s.Tt;
    s.Tt = tmp;
    return bad;
}

// ---- Algorithm 4 over one chunk ----------------------------------------------

template <typename T, int NX, int NW, bool UPPER, int TC = 0>
MHE_DEV void reduce_chunk(const LevelArgs<T>& a, int ci, T* smem, TcState* tcs = nullptr)
{
    constexpr int ld = Ws<T, NX>::ld;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    const bool last = (cd.flags & CH_LAST) != 0;
    const bool top = (cd.flags & CH_TOP) != 0;
    Ws<T, NX> s;
    s.carve(smem);
    const T* QN = UPPER ? a.QNk + (long long)b * NX * NX : nullptr;   // level 0: Q_{x,N} = 0
    const T* lN = UPPER ? (a.lNk ? a.lNk + (long long)b * NX : nullptr)
                        : (a.lN ? a.lN + (long long)b * NX : nullptr);
    wfor(NX * NX, [&](int idx) {
        int i = idx % NX, j = idx / NX;
        s.P[i + j * ld] = (last && QN) ? QN[idx] : (T)0;
        s.V[i + j * ld] = (T)(i == j ? 1 : 0);
        s.Qw[i + j * ld] = 0;
        if (idx < NX) {
            s.Psi[idx] = (last && lN) ? -lN[idx] : (T)0;
            s.v[idx] = 0;
        }
    });
    int bad_t = -1;
    if (!UPPER) prefetch_leaf<T, NX, NW>(a, b, cd.t0 + cd.len - 1);
    for (int tt = cd.len - 1; tt >= 0; --tt) {
        const int t = cd.t0 + tt;
        const long long g = cd.g0 + tt;
        if (!UPPER && tt > 0) prefetch_leaf<T, NX, NW>(a, b, t - 1);   // the next stage of the sweep
        bool bad;
        if (UPPER) {
            bad = reduce_step<T, NX, NX, KIND_UPPER, TC>(
                s, Addr<T, NX, NW>::upper(a, g), a.store_P ? a.Pst + g * NX * NX : nullptr,
                a.Lgst + g * NX * NX, a.Kst + g * NX * NX, a.kst + g * NX,
                last ? nullptr : a.Lst + g * NX * NX, !last, a.piv_rel, tcs);
        } else if (t == 0) {
            bad = reduce_step<T, NX, NX, KIND_ARRIVAL, TC>(
                s, Addr<T, NX, NW>::arrival(a, b), a.store_P ? a.Pst0 + (long long)b * NX * NX : nullptr,
                a.Lgst0 + (long long)b * NX * NX, a.Kst0 + (long long)b * NX * NX, a.kst0 + (long long)b * NX,
                last ? nullptr : a.Lst0 + (long long)b * NX * NX, !last, a.piv_rel, tcs);
        } else {
            bad = reduce_step<T, NX, NW, KIND_LEAF, TC>(
                s, Addr<T, NX, NW>::leaf(a, b, t), a.store_P ? a.Pst + g * NX * NX : nullptr,
                a.Lgst + g * NW * NW, a.Kst + g * NW * NX, a.kst + g * NW,
                last ? nullptr : a.Lst + g * NW * NX, !last, a.piv_rel, tcs);
        }
        if (bad && bad_t < 0) bad_t = t;
    }
    if (!last) {
        // Theorem 1 with the basis U_1 = S^T R^{-1} (orthonormal in the Q-bar^{-1}
        // inner product): Q^_w = I and B^ = R^T, where R^T R is the T-form
        // Q^_w = S Qbar^{-1} S^T accumulated above.  Same master problem with
        // w^' = R w^; its G = I + R P R^T is far better conditioned than
        // B^ + B^ P B^.
        // With leaf chunks too short for a full-rank Q^_w (leaf_len * nw < nx: S^T rank
        // deficient, Section IV-B's remark on a singular G^), the factorisation pivots and
        // stops at the numerical rank r, Pi^T Q^_w Pi = L L^T with L n x r, and the
        // master stage is B = Pi L padded with zero columns to width n, Q_w = I: a
        // basis U_1 = S^T Pi [L_11^{-T}; 0] of range(S^T) in Theorem 1; the down pass
        // recovers w^ = Pi [L_11^{-T} w^'_{1..r}; 0].
        int rank = NX;
        if (a.piv_up) {
            rank = chol_pivoted<T, NX, ld>(s.Qw, a.piv_rank, s.u, s.sc);
            if (rank == 0 && bad_t < 0) bad_t = cd.t0;
        } else if (chol_inplace<T, NX, NX>(s, s.Qw, a.piv_rel) && bad_t < 0) {
            bad_t = cd.t0;
        }
        // the master stage's data at cd.parent (and at its mirror cd.parent2, when given)
        const int copies = cd.parent2 >= 0 ? 2 : 1;
        wfor(copies * NX * NX, [&](int u) {
            const long long gp = u < NX * NX ? cd.parent : cd.parent2;
            const int idx = u % (NX * NX);
            int i = idx % NX, j = idx / NX;
            a.Ah_up[gp * NX * NX + idx] = s.V[j + i * ld];
            if (a.piv_up) {   // row Pi(i) of B is row i of L (columns j >= r are zero)
                const int pi = (int)s.u[i];
                a.Bh_up[gp * NX * NX + pi + j * NX] = (i >= j && j < rank) ? s.Qw[i + j * ld] : (T)0;
                if (j == 0) a.piv_up[gp * (NX + 1) + i] = pi;
                if (idx == 0) a.piv_up[gp * (NX + 1) + NX] = rank;
            } else {
                a.Bh_up[gp * NX * NX + idx] = i >= j ? s.Qw[i + j * ld] : (T)0;
            }
            a.Qxh_up[gp * NX * NX + idx] = s.P[i + j * ld];
            if (idx < NX) {
                a.ah_up[gp * NX + idx] = s.v[idx];
                a.lxh_up[gp * NX + idx] = -s.Psi[idx];
            }
        });
    } else if (!top) {
        wfor(NX * NX, [&](int idx) {
            a.QN_up[(long long)b * NX * NX + idx] = s.P[idx % NX + (idx / NX) * ld];
            if (idx < NX) a.lN_up[(long long)b * NX + idx] = -s.Psi[idx];
        });
    }
    if constexpr (TC != 0) {
        // a tensor-core wait that ran out: the products after it are not valid
        if (!tcs->ok) wone([&](int) { record_error(a.status, a.where, b, -7, a.level, ci, cd.t0); });
    }
    if (bad_t >= 0) wone([&](int) { record_error(a.status, a.where, b, -3, a.level, ci, bad_t); });
}

// ---- Algorithm 6 as printed: every subproblem solved again --------------------
//
// Level by level from the top, subproblem i of level k is solved with
// Algorithms 1-3 from its parent's data: the backward recursion (Algorithms 1-2,
// no V) over its stages from the cost-to-go of the level above at its end state,
// P^_{i+1} and Psi^_{i+1} (the last subproblem from the level's own terminal),
// then the forward recursion (Algorithm 3) from x^_i: w_t = K_t x_t + k_t,
// x_{t+1} = A_t x_t + B_t w_t + a_t, lambda_t = P_t x_t - Psi_t.  The re-solve
// writes P_t, Psi_t at every state of the subproblem for the level below.  The
// result equals the back-substitution of down_chunk; its cost is a second
// factorisation per stage.  The feedback K_t, k_t goes to scratch arrays: the
// reduction's stored factors stay as they are for later right-hand sides.
template <typename T, int NX, int NW, bool UPPER>
MHE_DEV void down_chunk_literal(const LevelArgs<T>& a, int ci, T* smem)
{
    constexpr int ld = Ws<T, NX>::ld;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    if (a.active && !a.active[b]) return;
    const bool last = (cd.flags & CH_LAST) != 0;
    const bool top = (cd.flags & CH_TOP) != 0;
    Ws<T, NX> s;
    s.carve(smem);
    const LevelInst li = a.li[b];
    const int t1 = cd.t0 + cd.len;
    // the terminal of the re-solve: the parent's cost-to-go at the chunk's end state, or
    // the level's own terminal (Q_{x,N} = 0, l_N at level 0; the level's QN, lN above)
    const T* QN = UPPER ? a.QNk + (long long)b * NX * NX : nullptr;
    const T* lN = UPPER ? (a.lNk ? a.lNk + (long long)b * NX : nullptr) : (a.lN ? a.lN + (long long)b * NX : nullptr);
    const T* Pt = last ? QN : a.Pd_up + (cd.px + 1) * NX * NX;
    const T* Pst = last ? nullptr : a.Psid_up + (cd.px + 1) * NX;
    // the end state's P, Psi are written here only for the level's last chunk; the end
    // state of any other chunk is the next chunk's first, which writes them
    T* Pd = a.Pd + (li.gx + t1) * NX * NX;
    T* Psd = a.Psid + (li.gx + t1) * NX;
    wfor(NX * NX, [&](int idx) {
        const int i = idx % NX, j = idx / NX;
        const T v = Pt ? Pt[idx] : (T)0;
        s.P[i + j * ld] = v;
        if (last) Pd[idx] = v;
        if (idx < NX) {
            const T ps = last ? (lN ? -lN[idx] : (T)0) : Pst[idx];
            s.Psi[idx] = ps;
            if (last) Psd[idx] = ps;
        }
    });
    int bad_t = -1;
    // backward: Algorithms 1-2 over the chunk; P_{t+1} of each stage to Pd at state t + 1
    for (int tt = cd.len - 1; tt >= 0; --tt) {
        const int t = cd.t0 + tt;
        const long long g = cd.g0 + tt;
        T* Po = a.Pd + (li.gx + t + 1) * NX * NX;
        if (tt < cd.len - 1)
            wfor(NX, [&](int i) { a.Psid[(li.gx + t + 1) * NX + i] = s.Psi[i]; });
        bool bad;
        if (UPPER) {
            bad = reduce_step<T, NX, NX, KIND_UPPER>(s, Addr<T, NX, NW>::upper(a, g), tt < cd.len - 1 ? Po : nullptr,
                                                     nullptr, a.Kalt + g * NX * NX, a.kalt + g * NX, nullptr, false,
                                                     a.piv_rel);
        } else if (t == 0) {
            bad = reduce_step<T, NX, NX, KIND_ARRIVAL>(s, Addr<T, NX, NW>::arrival(a, b),
                                                       tt < cd.len - 1 ? Po : nullptr, nullptr,
                                                       a.Kalt0 + (long long)b * NX * NX, a.kalt0 + (long long)b * NX,
                                                       nullptr, false, a.piv_rel);
        } else {
            bad = reduce_step<T, NX, NW, KIND_LEAF>(s, Addr<T, NX, NW>::leaf(a, b, t), tt < cd.len - 1 ? Po : nullptr,
                                                    nullptr, a.Kalt + g * NW * NX, a.kalt + g * NW, nullptr, false,
                                                    a.piv_rel);
        }
        if (bad && bad_t < 0) bad_t = t;
    }
    // P_0, Psi_0 of the chunk at its first state
    wfor(NX * NX, [&](int idx) {
        a.Pd[(li.gx + cd.t0) * NX * NX + idx] = s.P[idx % NX + (idx / NX) * ld];
        if (idx < NX) a.Psid[(li.gx + cd.t0) * NX + idx] = s.Psi[idx];
    });
    if (bad_t >= 0) wone([&](int) { record_error(a.status, a.where, b, -3, a.level, ci, bad_t); });
    // forward: Algorithm 3 from x^_i (the top: x~0)
    auto xo = [&](int t) -> T* { return a.xd + (li.gx + t) * NX; };
    auto lo = [&](int t) -> T* { return a.ld + (li.gx + t) * NX; };
    auto wo = [&](int t) -> T* {
        if (UPPER) return a.wd + (li.gs + t) * NX;
        return a.wd + a.w_off[b] + (t == 0 ? 0 : NX + (long long)(t - 1) * NW);
    };
    auto zxo = [&](int t) -> double* { return a.zx ? a.zx + (li.gx + t) * NX : nullptr; };
    auto zlo = [&](int t) -> double* { return a.zl ? a.zl + (li.gx + t) * NX : nullptr; };
    auto zwo = [&](int t) -> double* {
        return a.zw ? a.zw + a.w_off[b] + (t == 0 ? 0 : NX + (long long)(t - 1) * NW) : nullptr;
    };
    wfor(NX, [&](int i) { s.e[i] = top ? a.x0[(long long)b * NX + i] : a.xd_up[cd.px * NX + i]; });
    float dzm = 0.f;
    // lambda_t = P_t x_t - Psi_t (Algorithm 3), x_t and lambda_t written, z accumulated at level 0
    auto state_out = [&](int t) {
        const T* P = a.Pd + (li.gx + t) * NX * NX;
        const T* Ps = a.Psid + (li.gx + t) * NX;
        wfor(NX, [&](int i) {
            T acc = -Ps[i];
#pragma unroll
            for (int j = 0; j < NX; ++j) acc += P[i + j * NX] * s.e[j];
            xo(t)[i] = s.e[i];
            lo(t)[i] = acc;
            if (a.zx) {
                zxo(t)[i] += f64_of(s.e[i]);
                zlo(t)[i] += f64_of(acc);
                dzm = fmaxf(dzm, fmaxf(absf_of(s.e[i]), absf_of(acc)));
            }
        });
    };
    for (int tt = 0; tt < cd.len; ++tt) {
        const int t = cd.t0 + tt;
        const long long g = cd.g0 + tt;
        state_out(t);
        T* w = wo(t);
        double* zw = zwo(t);
        auto fwd = [&](const StageRef<T>& st, const T* K, const T* k, auto kind_tag, auto mt_tag) {
            constexpr int KIND = decltype(kind_tag)::value, MT = decltype(mt_tag)::value;
            using X = Acc<T, KIND, NX, MT>;
            wfor(MT, [&](int j) {
                T acc = k[j];
#pragma unroll
                for (int i = 0; i < NX; ++i) acc += K[j + i * MT] * s.e[i];
                s.tmp[j] = acc;
                w[j] = acc;
                if (zw) {
                    zw[j] += f64_of(acc);
                    dzm = fmaxf(dzm, absf_of(acc));
                }
            });
            wfor(NX, [&](int i) {
                T acc = X::a(st, i);
#pragma unroll
                for (int j = 0; j < NX; ++j) acc += X::A(st, i, j) * s.e[j];
#pragma unroll
                for (int j = 0; j < MT; ++j) acc += X::B(st, i, j) * s.tmp[j];
                s.u[i] = acc;
            });
            wfor(NX, [&](int i) { s.e[i] = s.u[i]; });
        };
        if (UPPER)
            fwd(Addr<T, NX, NW>::upper(a, g), a.Kalt + g * NX * NX, a.kalt + g * NX,
                std::integral_constant<int, KIND_UPPER>(), std::integral_constant<int, NX>());
        else if (t == 0)
            fwd(Addr<T, NX, NW>::arrival(a, b), a.Kalt0 + (long long)b * NX * NX, a.kalt0 + (long long)b * NX,
                std::integral_constant<int, KIND_ARRIVAL>(), std::integral_constant<int, NX>());
        else
            fwd(Addr<T, NX, NW>::leaf(a, b, t), a.Kalt + g * NW * NX, a.kalt + g * NW,
                std::integral_constant<int, KIND_LEAF>(), std::integral_constant<int, NW>());
    }
    if (last) state_out(t1);   // the level's final state (the next chunk writes the others' end states)
    if (a.zx && a.dznorm) wlanes([&](int) {
        if (dzm > 0.f) atomicMax(a.dznorm + b, __float_as_uint(dzm));
    });
}

MHE_TEAM_NS_END
}  // namespace mhe
