// reduce.cuh -- Algorithm 4's matrix recursion over one chunk, for shapes whose pivot
// blocks fit the lanes of a warp (nx <= 32).
//
// One backward stage from P, Psi, V, v at t+1 (W = [A | B], both from shared memory):
//   1. X = [P A | P B | P a],  BV = B^T V,  V^T a;  u = Psi - P a
//   2. W^T P W + Q, whose blocks are F, H and G (symmetric: one triangle);  W^T u
//   3. G = L L^T, and beside it A^T V
//   4. per column, in registers: Y = L^{-1} H^T, y = L^{-1} g, Z = L^{-1} BV and from them
//      K = -L^{-T} Y, k = L^{-T} y, L_t = -L^{-T} Z, straight to global memory, as L's columns scaled by 1 / L_jj
//   5. P <- F - Y^T Y,  V <- A^T V - Y^T Z,  Q^_w += Z^T Z,
//      Psi <- A^T u - l_x - Y^T y,  v <- v + V^T a + Z^T y
// (K^T B^T V = -Y^T Z and V^T (a + B k) = V^T a + Z^T y, so K, k and L_t are only stored.)
// Six team barriers a stage (one after each step, one once the stage's copies have landed), and in FP64 one more
// per pivot column of G while a single team factors it; the next stage's A, B and a are copied asynchronously from
// the end of step 3 on.
//
// What bounds it.  FP64: an instruction of a warp costs 64 cycles of its SM quarter whatever
// its number of active lanes, so the products are dealt to lanes entry by entry (no
// lane tile whose corners stick out) and only one triangle of the symmetric ones is formed.
// FP32: the latency of the chain at ten to twenty warps an SM, and the shared-memory loads of the products (register
// tiles, TM + TN loads of 16 bytes per 2 TM TN packed FMAs; ncu at nx = 24: 35% issue, 54% of the shared-memory
// wavefronts).
//
// Measured (GB300), before (some twenty barriers a stage, both triangles, divisions, blocks loaded as the
// stage came) and after: FP64 nx = 20, 16384 stages in chunks of 32, 3.75 -> 2.04 ms, with four warps a chunk; a
// master level of it 0.92 -> 0.22 ms; FP32 leaf level nx = 6, 1.10M stages, 1.02 -> 0.55 ms; nx = 12, 1.05M stages, 2.65 -> 2.04
// ms; nx = 24, 535k stages, 6.44 -> 5.85 ms.
#pragma once
#include <type_traits>

#include "common.h"
#include "stage.cuh"
#include "vec.cuh"
#include "warp.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// (i <= j) number k of the n(n+1)/2 pairs, the triangle folded into a rectangle
template <int N>
MHE_DEV void pair_of(int k, int& i, int& j)
{
    constexpr int C = N % 2 == 0 ? N + 1 : N;
    const int r = k / C, c = k % C;
    if constexpr (N % 2 == 0) {
        i = c > r ? r : N - 1 - r;
        j = c > r ? c - 1 : N - 1 - c;
    } else {
        i = c >= r ? r : N - r;
        j = c >= r ? c : N - 1 - c;
    }
}

// lane tile of a product with M x N outputs on LN lanes: the one with the least work, rounds x (FMAs + loads);
// FP64 loads cost next to nothing beside the FMAs
template <typename T>
constexpr int prod_tile(int M, int N, int LN, bool sym)
{
    int best = 1 * 64 + 1;
    long long cost = 1LL << 60;
    for (int tm = 1; tm <= 6; ++tm)
        for (int tn = 1; tn <= 6; ++tn) {
            if (sym && tm != tn) continue;
            if (tm * tn > (sizeof(T) == 8 ? 4 : 25)) continue;
            const int bm = (M + tm - 1) / tm, bn = (N + tn - 1) / tn;
            const int tasks = sym ? bm * (bm + 1) / 2 : bm * bn;
            const int rounds = (tasks + LN - 1) / LN;
            const long long c = (long long)rounds * (100 * tm * tn + (sizeof(T) == 8 ? 2 : 70) * (tm + tn)) + 60;
            if (c < cost) { cost = c; best = tm * 64 + tn; }
        }
    return best;
}

MHE_DEV void ldp(const float* p, F2 (&v)[2])
{
    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
    v[0] = q.x;
    v[1] = q.y;
}
MHE_DEV void ldp(const float* p, F2 (&v)[1]) { v[0] = *reinterpret_cast<const F2*>(p); }

// out(i, j, sum_p A[p + i LDA] B[p + j LDB] , q) for i < M, j < N (SYM: the pairs of a symmetric result, each
// once, in either order), on the lanes L0 .. L0 + LN - 1 of the team, no barrier.
// pre(i, j) is loaded before the sum and handed to out.  Both operands are read by columns in vectors.
template <typename T, int M, int N, int K, int LDA, int LDB, bool SYM, int L0, int LN, class FP, class FO>
MHE_DEV void prod(const T* A, const T* B, FP&& pre, FO&& out)
{
    constexpr int tile = prod_tile<T>(M, N, LN, SYM), TM = tile / 64, TN = tile % 64;
    constexpr int BM = (M + TM - 1) / TM, BN = (N + TN - 1) / TN;
    constexpr int TASKS = SYM ? BM * (BM + 1) / 2 : BM * BN;
    constexpr int VK = vec_of<T>(K), VA = LDA % VK == 0 && LDB % VK == 0 ? VK : 1;
    const int lane = lane_id() - L0;
    if (lane < 0 || lane >= LN) return;
#pragma unroll 1
    for (int k = lane; k < TASKS; k += LN) {
        int bi, bj;
        if constexpr (SYM) pair_of<BM>(k, bi, bj);
        else { bi = k % BM; bj = k / BM; }
        // rows bi + BM r and columns bj + BN c: neighbouring lanes read columns one leading dimension apart
        const T *ap[TM], *bp[TN];
#pragma unroll
        for (int r = 0; r < TM; ++r) ap[r] = A + (M % TM == 0 || bi + BM * r < M ? bi + BM * r : M - 1) * LDA;
#pragma unroll
        for (int c = 0; c < TN; ++c) bp[c] = B + (N % TN == 0 || bj + BN * c < N ? bj + BN * c : N - 1) * LDB;
        using V = decltype(pre(0, 0));
        V pv[TM][TN];
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c) {
                const int i = bi + BM * r, j = bj + BN * c;
                if ((M % TM == 0 || i < M) && (N % TN == 0 || j < N)) pv[r][c] = pre(i, j);
            }
        T acc[TM][TN];
        if constexpr (sizeof(T) == 4 && VA >= 2) {
            // the even and the odd terms side by side: pairs as they lie in memory, half the instructions
            F2 s[TM][TN];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) s[r][c] = 0ULL;
#pragma unroll(TM * TN >= 9 ? 3 : 6)
            for (int p = 0; p < K; p += VA) {
                F2 av[TM][VA / 2], bv[TN][VA / 2];
#pragma unroll
                for (int r = 0; r < TM; ++r) ldp(ap[r] + p, av[r]);
#pragma unroll
                for (int c = 0; c < TN; ++c) ldp(bp[c] + p, bv[c]);
#pragma unroll
                for (int q = 0; q < VA / 2; ++q)
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int c = 0; c < TN; ++c) s[r][c] = fma2(av[r][q], bv[c][q], s[r][c]);
            }
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const float2 v = unpack2(s[r][c]);
                    acc[r][c] = v.x + v.y;
                }
        } else {
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) acc[r][c] = (T)0;
#pragma unroll(sizeof(T) == 8 ? K / VA : (TM * TN >= 9 ? 3 : 6))
            for (int p = 0; p < K; p += VA) {
                T av[TM][VA], bv[TN][VA];
#pragma unroll
                for (int r = 0; r < TM; ++r) ldv(ap[r] + p, av[r]);
#pragma unroll
                for (int c = 0; c < TN; ++c) ldv(bp[c] + p, bv[c]);
#pragma unroll
                for (int q = 0; q < VA; ++q)
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int c = 0; c < TN; ++c) acc[r][c] += av[r][q] * bv[c][q];
            }
        }
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c) {
                const int i = bi + BM * r, j = bj + BN * c;
                if (SYM && r > c && bi == bj) continue;   // the mirror of (c, r)
                if ((M % TM == 0 || i < M) && (N % TN == 0 || j < N)) out(i, j, acc[r][c], pv[r][c]);
            }
    }
}
struct None {};

// Offsets (elements) of one team's workspace.  Every matrix block by columns, leading dimension ld (columns of n
// entries) or lm (columns of MT entries).
template <typename T, int NX, int MT, bool ARRIVAL>
struct RedSlots {
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int ld = pick_ld(NX, vec_of<T>(NX)), lm = pick_ld(MT, vec_of<T>(MT));
    static constexpr int n2 = round_to(ld * NX, V);
    // kept from stage to stage: P, Q^_w, and V and X alternating in two slots; X = [P A | P B | u] is
    // n + MT + 1 columns, so both slots hold that many
    static constexpr int oP = 0, oQw = n2, oV0 = 2 * n2;
    static constexpr int xslot = n2 + round_to(ld * (MT + 1), V);
    static constexpr int oS = oV0 + 2 * xslot;
    // W = [A | B | a]; [Y | y] and Z; G (columns), its factor by rows
    static constexpr int oW = oS, oY = oW + (ARRIVAL ? 0 : round_to(ld * (NX + MT + 1), V)),
                         oZ = oY + round_to(lm * (NX + 1), V), oG = oZ + round_to(lm * NX, V),
                         oR = oG + round_to(lm * MT, V), end = oR + round_to(lm * MT, V);
};
template <typename T, int NX, int NW, bool UPPER>
struct RedWs {
    static constexpr int V = 16 / (int)sizeof(T), nv = round_to(NX, V);
    using S = RedSlots<T, NX, UPPER ? NX : NW, false>;
    // the arrival stage (input width n, A = B = I): [Y | y], Z and G from S::oS on, G's factor in the slot of X
    static constexpr int lm0 = pick_ld(NX, vec_of<T>(NX));
    static constexpr int a_end = S::oS + round_to(lm0 * (NX + 1), V) + 2 * round_to(lm0 * NX, V);
    static constexpr int vec = UPPER ? S::end : max_int(S::end, a_end);
    static constexpr int count = vec + 5 * nv + round_to(8, V);   // Psi, v, t, va, thr; flags
};

// G = L L^T for the M x M block at G (by columns, leading dimension LD, both triangles or the lower one given).
// On return the lower triangle holds L with 1 / L_jj on the diagonal, and R the same by rows (leading dimension
// LD).  A pivot not above piv_rel times its column's diagonal before elimination is replaced by 1 and
// reported in *flag.  The lanes below LN work (whole warps or the whole team); barriers among them only.
// FP32: one row per lane in registers, columns passed by shuffles.  FP64: every lane takes entries of the
// trailing triangle; a column costs one reciprocal (computed by every lane at once) and one barrier, and
// the square roots of all pivots are taken together at the end.
template <int LN>
MHE_DEV void sub_sync()
{
    if constexpr (LN == MHE_TEAM) wsync();
    else __syncwarp();
}

template <typename T, int M, int LD, int LN>
MHE_DEV void factor_block(T* G, T* R, T* thr, double piv_rel, T* flag)
{
    const int lane = lane_id();
    if constexpr (sizeof(T) == 4) {
        constexpr int CW = LN < 32 ? LN : 32;
        static_assert(M <= CW, "one row per lane of one warp");
        if (lane < CW) {
            const unsigned mask =
                CW == 32 ? 0xffffffffu : (((1u << CW) - 1u) << ((threadIdx.x & 31) & ~(CW - 1)));
            T g[M];
#pragma unroll
            for (int c = 0; c < M; ++c) g[c] = (lane < M && c <= lane) ? G[lane + c * LD] : (T)0;
            const T thr_i = lane < M ? (T)(piv_rel * (double)mabs(G[lane + lane * LD])) : (T)0;
            int bad = 0;
#pragma unroll
            for (int j = 0; j < M; ++j) {
                T d = __shfl_sync(mask, g[j], j, CW);
                const T th = __shfl_sync(mask, thr_i, j, CW);
                if (!(d > th)) {
                    bad = 1;
                    d = (T)1;
                }
                const T inv = mrsqrt(d);
                const T lij = g[j] * inv;
                const T lv = lane > j ? lij : (T)0;
                if (lane == j) g[j] = inv;
                if (lane > j) g[j] = lij;
#pragma unroll
                for (int c = j + 1; c < M; ++c) g[c] -= lv * __shfl_sync(mask, lv, c, CW);
            }
            if (lane < M) {
#pragma unroll
                for (int c = 0; c < M; ++c)
                    if (c <= lane) {
                        G[lane + c * LD] = g[c];
                        R[c + lane * LD] = g[c];
                    }
            }
            if (lane == 0) *flag = (T)bad;
        }
    } else {
        for (int i = lane; i < M; i += LN) thr[i] = (T)(piv_rel * (double)mabs(G[i + i * LD]));
        if (lane == 0) *flag = (T)0;
        sub_sync<LN>();
#pragma unroll 1
        for (int j = 0; j + 1 < M; ++j) {
            const T d = G[j + j * LD];
            const T r = (T)1 / (d > thr[j] ? d : (T)1);
            const int rem = M - 1 - j, cnt = rem * (rem + 1) / 2;
            const T* gj = G + j * LD;
            for (int k = lane; k < cnt; k += LN) {
                // entry (i >= c) of the trailing triangle: row by row, rows j + 1 .. M - 1
                int i = (int)((sqrtf(8.0f * (float)k + 1.0f) - 1.0f) * 0.5f);
                i += (i + 1) * (i + 2) / 2 <= k;
                i -= i * (i + 1) / 2 > k;
                const int c = j + 1 + k - i * (i + 1) / 2;
                i += j + 1;
                G[i + c * LD] -= (gj[i] * r) * gj[c];
            }
            sub_sync<LN>();
        }
        // the pivots' square roots together, then every column scaled
        for (int j = lane; j < M; j += LN) {
            const T d = G[j + j * LD];
            const bool ok = d > thr[j];
            if (!ok) *flag = (T)1;
            thr[j] = mrsqrt(ok ? d : (T)1);
        }
        sub_sync<LN>();
        for (int k = lane; k < M * M; k += LN) {
            const int i = k % M, j = k / M;
            if (i >= j) {
                const T l = i == j ? thr[j] : G[i + j * LD] * thr[j];
                G[i + j * LD] = l;
                R[j + i * LD] = l;
            }
        }
    }
}

// Rank-revealing (pivoted) Cholesky of the symmetric NX x NX matrix Gm (both
// triangles held): at step j the largest remaining diagonal is brought to (j, j)
// by a symmetric row and column swap; the factorisation stops at the first step
// whose largest remaining diagonal is at or below rank_rel * max diag, and that
// step is the numerical rank r.  On return Pi^T Gm_in Pi = L L^T restricted to
// r columns: L (lower trapezoidal, NX x r) in Gm's lower part, the pivot order
// Pi in permv (as values of T), and r is returned.  sc: five entries of scratch.
template <typename T, int NX, int ld>
MHE_DEV int chol_pivoted(T* Gm, double rank_rel, T* permv, T* sc)
{
    wone([&](int) {
        T mx = 0;
        for (int i = 0; i < NX; ++i) {
            mx = mmax(mx, mabs(Gm[i + i * ld]));
            permv[i] = (T)i;
        }
        sc[0] = (T)(rank_rel * (double)mx);
        sc[3] = (T)NX;
    });
    for (int j = 0; j < NX; ++j) {
        wone([&](int) {
            int p = j;
            T best = Gm[j + j * ld];
            for (int i = j + 1; i < NX; ++i)
                if (Gm[i + i * ld] > best) { best = Gm[i + i * ld]; p = i; }
            sc[4] = (T)p;
            if (!(best > sc[0])) sc[3] = (T)j;   // the rank: nothing above the threshold remains
        });
        if ((int)sc[3] == j) break;   // the same value for every lane (read after the barrier)
        const int p = (int)sc[4];
        if (p != j) {
            wfor(NX, [&](int q) {
                const T t = Gm[j + q * ld];
                Gm[j + q * ld] = Gm[p + q * ld];
                Gm[p + q * ld] = t;
            });
            wfor(NX, [&](int q) {
                const T t = Gm[q + j * ld];
                Gm[q + j * ld] = Gm[q + p * ld];
                Gm[q + p * ld] = t;
            });
            wone([&](int) {
                const T t = permv[j];
                permv[j] = permv[p];
                permv[p] = t;
            });
        }
        wone([&](int) {
            const T l = msqrt(Gm[j + j * ld]);
            Gm[j + j * ld] = l;
            sc[2] = l;
        });
        const T ljj = sc[2];
        wfor(NX, [&](int i) {
            if (i > j) Gm[i + j * ld] /= ljj;
        });
        // the trailing block, both triangles (the next pivot search and swaps read them)
        const int rem = NX - j - 1;
        wfor(rem * rem, [&](int u) {
            const int i = j + 1 + u % rem, c = j + 1 + u / rem;
            Gm[i + c * ld] -= Gm[i + j * ld] * Gm[c + j * ld];
        });
    }
    return (int)sc[3];
}

// The factor L in G (columns LD apart, 1 / L_jj on the diagonal) to dst as the vector passes want it, columns MT apart:
// L D^{-1/2}, D = diag(L_jj^2), below the diagonal and 1 / D_j on it; whatever lies above goes with it
template <typename T, int MT, int LD>
MHE_DEV void store_factor(T* dst, const T* G)
{
    if constexpr (sizeof(T) == 4 && MT % 4 == 0 && LD % 4 == 0) {
        each<MT * MT / 4>([&](int u) {
            const int i = 4 * (u % (MT / 4)), j = u / (MT / 4);
            const float d = G[j + j * LD];
            float v[4];
            ld16(G + i + j * LD, v);
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] *= d;
            st16(dst + 4 * u, v);
        });
    } else {
        each<MT * MT>([&](int r) {
            const int j = r / MT;
            dst[r] = G[r % MT + j * LD] * G[j + j * LD];
        });
    }
}

// Step 4: one column per lane (or per pair of lanes, H = 2, each holding every other row) through both
// substitutions.  Columns 0 .. n-1: H^T -> Y, K; n: g -> y, k; then BV -> Z, L_t.
template <typename T, int NX, int MT, int LM, int H>
MHE_DEV void solve_columns(T* Y, T* Z, const T* G, const T* R, bool want_v, T* Kout, T* kout, T* Lout)
{
    constexpr int MH = (MT + H - 1) / H, VK = vec_of<T>(MT);
    static_assert(MT % VK == 0 && LM % VK == 0, "whole vectors of a column");
    const int nc = NX + 1 + (want_v ? NX : 0);
    const int half = H == 1 ? 0 : (lane_id() & 1);
    const unsigned mask = H == 1 ? 0u : 0xffffffffu;
    (void)mask;
#pragma unroll 1
    for (int c0 = 0; c0 < nc; c0 += MHE_TEAM / H) {
        const int c = c0 + lane_id() / H;
        const bool on = c < nc;
        const bool zc = c > NX;
        T* col = !on ? nullptr : (zc ? Z + (c - NX - 1) * LM : Y + c * LM);
        T y[MH];
        if constexpr (H == 1) {
            if (!on) continue;
#pragma unroll
            for (int i = 0; i < MT; ++i) y[i] = col[i];
#pragma unroll
            for (int i = 0; i < MT; ++i) {
                T a[2] = {y[i], (T)0};
#pragma unroll
                for (int p = 0; p < i; p += VK) {
                    T l[VK];
                    ldv(R + i * LM + p, l);
#pragma unroll
                    for (int q = 0; q < VK; ++q)
                        if (p + q < i) a[q & 1] -= l[q] * y[p + q];
                }
                y[i] = (a[0] + a[1]) * R[i + i * LM];
            }
#pragma unroll
            for (int i = 0; i < MT; ++i) col[i] = y[i];
            T* dst = zc ? (Lout ? Lout + (c - NX - 1) * MT : nullptr) : (c < NX ? Kout + c * MT : kout);
            if (!dst) continue;
#pragma unroll
            for (int i = MT - 1; i >= 0; --i) {
                T a[2] = {y[i], (T)0};
#pragma unroll
                for (int p = (i + 1) / VK * VK; p < MT; p += VK) {
                    T l[VK];
                    ldv(G + i * LM + p, l);
#pragma unroll
                    for (int q = 0; q < VK; ++q)
                        if (p + q > i) a[q & 1] -= l[q] * y[p + q];
                }
                y[i] = (a[0] + a[1]) * G[i + i * LM];
            }
#pragma unroll
            for (int i = 0; i < MT; ++i) dst[i] = c == NX ? y[i] : -y[i];
        } else {
            // rows half, half + 2, ..: as each entry is finished its holder passes it on
#pragma unroll
            for (int q = 0; q < MH; ++q) {
                const int i = 2 * q + half;
                y[q] = on && i < MT ? col[i] : (T)0;
            }
#pragma unroll
            for (int p = 0; p < MT; ++p) {
                const T f = __shfl_sync(mask, y[p / 2] * R[p + p * LM], p & 1, 2);
#pragma unroll
                for (int q = p / 2; q < MH; ++q) {
                    const int i = 2 * q + half;
                    if (i > p && i < MT) y[q] -= G[i + p * LM] * f;
                    else if (i == p) y[q] = f;
                }
            }
#pragma unroll
            for (int q = 0; q < MH; ++q) {
                const int i = 2 * q + half;
                if (on && i < MT) col[i] = y[q];
            }
#pragma unroll
            for (int p = MT - 1; p >= 0; --p) {
                const T f = __shfl_sync(mask, y[p / 2] * R[p + p * LM], p & 1, 2);
#pragma unroll
                for (int q = 0; q <= p / 2; ++q) {
                    const int i = 2 * q + half;
                    if (i < p) y[q] -= R[i + p * LM] * f;
                    else if (i == p) y[q] = f;
                }
            }
            T* dst = !on ? nullptr : (zc ? (Lout ? Lout + (c - NX - 1) * MT : nullptr) : (c < NX ? Kout + c * MT : kout));
#pragma unroll
            for (int q = 0; q < MH; ++q) {
                const int i = 2 * q + half;
                if (dst && i < MT) dst[i] = c == NX ? y[q] : -y[q];
            }
        }
    }
}

// the stage's A, B and a, asynchronously into W = [A | B | a]
template <typename T, int NX, int MT, int KIND>
MHE_DEV void load_stage(T* W, const StageRef<T>& st)
{
    using S = RedSlots<T, NX, MT, false>;
    constexpr int ld = S::ld;
    constexpr int aB = piece_of(ld * NX * (int)sizeof(T)), aa = piece_of(ld * (NX + MT) * (int)sizeof(T));
    async_block<T, NX, NX, ld>(W, st.A);
    async_block<T, NX, MT, ld, NX, aB>(W + ld * NX, st.B);
    async_vec<T, NX, aa>(W + ld * (NX + MT), st.a);
}

// Workspace pointers of a chunk's sweep
template <typename T>
struct RedPtr {
    T *P, *Qw, *V, *X, *W, *Y, *Z, *G, *R, *Psi, *v, *t, *va, *thr, *flag;
};

// One backward stage (see above).  want_v: V, v and Q^_w are carried and L_t stored.  after3() runs once A, B
// and a are no longer needed.  Returns true on a failed pivot.
template <typename T, int NX, int MT, int KIND, class FN>
MHE_DEV bool reduce_stage(RedPtr<T>& s, const StageRef<T>& st, T* Pout, T* Lgout, T* Kout, T* kout, T* Lout,
                          bool want_v, double piv_rel, FN&& after3)
{
    constexpr bool ARR = KIND == KIND_ARRIVAL;
    using S = RedSlots<T, NX, MT, ARR>;
    using X = Acc<T, KIND, NX, MT>;
    constexpr int ld = S::ld, lm = S::lm, TL = MHE_TEAM;
    constexpr bool wide = TL >= 64;   // several warps: the first factors while the others form A^T V
    auto none = [](int, int) { return None(); };
    if (Pout) {
        if constexpr (sizeof(T) == 4 && NX % 4 == 0) {
            each<NX * NX / 4>([&](int u) {
                const int i = 4 * (u % (NX / 4)), j = u / (NX / 4);
                st16(Pout + 4 * u, ld16g(s.P + i + j * ld));
            });
        } else {
            each<NX * NX>([&](int r) { Pout[r] = s.P[r % NX + (r / NX) * ld]; });
        }
    }
    // 1. X = [P A | P B], u = Psi - P a; BV -> Z, V^T a -> va
    if constexpr (ARR) {   // A = B = I, a = st.a (or zero)
        each<NX>([&](int i) {
            T acc = s.Psi[i];
            if (st.a) {
#pragma unroll 4
                for (int p = 0; p < NX; ++p) acc -= s.P[p + i * ld] * st.a[p];
            }
            s.t[i] = acc;
            s.Y[NX * lm + i] = acc - X::lw(st, i);
            if (want_v) {
                T d = (T)0;
                if (st.a) {
#pragma unroll 4
                    for (int p = 0; p < NX; ++p) d += s.V[p + i * ld] * st.a[p];
                }
                s.va[i] = d;
            }
        });
        each<NX * NX>([&](int r) {
            const int i = r % NX, j = r / NX;
            const T p = s.P[i + j * ld];
            s.Y[i + j * lm] = p;
            s.G[i + j * lm] = p + st.Qw0[r];
            if (want_v) s.Z[i + j * lm] = s.V[i + j * ld];
        });
        wsync();
        factor_block<T, NX, lm, TL>(s.G, s.R, s.thr, piv_rel, s.flag);
        wsync();
    } else {
        T* u = s.X + ld * (NX + MT);
        prod<T, NX, NX + MT + 1, NX, ld, ld, false, 0, TL>(s.P, s.W, none, [&](int i, int j, T v, None) {
            s.X[i + j * ld] = j < NX + MT ? v : s.Psi[i] - v;
        });
        if (want_v)
            prod<T, NX, MT + 1, NX, ld, ld, false, 0, TL>(s.V, s.W + ld * NX, none, [&](int c, int q, T v, None) {
                if (q < MT) s.Z[q + c * lm] = v;
                else s.va[c] = v;
            });
        wsync();
        // 2. the blocks of W^T P W + Q:  F -> P,  H^T -> Y,  G;  A^T u -> t,  g = B^T u - l_w -> Y's last column
        if constexpr (sizeof(T) == 8 || NX < 16) {   // all blocks dealt out together: the fewest rounds
            prod<T, NX + MT, NX + MT, NX, ld, ld, true, 0, TL>(
                s.W, s.X, [&](int i, int j) -> T { return i <= j ? X::q(st, i, j) : X::q(st, j, i); },
                [&](int i, int j, T v, T q) {
                    v += q;
                    if (i > j) {
                        const int k = i;
                        i = j;
                        j = k;
                    }
                    if (j < NX) {
                        s.P[i + j * ld] = v;
                        s.P[j + i * ld] = v;
                    } else if (i < NX) {
                        s.Y[(j - NX) + i * lm] = v;
                    } else {
                        s.G[(j - NX) + (i - NX) * lm] = v;
                    }
                });
        } else {
            prod<T, NX, NX, NX, ld, ld, true, 0, TL>(
                s.W, s.X, [&](int i, int j) -> T { return X::qx(st, i, j); },
                [&](int i, int j, T v, T q) { s.P[i + j * ld] = s.P[j + i * ld] = v + q; });
            prod<T, NX, MT, NX, ld, ld, false, 0, TL>(
                s.W, s.X + ld * NX, [&](int i, int j) -> T { return X::qxw(st, i, j); },
                [&](int i, int j, T v, T q) { s.Y[j + i * lm] = v + q; });
            prod<T, MT, MT, NX, ld, ld, true, 0, TL>(
                s.W + ld * NX, s.X + ld * NX, [&](int i, int j) -> T { return X::qw(st, i, j); },
                [&](int i, int j, T v, T q) { s.G[i + j * lm] = s.G[j + i * lm] = v + q; });
        }
        each<NX + MT>([&](int i) {
            const T d = coldot<NX>(s.W + i * ld, u, (T)0);
            if (i < NX) s.t[i] = d;
            else s.Y[NX * lm + i - NX] = d - X::lw(st, i - NX);
        });
        wsync();
        // 3. the factor of G, and A^T V -> X (P A is done with)
        auto av = [&](int i, int j, T v, None) { s.X[i + j * ld] = v; };
        if constexpr (wide) {
            if (lane_id() < 32) factor_block<T, MT, lm, 32>(s.G, s.R, s.thr, piv_rel, s.flag);
            else if (want_v) prod<T, NX, NX, NX, ld, ld, false, 32, TL - 32>(s.W, s.V, none, av);
        } else {
            if (want_v) prod<T, NX, NX, NX, ld, ld, false, 0, TL>(s.W, s.V, none, av);
            factor_block<T, MT, lm, TL>(s.G, s.R, s.thr, piv_rel, s.flag);
        }
        wsync();
        after3();
    }
    const bool bad = *s.flag != (T)0;
    // 4.
    constexpr int H = sizeof(T) == 8 && TL >= 128 ? 2 : 1;
    if (Lgout) store_factor<T, MT, lm>(Lgout, s.G);
    solve_columns<T, NX, MT, lm, H>(s.Y, s.Z, s.G, s.R, want_v, Kout, kout, Lout);
    wsync();
    // 5. (the arrival stage: A^T V = V, F = P)
    const T* y = s.Y + NX * lm;
    prod<T, NX, NX, MT, lm, lm, true, 0, TL>(s.Y, s.Y, none, [&](int i, int j, T v, None) {
        const T p = s.P[i + j * ld] - v;
        s.P[i + j * ld] = p;
        s.P[j + i * ld] = p;
    });
    if (want_v) {
        T* Vo = ARR ? s.V : s.X;
        prod<T, NX, NX, MT, lm, lm, false, 0, TL>(s.Y, s.Z, none,
                                                  [&](int i, int j, T v, None) { Vo[i + j * ld] -= v; });
        prod<T, NX, NX, MT, lm, lm, true, 0, TL>(s.Z, s.Z, none, [&](int i, int j, T v, None) {
            const T q = s.Qw[i + j * ld] + v;
            s.Qw[i + j * ld] = q;
            s.Qw[j + i * ld] = q;
        });
    }
    each<NX>([&](int i) {
        s.Psi[i] = s.t[i] - X::lx(st, i) - coldot<MT>(s.Y + i * lm, y, (T)0);
        if (want_v) s.v[i] += coldot<MT>(s.Z + i * lm, y, s.va[i]);
    });
    wsync();
    if (want_v && !ARR) {
        T* x = s.V;
        s.V = s.X;
        s.X = x;
    }
    return bad;
}

// Algorithm 4 over one chunk
template <typename T, int NX, int NW, bool UPPER>
MHE_DEV void reduce_chunk_small(const LevelArgs<T>& a, int ci, T* smem)
{
    using WS = RedWs<T, NX, NW, UPPER>;
    using S = typename WS::S;
    constexpr int MT = UPPER ? NX : NW, ld = S::ld;
    constexpr int KIND = UPPER ? KIND_UPPER : KIND_LEAF;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    const bool last = (cd.flags & CH_LAST) != 0;
    const bool top = (cd.flags & CH_TOP) != 0;
    const long long si = UPPER ? 0 : a.in_off[b] - 1, sr = UPPER ? 0 : a.rhs_off[b] - 1;
    RedPtr<T> s;
    s.P = smem + S::oP; s.Qw = smem + S::oQw; s.V = smem + S::oV0; s.X = smem + S::oV0 + S::xslot;
    s.W = smem + S::oW; s.Y = smem + S::oY; s.Z = smem + S::oZ; s.G = smem + S::oG; s.R = smem + S::oR;
    T* vec = smem + WS::vec;
    s.Psi = vec; s.v = vec + WS::nv; s.t = vec + 2 * WS::nv; s.va = vec + 3 * WS::nv; s.thr = vec + 4 * WS::nv;
    s.flag = vec + 5 * WS::nv;
    const T* QN = UPPER ? a.QNk + (long long)b * NX * NX : nullptr;   // level 0: Q_{x,N} = 0
    const T* lN = UPPER ? (a.lNk ? a.lNk + (long long)b * NX : nullptr)
                        : (a.lN ? a.lN + (long long)b * NX : nullptr);
    auto ref = [&](int tt) {
        return UPPER ? Addr<T, NX, NW>::upper(a, cd.g0 + tt)
                     : Addr<T, NX, NW>::leaf_at(a, b, si + cd.t0 + tt, sr + cd.t0 + tt);
    };
    auto load = [&](int tt) {   // A, B, a of stage tt into W; the arrival stage has none
        if (tt >= 0 && (UPPER || cd.t0 + tt > 0)) {
            const StageRef<T> st = ref(tt);
            load_stage<T, NX, MT, KIND>(s.W, st);
            // the part of Q the products add, into L2
            if constexpr (UPPER) prefetch_l2(st.Qx, (int)sizeof(T) * NX * NX);
            else prefetch_l2(st.Q, (int)sizeof(T) * (NX + NW) * (NX + NW));
        }
        cp_commit();
    };
    load(cd.len - 1);
    each<NX * NX>([&](int idx) {
        const int i = idx % NX, j = idx / NX;
        s.P[i + j * ld] = (last && QN) ? QN[idx] : (T)0;
        s.V[i + j * ld] = (T)(i == j ? 1 : 0);
        s.Qw[i + j * ld] = (T)0;
        if (idx < NX) {
            s.Psi[idx] = (last && lN) ? -lN[idx] : (T)0;
            s.v[idx] = (T)0;
        }
    });
    int bad_t = -1;
#pragma unroll 1
    for (int tt = cd.len - 1; tt >= 0; --tt) {
        const int t = cd.t0 + tt;
        const long long g = cd.g0 + tt;
        cp_wait<0>();
        wsync();
        bool bad;
        if (!UPPER && t == 0) {
            // the widths of this stage's blocks are n: they lie over the other stages' scratch
            constexpr int n2 = round_to(WS::lm0 * NX, WS::V);
            RedPtr<T> r = s;
            r.Y = smem + S::oS;
            r.Z = r.Y + round_to(WS::lm0 * (NX + 1), WS::V);
            r.G = r.Z + n2;
            r.R = s.X;
            bad = reduce_stage<T, NX, NX, KIND_ARRIVAL>(
                r, Addr<T, NX, NW>::arrival(a, b), a.store_P ? a.Pst0 + (long long)b * NX * NX : nullptr,
                a.Lgst0 ? a.Lgst0 + (long long)b * NX * NX : nullptr, a.Kst0 + (long long)b * NX * NX, a.kst0 + (long long)b * NX,
                last ? nullptr : a.Lst0 + (long long)b * NX * NX, !last, a.piv_rel, [] {});
        } else {
            bad = reduce_stage<T, NX, MT, KIND>(s, ref(tt), a.store_P ? a.Pst + g * NX * NX : nullptr,
                                                a.Lgst ? a.Lgst + g * MT * MT : nullptr, a.Kst + g * MT * NX, a.kst + g * MT,
                                                last ? nullptr : a.Lst + g * MT * NX, !last, a.piv_rel,
                                                [&] { load(tt - 1); });
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
            rank = chol_pivoted<T, NX, ld>(s.Qw, a.piv_rank, s.t, s.flag);
            if (rank == 0 && bad_t < 0) bad_t = cd.t0;
        } else {
            factor_block<T, NX, ld, MHE_TEAM>(s.Qw, s.X, s.thr, a.piv_rel, s.flag);
            wsync();
            if (*s.flag != (T)0 && bad_t < 0) bad_t = cd.t0;
        }
        // the master stage's data at cd.parent (and at its mirror cd.parent2, when given)
        const int copies = cd.parent2 >= 0 ? 2 : 1;
        wfor(copies * NX * NX, [&](int u) {
            const long long gp = u < NX * NX ? cd.parent : cd.parent2;
            const int idx = u % (NX * NX);
            const int i = idx % NX, j = idx / NX;
            a.Ah_up[gp * NX * NX + idx] = s.V[j + i * ld];
            if (a.piv_up) {   // row Pi(i) of B is row i of L (columns j >= r are zero)
                const int pi = (int)s.t[i];
                a.Bh_up[gp * NX * NX + pi + j * NX] = (i >= j && j < rank) ? s.Qw[i + j * ld] : (T)0;
                if (j == 0) a.piv_up[gp * (NX + 1) + i] = pi;
                if (idx == 0) a.piv_up[gp * (NX + 1) + NX] = rank;
            } else {
                // (the factor's diagonal is kept as its reciprocal)
                const T l = s.Qw[i + j * ld];
                a.Bh_up[gp * NX * NX + idx] = i > j ? l : (i == j ? (T)1 / l : (T)0);
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
    if (bad_t >= 0) wone([&](int) { record_error(a.status, a.where, b, -3, a.level, ci, bad_t); });
}

MHE_TEAM_NS_END
}  // namespace mhe
