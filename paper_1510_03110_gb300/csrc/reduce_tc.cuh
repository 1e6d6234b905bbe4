// reduce_tc.cuh -- Algorithms 1-2 over whole instances (one chunk each, no master problem above) with the
// stage products on the tensor cores, in a workspace two teams of an SM can hold.
//
// A stage is a chain: operands split and laid out as tiles, two products, the factor of G by one
// warp, a column solve per lane, P's update.  One team leaves its SM idle most of that time (issue 16%, one
// warp a scheduler, ncu), so the rate is the number of teams.  The general workspace (tree.cuh: ten n x n slots and a
// 32 KB tile, 204 KB, all 512 TMEM columns) allows one.  Without V the slots shrink to what is live at a time:
//   stage data [A | B], then its tiles (hi, lo), then the next stage's data as it arrives;
//   P, then its tiles, then those of X = P [A | B], then F, H^T, G and the factor.
// Every matrix is read into registers before its tiles overwrite it.  The second product's accumulator
// takes the columns of the first (read by then), so 256 of the 512 columns suffice.
#pragma once
#include "tree.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// the workspace, in floats
template <int NX, int NW>
struct TcWs {
    static constexpr int NAB = NX + NW;
    static constexpr int ld = pick_ld(NX, 4), lm = pick_ld(NW, 4);
    static constexpr int tile = NAB * NX;               // one of the two [A | B]^T tiles
    static constexpr int oA = 0, oB = oA + NX * ld;     // stage data, over the tiles
    static constexpr int oX = 2 * tile;                 // the stacked tiles of P, then of X^T
    static constexpr int oP = oX, oY = oP + NX * ld, oG = oY + (NX + 1) * lm, oR = oG + NW * lm;
    static constexpr int xlen = 2 * NAB * NX;
    static constexpr int vec = oX + xlen;
    static constexpr int nvec = 7;                      // Psi, u, e, t, g, tmp and scratch
    static constexpr int count = vec + nvec * NX + 8;
    // the arrival stage's n x n blocks: two below the tiles' end, P, one above it
    static constexpr int aG = 0, aY = NX * ld, aK = oP + NX * ld;
    static_assert(NX % 16 == 0 && NW % 16 == 0 && NAB <= 128, "MMA shapes");
    static_assert(oB + NW * ld <= oX && oR + NW * lm <= vec && 2 * NX * NX <= xlen, "what shares a region fits it");
    static_assert(2 * NX * ld <= oX && aK + NX * ld <= vec, "the arrival stage fits");
    // an MMA reads 128 rows of a tile: those past n + m (any values; their results are not read) lie in what follows
    static_assert(128 * NX - tile <= xlen, "rows past a tile stay in the workspace");
};

// shapes it is compiled for: the column solves take one warp's factor of at most 32 rows
template <int NX, int NW>
constexpr bool tc_last_shape()
{
    return MHE_TEAM == 128 && NX % 16 == 0 && NW % 16 == 0 && NX + NW <= 128 && 2 * (NX + NW) <= 256 && NW <= 32 &&
           (NX + NW) * (NX / 4) % MHE_TEAM == 0 && NX * (NX / 4) % MHE_TEAM == 0;
}

// F, G, H of one stage (tree.cuh: tc_stage_products has the arithmetic): F -> P, H^T -> Y, G.  before() runs
// once the stage's tiles have been read.
template <int NX, int NW, class FB>
MHE_DEV void tc_last_products(float* sm, const StageRef<float>& st, TcState& tcs, FB&& before)
{
    using X = Acc<float, KIND_LEAF, NX, NW>;
    using W = TcWs<NX, NW>;
    constexpr int ld = W::ld, lm = W::lm, NAB = W::NAB;
    constexpr int LBO = 128, SBO = (NX / 4) * 128;
    constexpr int PAB = NAB * (NX / 4) / MHE_TEAM, PP = NX * (NX / 4) / MHE_TEAM;   // 16-byte pieces a lane
    char* ABh = reinterpret_cast<char*>(sm);
    char* ABl = reinterpret_cast<char*>(sm + W::tile);
    char* Xh = reinterpret_cast<char*>(sm + W::oX);
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
    {
        // row r of [A|B]^T is column r of A or B (B's columns follow A's), row r of P its column r
        const int lane = lane_id();
        float ab[PAB][4], p[PP][4];
#pragma unroll
        for (int q = 0; q < PAB; ++q) {
            const int u = lane + q * MHE_TEAM;
            ld16(sm + W::oA + (u % NAB) * ld + 4 * (u / NAB), ab[q]);
        }
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int u = lane + q * MHE_TEAM;
            ld16(sm + W::oP + (u % NX) * ld + 4 * (u / NX), p[q]);
        }
        wsync();
#pragma unroll
        for (int q = 0; q < PAB; ++q) {
            const int u = lane + q * MHE_TEAM;
            split_store(ABh, ABl, tc::kmaj_off(u % NAB, 4 * (u / NAB), LBO, SBO), ab[q]);
        }
#pragma unroll
        for (int q = 0; q < PP; ++q) {
            const int u = lane + q * MHE_TEAM;
            split_store(Xh, Xh + (NX / 8) * SBO, tc::kmaj_off(u % NX, 4 * (u / NX), LBO, SBO), p[q]);
        }
        tc::fence_smem_to_async();
        tc::fence_before();
        wsync();
    }
    // [hi*hi | hi*lo + lo*hi] of the 128-row tile times the stacked one of N rows, from TMEM column 0
    auto issue = [&](int N, uint32_t id1, uint32_t id2) {
        tc::fence_after();
#pragma unroll 1
        for (int k = 0; k < NX / 8; ++k) {
            const uint64_t ah = tc::sdesc(ABh + 256 * k, LBO, SBO), al = tc::sdesc(ABl + 256 * k, LBO, SBO);
            const uint64_t b = tc::sdesc(Xh + 256 * k, LBO, SBO);
            tc::mma_tf32(tcs.tbase, ah, b, id2, k > 0);
            tc::mma_tf32(tcs.tbase + N, al, b, id1, true);
        }
        tc::commit(tcs.mbar);
    };
    if (lane_id() == 0 && tcs.ok) issue(NX, tc::idesc_tf32(128, NX), tc::idesc_tf32(128, 2 * NX));
    tc_team_wait(tcs);
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
                    split_store(Xh, Xh + (NAB / 8) * SBO, tc::kmaj_off(r, c + 4 * q, LBO, SBO), x);
                }
            }
        }
    });
    if (lane_id() == 0 && tcs.ok) issue(NAB, tc::idesc_tf32(128, NAB), tc::idesc_tf32(128, 2 * NAB));
    const int r = lane_id();
    const bool row = r < NAB;   // whole warps
    float qv[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, i) : 0.f;
    tc_team_wait(tcs);
    before();
#pragma unroll 1
    for (int c = 0; c < NAB; c += 16) {
        float v[16], w[16];
        tmem_pair(tcs, r, c, NAB + c, v, w);
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = qv[i] + (v[i] + w[i]);
        if (c + 16 < NAB) {
#pragma unroll
            for (int i = 0; i < 16; ++i) qv[i] = row ? X::q(st, r, c + 16 + i) : 0.f;
        }
        if (r < NX && c >= NX) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float x[4] = {v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]};
                st16(sm + W::oY + r * lm + (c - NX) + 4 * q, x);
            }
        } else if (r < NX) {
#pragma unroll
            for (int i = 0; i < 16; ++i) sm[W::oP + r + (c + i) * ld] = v[i];
        } else if (row && c >= NX) {
#pragma unroll
            for (int i = 0; i < 16; ++i) sm[W::oG + (r - NX) + (c - NX + i) * lm] = v[i];
        }
    }
    tc::fence_before();
    wsync();
}

template <int NX, int NW>
MHE_DEV void reduce_last_tc(const LevelArgs<float>& a, int ci, float* sm, TcState& tcs)
{
    using W = TcWs<NX, NW>;
    using X = Acc<float, KIND_LEAF, NX, NW>;
    constexpr int ld = W::ld, lm = W::lm;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    const float* lN = a.lN ? a.lN + (long long)b * NX : nullptr;   // level 0: Q_{x,N} = 0
    float *P = sm + W::oP, *Y = sm + W::oY, *G = sm + W::oG, *R = sm + W::oR;
    float *Psi = sm + W::vec, *u = Psi + NX, *e = u + NX, *tv = e + NX, *g = tv + NX, *tmp = g + NX, *sc = tmp + NX;
    auto load = [&](int t) {
        if (t < 1) return;
        const StageRef<float> st = Addr<float, NX, NW>::leaf(a, b, t);
        async_block<float, NX, NX, ld>(sm + W::oA, st.A);
        async_block<float, NX, NW, ld>(sm + W::oB, st.B);
        if (st.a) async_vec<float, NX>(e, st.a);
        cp_commit();
    };
    each<NX>([&](int i) {
        Psi[i] = lN ? -lN[i] : 0.f;
        e[i] = 0.f;
    });
    wfor(NX * NX, [&](int k) { P[k % NX + (k / NX) * ld] = 0.f; });
    int bad_t = -1;
    prefetch_leaf<float, NX, NW>(a, b, cd.t0 + cd.len - 1);
    load(cd.t0 + cd.len - 1);
    for (int tt = cd.len - 1; tt >= 0; --tt) {
        const int t = cd.t0 + tt;
        const long long gs = cd.g0 + tt;
        bool bad;
        if (t > 0) {
            if (tt > 0) prefetch_leaf<float, NX, NW>(a, b, t - 1);
            const StageRef<float> st = Addr<float, NX, NW>::leaf(a, b, t);
            cp_wait<0>();
            wsync();
            // u = Psi - P a;  A^T u,  g = B^T u - l_w
            each<NX>([&](int i) { u[i] = Psi[i] - coldot<NX>(P + i * ld, e, 0.f); });
            if (a.store_P) store_block<float, NX, NX, ld>(a.Pst + gs * NX * NX, P, 1.f, 0, [](int) {});
            else wsync();
            each<NX + NW>([&](int i) {
                const float d = coldot<NX>(sm + W::oA + i * ld, u, 0.f);
                if (i < NX) tv[i] = d;
                else g[i - NX] = d - X::lw(st, i - NX);
            });
            tc_last_products<NX, NW>(sm, st, tcs, [&] { load(t - 1); });
            each<NW>([&](int j) { Y[NX * lm + j] = g[j]; });
            factor_block<float, NW, lm, MHE_TEAM>(G, R, tmp, a.piv_rel, sc);
            wsync();
            bad = sc[0] != 0.f;
            store_factor<float, NW, lm>(a.Lgst + gs * NW * NW, G);
            solve_columns<float, NX, NW, lm, 1>(Y, Y, G, R, false, a.Kst + gs * NW * NX, a.kst + gs * NW, nullptr);
            wsync();
            prod<float, NX, NX, NW, lm, lm, true, 0, MHE_TEAM>(
                Y, Y, [](int, int) { return None(); }, [&](int i, int j, float v, None) {
                    P[i + j * ld] = P[j + i * ld] = (i < j ? P[i + j * ld] : P[j + i * ld]) - v;
                });
            each<NX>([&](int i) { Psi[i] = tv[i] - X::lx(st, i) - coldot<NW>(Y + i * lm, Y + NX * lm, 0.f); });
            wsync();
        } else {
            // the arrival stage: A = B = I, Q = diag(0, P~0^{-1}), so F = H = P and G = P~0^{-1} + P
            using XA = Acc<float, KIND_ARRIVAL, NX, NX>;
            const StageRef<float> st = Addr<float, NX, NW>::arrival(a, b);
            Ws<float, NX> s;
            s.P = P;
            s.G = sm + W::aG;
            s.PB = sm + W::aY;
            s.K = s.H = sm + W::aK;
            s.Psi = Psi; s.g = g; s.k = e; s.tmp = tmp; s.sc = sc; s.tv = tv;
            each<NX>([&](int i) {
                tv[i] = Psi[i];
                for (int p = 0; p < NX; ++p) tv[i] -= P[i + p * ld] * XA::a(st, p);
                g[i] = tv[i] - XA::lw(st, i);
            });
            wfor(NX * NX, [&](int k) {
                const int i = k % NX, j = k / NX;
                s.G[i + j * ld] = XA::qw(st, i, j) + P[i + j * ld];
            });
            if (a.store_P) store_block<float, NX, NX, ld>(a.Pst0 + (long long)b * NX * NX, P, 1.f, 0, [](int) {});
            bad = chol_G<float, NX, NX>(s, a.piv_rel);
            auto rhs = [&](int i, int c) -> float { return c < NX ? P[c + i * ld] : g[i]; };
            auto getY = [&](int i, int c) -> float { return c < NX ? s.PB[i + c * ld] : u[i]; };
            auto putY = [&](int i, int c, float v) { (c < NX ? s.PB[i + c * ld] : u[i]) = v; };
            auto getX = [&](int i, int c) -> float { return c < NX ? -s.K[i + c * ld] : e[i]; };
            auto putX = [&](int i, int c, float v) {
                if (c < NX) s.K[i + c * ld] = -v;
                else e[i] = v;
            };
            lower_solve<float, NX, NX, NX + 1>(s, rhs, getY, putY);
            upper_solve<float, NX, NX, NX + 1>(s, getY, getX, putX);
            store_block<float, NX, NX, ld>(a.Kst0 + (long long)b * NX * NX, s.K, 1.f, NX,
                                           [&](int j) { a.kst0[(long long)b * NX + j] = e[j]; });
            // nothing reads P_0, Psi_0: no problem lies above, and x_0 is known
            store_factor<float, NX, ld>(a.Lgst0 + (long long)b * NX * NX, s.G);
        }
        if (bad && bad_t < 0) bad_t = t;
    }
    cp_wait<0>();
    // a tensor-core wait that ran out: the products after it are not valid
    if (!tcs.ok) wone([&](int) { record_error(a.status, a.where, b, -7, a.level, ci, cd.t0); });
    if (bad_t >= 0) wone([&](int) { record_error(a.status, a.where, b, -3, a.level, ci, bad_t); });
}

MHE_TEAM_NS_END
}  // namespace mhe
