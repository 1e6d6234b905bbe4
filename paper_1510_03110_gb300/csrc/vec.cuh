// vec.cuh -- the vector passes over one chunk: the right-hand-side part of Algorithm 4
// with stored factors, and Algorithm 6 as back-substitution.
//
// Both passes walk a chunk's stages one after another and do a few matrix-vector
// products per stage, so they are bound by how fast a stage's data arrive (HBM for a
// full chip, one load's latency after another for a few chunks).  Every team therefore
// keeps a ring of stage slots in shared memory that asynchronous copies (cp.async)
// fill DEPTH - 1 stages ahead; the products read shared memory only.  The matrices a
// product reads by columns (A^T u, K^T g) get a padded leading dimension, so the lanes'
// 16-byte loads fall in distinct bank groups; those read by rows stay as they are.
//
// k = G^{-1} g by two substitutions with the stored factor (factor_solve below).  L^{-1} stored instead and applied as
// two products was faster by up to 8% of a solve, but its error grows with |L^{-1}| |g|, not with |L^{-1} g|: residuals up
// to 100 times those of substitutions, and an FP32 interior-point loop (256 of nx = nw = 20, leaves of 16) that did not
// converge in 150 iterations where it now takes 29.
//
// Measured against passes that loaded each stage as they came to it (GB300, first full pass): down pass
// nx = 24, 535k stages, 1.91 -> 1.36 ms (4.8 TB/s); nx = 12, 1.05M stages, 1.10 -> 0.70 ms; nx = 64, 131k stages,
// 3.57 -> 1.59 ms; right-hand-side pass nx = 24 1.45 -> 1.15 ms, nx = 64 3.11 -> 1.39 ms; one master level of
// four-stage chunks at nx = 24 22 -> 14 us.
#pragma once
#include <stdint.h>

#include "common.h"
#include "stage.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// ---- asynchronous copies ------------------------------------------------------

// the widest piece (16, 8 or 4 bytes) that divides `bytes`
constexpr int piece_of(int bytes) { return bytes % 16 == 0 ? 16 : (bytes % 8 == 0 ? 8 : 4); }
constexpr int min_int(int a, int b) { return a < b ? a : b; }
// FP64 arrays may be the caller's (8-byte aligned); FP32 ones are the library's own, back to
// back blocks in 256-byte aligned arenas
template <typename T>
constexpr int max_piece() { return sizeof(T) == 4 ? 16 : 8; }

template <int BYTES>
MHE_DEV void cp_async(void* dst, const void* src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
    else if constexpr (BYTES == 8) asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d), "l"(src) : "memory");
}
MHE_DEV void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
MHE_DEV void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// R x C column-major block, columns SLD apart at src, to columns LD apart at dst (both multiples of
// one piece); ALIGN: bytes every block's start is a multiple of, when less than a column's own
template <typename T, int R, int C, int LD, int SLD = R, int ALIGN = 16>
MHE_DEV void async_block(T* dst, const T* src)
{
    constexpr int B = (int)sizeof(T);
    constexpr bool flat = LD == R && SLD == R;
    constexpr int g0 = flat ? piece_of(R * C * B) : min_int(piece_of(R * B), min_int(piece_of(LD * B), piece_of(SLD * B)));
    constexpr int g = min_int(min_int(g0, max_piece<T>()), ALIGN);
    constexpr int E = g / B;
    static_assert(g >= B && (flat || R % E == 0), "whole pieces");
    constexpr int NP = R * C / E;
#pragma unroll
    for (int k = 0; k < (NP + MHE_TEAM - 1) / MHE_TEAM; ++k) {
        const int u = lane_id() + k * MHE_TEAM;
        if (u < NP) {
            if constexpr (flat) {
                cp_async<g>(dst + u * E, src + u * E);
            } else {
                constexpr int PC = R / E;
                const int c = u / PC, q = (u % PC) * E;
                cp_async<g>(dst + c * LD + q, src + c * SLD + q);
            }
        }
    }
}

// n entries, zeros when src is null
template <typename T, int N, int ALIGN = 16>
MHE_DEV void async_vec(T* dst, const T* src)
{
    if (src) async_block<T, N, 1, N, N, ALIGN>(dst, src);
    else
        for (int i = lane_id(); i < N; i += MHE_TEAM) dst[i] = (T)0;
}

// ---- packed FP32 pairs (fma.rn.f32x2 and the like work on register pairs) ------

using F2 = unsigned long long;
MHE_DEV F2 pack2(float x, float y)
{
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
MHE_DEV float2 unpack2(F2 v)
{
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
MHE_DEV F2 fma2(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
MHE_DEV F2 add2(F2 a, F2 b)
{
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
MHE_DEV F2 mul2(F2 a, F2 b)
{
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// ---- products with shared-memory operands -------------------------------------

// the widest vector (16 or 8 bytes, else one entry) whole columns of n entries can be read in
template <typename T>
constexpr int vec_of(int n)
{
    return sizeof(T) == 8 ? (n % 2 == 0 ? 2 : 1) : (n % 4 == 0 ? 4 : (n % 2 == 0 ? 2 : 1));
}
template <typename T, int V>
MHE_DEV void ldv(const T* p, T (&v)[V])
{
    if constexpr (V * sizeof(T) == 16) {
        ld16(p, v);
    } else if constexpr (V == 2) {
        const float2 q = *reinterpret_cast<const float2*>(p);
        v[0] = q.x; v[1] = q.y;
    } else {
        v[0] = p[0];
    }
}

// sum_{p < K} col[p] v[p]: a contiguous column and a vector, both aligned to vec_of(K) entries
template <int K, typename T>
MHE_DEV T coldot(const T* col, const T* v, T init)
{
    constexpr int V = vec_of<T>(K);
    T acc[V];
#pragma unroll
    for (int q = 0; q < V; ++q) acc[q] = (T)0;
#pragma unroll
    for (int p = 0; p < K; p += V) {
        T a[V], b[V];
        ldv(col + p, a);
        ldv(v + p, b);
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] += a[q] * b[q];
    }
    T s = init;
#pragma unroll
    for (int q = 0; q < V; ++q) s += acc[q];
    return s;
}

// sum_{p < K} row[p LD] v[p]: one entry of K columns LD apart, v 16-byte aligned
template <int K, int LD, typename T>
MHE_DEV T rowdot(const T* row, const T* v, T init)
{
    constexpr int V = vec_of<T>(K);
    T acc[V];
#pragma unroll
    for (int q = 0; q < V; ++q) acc[q] = (T)0;
#pragma unroll
    for (int p = 0; p < K; p += V) {
        T b[V];
        ldv(v + p, b);
#pragma unroll
        for (int q = 0; q < V; ++q) acc[q] += row[(p + q) * LD] * b[q];
    }
    T s = init;
#pragma unroll
    for (int q = 0; q < V; ++q) s += acc[q];
    return s;
}

// f(idx) for idx < COUNT, lanes round-robin, no barrier
template <int COUNT, class F>
MHE_DEV void each(F&& f)
{
#pragma unroll
    for (int k = 0; k < (COUNT + MHE_TEAM - 1) / MHE_TEAM; ++k) {
        const int i = lane_id() + k * MHE_TEAM;
        if (i < COUNT) f(i);
    }
}

// ---- the slots ----------------------------------------------------------------

constexpr int round_to(int n, int v) { return (n + v - 1) / v * v; }

// offsets (elements of T) of a stage's data in a slot; MT = the stage's input width
template <typename T, int NX, int MT, int KIND>
struct RhsSlot {   // right-hand-side pass: [A | B], P, [K | factor of G], a, l, k
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int ldA = pick_ld(NX, vec_of<T>(NX)), ldK = pick_ld(MT, vec_of<T>(MT));
    static constexpr int oA = 0;
    static constexpr int oB = KIND == KIND_ARRIVAL ? 0 : ldA * NX;   // next to A: a column of [A | B] is one of A's
    static constexpr int oP = KIND == KIND_ARRIVAL ? 0 : round_to(oB + ldA * MT, V);
    static constexpr int oK = oP + round_to(NX * NX, V);
    static constexpr int oL = oK + ldK * NX;
    static constexpr int oa = round_to(oL + ldK * MT, V);
    static constexpr int ol = oa + round_to(NX, V);
    static constexpr int ok = ol + round_to(NX + MT, V);
    static constexpr int size = ok + round_to(MT, V);
    // pieces the unrounded offsets allow
    static constexpr int aB = piece_of(oB * (int)sizeof(T)), aL = piece_of(oL * (int)sizeof(T));
};
template <typename T, int NX, int MT, int KIND>
struct FwdSlot {   // down pass, forward: A, B, [K, L], k, a
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int oA = 0;
    static constexpr int oB = KIND == KIND_ARRIVAL ? 0 : round_to(NX * NX, V);
    static constexpr int oK = KIND == KIND_ARRIVAL ? 0 : oB + round_to(NX * MT, V);
    static constexpr int oL = oK + round_to(MT * NX, V);
    static constexpr int ok = oL + round_to(MT * NX, V);
    static constexpr int oa = ok + round_to(MT, V);
    static constexpr int size = oa + round_to(NX, V);
};
template <typename T, int NX, int MT, int KIND>
struct BwdSlot {   // down pass, backward: A, rows x of Q, x, w, l_x, and the FP64 targets
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int ldA = pick_ld(NX, vec_of<T>(NX));
    static constexpr int nq = KIND == KIND_LEAF ? NX + MT : NX;   // columns of Q held
    static constexpr int oA = 0;
    static constexpr int oQ = KIND == KIND_ARRIVAL ? 0 : round_to(ldA * NX, V);
    static constexpr int ox = KIND == KIND_ARRIVAL ? 0 : oQ + round_to(NX * nq, V);
    static constexpr int ow = ox + round_to(NX, V);
    static constexpr int ol = ow + round_to(MT, V);
    static constexpr int oz = ol + round_to(NX, V);
    static constexpr int size = oz + round_to((2 * NX + MT) * 8 / (int)sizeof(T), V);
};

constexpr int max_int(int a, int b) { return a > b ? a : b; }

template <typename T, int NX, int NW, bool UPPER>
struct VecWs {
    static constexpr int V = 16 / (int)sizeof(T);
    static constexpr int nv = round_to(NX, V);
    static constexpr int rhs_vectors = 6 * nv, down_vectors = 7 * nv;
    static constexpr int rhs_slot =
        UPPER ? RhsSlot<T, NX, NX, KIND_UPPER>::size
              : max_int(RhsSlot<T, NX, NW, KIND_LEAF>::size, RhsSlot<T, NX, NX, KIND_ARRIVAL>::size);
    static constexpr int down_slot =
        UPPER ? max_int(FwdSlot<T, NX, NX, KIND_UPPER>::size, BwdSlot<T, NX, NX, KIND_UPPER>::size)
              : max_int(max_int(FwdSlot<T, NX, NW, KIND_LEAF>::size, FwdSlot<T, NX, NX, KIND_ARRIVAL>::size),
                        max_int(BwdSlot<T, NX, NW, KIND_LEAF>::size, BwdSlot<T, NX, NX, KIND_ARRIVAL>::size));
    // slots of the ring.  Two where a stage is under 1 KB (nx <= 6: the copies are cheap to wait for and
    // warps count more: the nx = 6 down pass 0.34 ms with two slots, 0.46 with four) or over 4 KB (nx = 24: two
    // stages of every resident team already cover the memory latency), three between; a single slot where
    // two do not fit an SM (FP64 at nx = 64)
    static constexpr int depth_of(int slot)
    {
        const int bytes = slot * (int)sizeof(T);
        return NX >= 48 ? (sizeof(T) == 8 ? 1 : 2) : (bytes <= 1024 || bytes > 4096 ? 2 : 3);
    }
    static constexpr int rhs_depth = depth_of(rhs_slot), down_depth = depth_of(down_slot);
    static constexpr int rhs_count = rhs_depth * rhs_slot + rhs_vectors;
    static constexpr int down_count = down_depth * down_slot + down_vectors;
};

// a sweep of `len` stages through a ring of DEPTH slots: load(i, slot) starts stage i's copies,
// step(i, slot) runs once they have arrived
template <int DEPTH, typename T, class FL, class FS>
MHE_DEV void sweep(T* ring, int slot, int len, FL&& load, FS&& step)
{
    constexpr int AHEAD = DEPTH > 1 ? DEPTH - 1 : 1;
#pragma unroll 1
    for (int i = 0; i < AHEAD; ++i) {
        if (i < len) load(i, ring + i * slot);
        cp_commit();
    }
    int cur = 0, nxt = DEPTH > 1 ? AHEAD : 0;
#pragma unroll 1
    for (int i = 0; i < len; ++i) {
        cp_wait<AHEAD - 1>();
        wsync();   // stage i is there for every lane, and slot nxt (stage i - 1's) is free
        if constexpr (DEPTH > 1) {
            if (i + AHEAD < len) load(i + AHEAD, ring + nxt * slot);
            cp_commit();
        }
        step(i, ring + cur * slot);
        if constexpr (DEPTH == 1) {
            wsync();
            if (i + 1 < len) load(i + 1, ring);
            cp_commit();
        }
        cur = cur + 1 == DEPTH ? 0 : cur + 1;
        nxt = nxt + 1 == DEPTH ? 0 : nxt + 1;
    }
    cp_wait<0>();
    wsync();
}

// ---- right-hand-side pass -----------------------------------------------------

// out = G^{-1} g from G = U D U^T: the unit lower triangular U below the diagonal of the MT x MT block at L (columns LD
// apart), 1 / D_j on it; what lies above is not used.  A warp's lanes hold the entries, each finished one is passed on by
// a shuffle: with a unit diagonal a step of the chain is a shuffle and an FMA.  (One entry a lane; two at MT = 64.)
template <typename T, int MT, int LD>
MHE_DEV void factor_solve(const T* L, const T* g, T* out)
{
    constexpr int CW = MHE_TEAM < 32 ? MHE_TEAM : 32, R = (MT + CW - 1) / CW, VK = vec_of<T>(MT);
    static_assert(CW % VK == 0 && LD % VK == 0, "whole vectors of a column");
    if (MHE_TEAM > CW && lane_id() >= CW) return;
    const unsigned mask = CW == 32 ? 0xffffffffu : (((1u << CW) - 1u) << ((threadIdx.x & 31) & ~(CW - 1)));
    T v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = lane_id() + r * CW;
        v[r] = i < MT ? g[i] : (T)0;
    }
#pragma unroll
    for (int b = 0; b < R; ++b)
#pragma unroll 8
        for (int p = b * CW; p < min_int(MT, (b + 1) * CW); ++p) {
            const T f = __shfl_sync(mask, v[b], p - b * CW, CW);
#pragma unroll
            for (int r = b; r < R; ++r) {
                const int i = lane_id() + r * CW;
                if (i > p && i < MT) v[r] -= L[i + p * LD] * f;
            }
        }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = lane_id() + r * CW;
        if (i < MT) v[r] *= L[i + i * LD];
    }
#pragma unroll
    for (int b = R - 1; b >= 0; --b)
#pragma unroll 2
        for (int p0 = min_int(MT, (b + 1) * CW) - VK; p0 >= b * CW; p0 -= VK) {
            T c[R][VK];
#pragma unroll
            for (int r = 0; r <= b; ++r) {
                const int i = lane_id() + r * CW;
                if (i < MT) ldv(L + i * LD + p0, c[r]);
            }
#pragma unroll
            for (int q = VK - 1; q >= 0; --q) {
                const T f = __shfl_sync(mask, v[b], p0 + q - b * CW, CW);
#pragma unroll
                for (int r = 0; r <= b; ++r)
                    if (lane_id() + r * CW < p0 + q) v[r] -= c[r][q] * f;
            }
        }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int i = lane_id() + r * CW;
        if (i < MT) out[i] = v[r];
    }
}

// Psi_t from Psi_{t+1} (both in s_psi), k_t to kout:
//   u = Psi - P a,  [t | g] = [A | B]^T u - [0 | l_w],  Psi = t - l_x + K^T g,  k = G^{-1} g
template <typename T, int NX, int MT, int KIND>
MHE_DEV void rhs_stage(const T* sl, T* s_psi, T* s_u, T* s_tg, T* kout)
{
    using S = RhsSlot<T, NX, MT, KIND>;
    T* s_g = s_tg + round_to(NX, S::V);
    each<NX>([&](int i) { s_u[i] = s_psi[i] - rowdot<NX, NX>(sl + S::oP + i, sl + S::oa, (T)0); });
    wsync();
    if constexpr (KIND == KIND_ARRIVAL) {   // A = B = I
        each<NX>([&](int i) {
            s_tg[i] = s_u[i];
            s_g[i] = s_u[i] - sl[S::ol + NX + i];
        });
    } else {
        each<NX + MT>([&](int i) {   // column i of [A | B]
            const T d = coldot<NX>(sl + S::oA + i * S::ldA, s_u, (T)0);
            if (i < NX) s_tg[i] = d;
            else s_g[i - NX] = KIND == KIND_LEAF ? d - sl[S::ol + i] : d;
        });
    }
    wsync();
    each<NX>([&](int i) { s_psi[i] = s_tg[i] - sl[S::ol + i] + coldot<MT>(sl + S::oK + i * S::ldK, s_g, (T)0); });
    factor_solve<T, MT, S::ldK>(sl + S::oL, s_g, kout);
    wsync();
}

// x <- A x + B (K x + k) + a  (x in s_x)
template <typename T, int NX, int MT, int KIND>
MHE_DEV void closed_loop_stage(const T* sl, T* s_x, T* s_z, T* s_w)
{
    using S = RhsSlot<T, NX, MT, KIND>;
    each<NX>([&](int i) {
        const T a = sl[S::oa + i];
        s_z[i] = KIND == KIND_ARRIVAL ? a + s_x[i] : rowdot<NX, S::ldA>(sl + S::oA + i, s_x, a);
    });
    each<MT>([&](int j) { s_w[j] = rowdot<NX, S::ldK>(sl + S::oK + j, s_x, sl[S::ok + j]); });
    wsync();
    each<NX>([&](int i) {
        s_x[i] = KIND == KIND_ARRIVAL ? s_z[i] + s_w[i] : rowdot<MT, S::ldA>(sl + S::oB + i, s_w, s_z[i]);
    });
}

template <typename T, int NX, int NW, bool UPPER>
MHE_DEV void rhs_chunk(const LevelArgs<T>& a, int ci, T* smem)
{
    using W = VecWs<T, NX, NW, UPPER>;
    constexpr int MT = UPPER ? NX : NW;
    constexpr int KIND = UPPER ? KIND_UPPER : KIND_LEAF;
    using S = RhsSlot<T, NX, MT, KIND>;
    using S0 = RhsSlot<T, NX, NX, KIND_ARRIVAL>;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    if (a.active && !a.active[b]) return;
    const bool last = (cd.flags & CH_LAST) != 0;
    const bool top = (cd.flags & CH_TOP) != 0;
    // the instance's offsets once per chunk: the copies clobber memory, so the compiler would
    // load them again for every stage
    const long long si = UPPER ? 0 : a.in_off[b] - 1, sr = UPPER ? 0 : a.rhs_off[b] - 1;
    T* ring = smem + W::rhs_vectors;
    T *s_psi = smem, *s_u = smem + W::nv, *s_tg = smem + 2 * W::nv, *s_y = smem + 4 * W::nv, *s_x = smem + 5 * W::nv;
    const T* lN = UPPER ? (a.lNk ? a.lNk + (long long)b * NX : nullptr)
                        : (a.lN ? a.lN + (long long)b * NX : nullptr);
    each<NX>([&](int i) {
        s_psi[i] = (last && lN) ? -lN[i] : (T)0;
        s_x[i] = (T)0;
    });
    // backward: Psi and k of every stage
    sweep<W::rhs_depth>(
        ring, W::rhs_slot, cd.len,
        [&](int i, T* sl) {
            const int t = cd.t0 + cd.len - 1 - i;
            const long long g = cd.g0 + cd.len - 1 - i;
            if (!UPPER && t == 0) {
                const StageRef<T> st = Addr<T, NX, NW>::arrival(a, b);
                async_block<T, NX, NX, NX>(sl + S0::oP, a.Pst0 + (long long)b * NX * NX);
                async_block<T, NX, NX, S0::ldK, NX, S0::aL>(sl + S0::oL, a.Lgst0 + (long long)b * NX * NX);
                async_block<T, NX, NX, S0::ldK>(sl + S0::oK, a.Kst0 + (long long)b * NX * NX);
                async_vec<T, NX>(sl + S0::oa, st.a);
                async_vec<T, 2 * NX>(sl + S0::ol, st.l);
            } else {
                const StageRef<T> st = UPPER ? Addr<T, NX, NW>::upper(a, g) : Addr<T, NX, NW>::leaf_at(a, b, si + t, sr + t);
                async_block<T, NX, NX, S::ldA>(sl + S::oA, st.A);
                async_block<T, NX, MT, S::ldA, NX, S::aB>(sl + S::oB, st.B);
                async_block<T, NX, NX, NX>(sl + S::oP, a.Pst + g * NX * NX);
                async_block<T, MT, MT, S::ldK, MT, S::aL>(sl + S::oL, a.Lgst + g * MT * MT);
                async_block<T, MT, NX, S::ldK>(sl + S::oK, a.Kst + g * MT * NX);
                async_vec<T, NX>(sl + S::oa, st.a);
                async_vec<T, UPPER ? NX : NX + NW>(sl + S::ol, st.l);
            }
        },
        [&](int i, const T* sl) {
            const int t = cd.t0 + cd.len - 1 - i;
            const long long g = cd.g0 + cd.len - 1 - i;
            if (!UPPER && t == 0)
                rhs_stage<T, NX, NX, KIND_ARRIVAL>(sl, s_psi, s_u, s_tg, a.kst0 + (long long)b * NX);
            else
                rhs_stage<T, NX, MT, KIND>(sl, s_psi, s_u, s_tg, a.kst + g * MT);
        });
    if (!last) {
        // a^: the closed loop from x = 0 over the chunk (Eq. a)
        sweep<W::rhs_depth>(
            ring, W::rhs_slot, cd.len,
            [&](int i, T* sl) {
                const int t = cd.t0 + i;
                const long long g = cd.g0 + i;
                if (!UPPER && t == 0) {
                    const StageRef<T> st = Addr<T, NX, NW>::arrival(a, b);
                    async_block<T, NX, NX, S0::ldK>(sl + S0::oK, a.Kst0 + (long long)b * NX * NX);
                    async_vec<T, NX>(sl + S0::oa, st.a);
                    async_vec<T, NX>(sl + S0::ok, a.kst0 + (long long)b * NX);
                } else {
                    const StageRef<T> st = UPPER ? Addr<T, NX, NW>::upper(a, g) : Addr<T, NX, NW>::leaf_at(a, b, si + t, sr + t);
                    async_block<T, NX, NX, S::ldA>(sl + S::oA, st.A);
                    async_block<T, NX, MT, S::ldA, NX, S::aB>(sl + S::oB, st.B);
                    async_block<T, MT, NX, S::ldK>(sl + S::oK, a.Kst + g * MT * NX);
                    async_vec<T, NX>(sl + S::oa, st.a);
                    async_vec<T, MT>(sl + S::ok, a.kst + g * MT);
                }
            },
            [&](int i, const T* sl) {
                if (!UPPER && cd.t0 + i == 0) closed_loop_stage<T, NX, NX, KIND_ARRIVAL>(sl, s_x, s_u, s_y);
                else closed_loop_stage<T, NX, MT, KIND>(sl, s_x, s_u, s_y);
            });
        const int copies = cd.parent2 >= 0 ? 2 : 1;
        wfor(copies * NX, [&](int u) {
            const long long gp = u < NX ? cd.parent : cd.parent2;
            const int i = u % NX;
            a.ah_up[gp * NX + i] = s_x[i];
            a.lxh_up[gp * NX + i] = -s_psi[i];
        });
    } else if (!top) {
        wfor(NX, [&](int i) { a.lN_up[(long long)b * NX + i] = -s_psi[i]; });
    }
}

// ---- down pass ----------------------------------------------------------------

// |v| as a float (the size of a correction; float is ample for a norm)
MHE_DEV float absf_of(float v) { return fabsf(v); }
MHE_DEV float absf_of(double v) { return abs_to_float(v); }

// x <- L^{-T} x for the lower triangular L of a master stage's B = R^T (shared memory, leading dimension LD;
// x the same): the lanes of one warp hold the entries, each finished entry passed on by a shuffle
template <typename T, int NX, int LD>
MHE_DEV void back_substitute(const T* L, T* x)
{
    constexpr int CW = MHE_TEAM < 32 ? MHE_TEAM : 32, R = (NX + CW - 1) / CW;
    if (lane_id() < CW) {
        const unsigned mask =
            CW == 32 ? 0xffffffffu : (((1u << CW) - 1u) << ((threadIdx.x & 31) & ~(CW - 1)));
        T v[R], inv[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = lane_id() + r * CW;
            v[r] = i < NX ? x[i] : (T)0;
            inv[r] = i < NX ? (T)1 / L[i + i * LD] : (T)0;
        }
#pragma unroll 4
        for (int p = NX - 1; p >= 0; --p) {
            T f = (T)0;
#pragma unroll
            for (int r = 0; r < R; ++r)
                if (p / CW == r) f = v[r] * inv[r];
            f = __shfl_sync(mask, f, p % CW, CW);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const int i = lane_id() + r * CW;
                if (i < p) v[r] -= L[p + i * LD] * f;
                else if (i == p) x[i] = f;
            }
        }
    }
    wsync();
}

// x_t (s_x) and w_t out, s_x = x_{t+1} = A x + B w + a with w = k + K x - L w^
template <typename T, int NX, int MT, int KIND>
MHE_DEV void down_fwd_stage(const T* sl, T* s_x, T* s_z, T* s_t, const T* s_wh, bool use_wh, T* xo, T* wo)
{
    using S = FwdSlot<T, NX, MT, KIND>;
    constexpr int nm = round_to(MT, S::V);
    each<NX>([&](int i) {
        xo[i] = s_x[i];
        const T a = sl[S::oa + i];
        s_z[i] = KIND == KIND_ARRIVAL ? a + s_x[i] : rowdot<NX, NX>(sl + S::oA + i, s_x, a);
    });
    each<2 * MT>([&](int j) {   // K x + k, and L w^
        const bool k = j < MT;
        const int i = k ? j : j - MT;
        if (!k && !use_wh) {   // the last chunk of a level: no L, w^ = 0
            s_t[nm + i] = (T)0;
            return;
        }
        const T d = rowdot<NX, MT>(sl + (k ? S::oK : S::oL) + i, k ? s_x : s_wh, k ? sl[S::ok + i] : (T)0);
        s_t[k ? i : nm + i] = d;
    });
    wsync();
    each<MT>([&](int j) {
        const T w = s_t[j] - s_t[nm + j];
        wo[j] = w;
        s_t[2 * nm + j] = w;
    });
    wsync();
    each<NX>([&](int i) {
        s_x[i] = KIND == KIND_ARRIVAL ? s_z[i] + s_t[2 * nm + i] : rowdot<MT, NX>(sl + S::oB + i, s_t + 2 * nm, s_z[i]);
    });
}

// lambda_t = Q_x x_t + Q_xw w_t + l_x + A^T lambda_{t+1} (s_l), out to lo; with FP64 targets given,
// z += (x_t, w_t, lambda_t) and dzm keeps the lane's largest |added value|
template <typename T, int NX, int MT, int KIND>
MHE_DEV void down_bwd_stage(const T* sl, T* s_l, T* s_n, T* lo, double* zx, double* zw, double* zl, float& dzm)
{
    using S = BwdSlot<T, NX, MT, KIND>;
    each<NX>([&](int i) {
        T q = sl[S::ol + i];
        if constexpr (KIND == KIND_ARRIVAL) {
            q += s_l[i];
        } else {
            q = rowdot<NX, NX>(sl + S::oQ + i, sl + S::ox, q);
            if constexpr (KIND == KIND_LEAF) q = rowdot<MT, NX>(sl + S::oQ + NX * NX + i, sl + S::ow, q);
            q = coldot<NX>(sl + S::oA + i * S::ldA, s_l, q);
        }
        s_n[i] = q;
        lo[i] = q;
    });
    if (zx) {
        const double* z = reinterpret_cast<const double*>(sl + S::oz);
        each<NX>([&](int i) {
            const T l = s_n[i], x = sl[S::ox + i];
            zl[i] = z[i] + f64_of(l);
            zx[i] = z[NX + i] + f64_of(x);
            dzm = fmaxf(dzm, fmaxf(absf_of(l), absf_of(x)));
        });
        each<MT>([&](int j) {
            const T w = sl[S::ow + j];
            zw[j] = z[2 * NX + j] + f64_of(w);
            dzm = fmaxf(dzm, absf_of(w));
        });
    }
    wsync();
    each<NX>([&](int i) { s_l[i] = s_n[i]; });
}

template <typename T, int NX, int NW, bool UPPER>
MHE_DEV void down_chunk(const LevelArgs<T>& a, int ci, T* smem)
{
    using W = VecWs<T, NX, NW, UPPER>;
    constexpr int MT = UPPER ? NX : NW;
    constexpr int KIND = UPPER ? KIND_UPPER : KIND_LEAF;
    using F = FwdSlot<T, NX, MT, KIND>;
    using F0 = FwdSlot<T, NX, NX, KIND_ARRIVAL>;
    using S = BwdSlot<T, NX, MT, KIND>;
    using S0 = BwdSlot<T, NX, NX, KIND_ARRIVAL>;
    const ChunkDesc cd = a.chunks[ci];
    const int b = cd.inst;
    if (a.active && !a.active[b]) return;
    const bool last = (cd.flags & CH_LAST) != 0;
    const bool top = (cd.flags & CH_TOP) != 0;
    const long long si = UPPER ? 0 : a.in_off[b] - 1, sr = UPPER ? 0 : a.rhs_off[b] - 1, wb = UPPER ? 0 : a.w_off[b];
    T* ring = smem + W::down_vectors;
    T *s_x = smem, *s_wh = smem + W::nv, *s_l = smem + 2 * W::nv, *s_z = smem + 3 * W::nv, *s_t = smem + 4 * W::nv;
    const LevelInst li = a.li[b];
    // x^_i, w^_i, lambda^_{i+1}
    each<NX>([&](int i) {
        s_x[i] = top ? a.x0[(long long)b * NX + i] : a.xd_up[cd.px * NX + i];
        s_wh[i] = last ? (T)0 : a.wd_up[cd.pw * NX + i];
        s_l[i] = last ? (T)0 : a.ld_up[(cd.px + 1) * NX + i];
    });
    wsync();
    if (!last && a.piv_up) {
        // rank-revealing master stage B = Pi L (n x r, zero-padded): the parent solved for
        // w^'; w^ = Pi [L_11^{-T} w^'_{1..r}; 0], with L(i, j) = B(Pi(i), j)
        const int* pv = a.piv_up + cd.parent * (NX + 1);
        const T* Bq = a.Bh_up + cd.parent * NX * NX;
        wone([&](int) {
            const int r = pv[NX];
            for (int i = r - 1; i >= 0; --i) {
                T acc = s_wh[i];
                for (int p = i + 1; p < r; ++p) acc -= Bq[pv[p] + i * NX] * s_wh[p];
                s_wh[i] = acc / Bq[pv[i] + i * NX];
            }
            for (int i = 0; i < NX; ++i) s_z[i] = s_wh[i];
            for (int i = 0; i < NX; ++i) s_wh[pv[i]] = i < r ? s_z[i] : (T)0;
        });
    } else if (!last) {
        // the parent solved for w^' = R w^ (square-root master stage): w^ = R^{-1} w^', R^T in B
        constexpr int ld = pick_ld(NX, W::V);
        static_assert(ld * NX <= W::down_slot * W::down_depth, "R^T fits the ring");
        async_block<T, NX, NX, ld>(ring, a.Bh_up + cd.parent * NX * NX);
        cp_commit();
        cp_wait<0>();
        wsync();
        back_substitute<T, NX, ld>(ring, s_wh);
    }
    auto xo = [&](int t) -> T* { return a.xd + (li.gx + t) * NX; };
    auto lo = [&](int t) -> T* { return a.ld + (li.gx + t) * NX; };
    auto wo = [&](int t) -> T* {
        if (UPPER) return a.wd + (li.gs + t) * NX;
        return a.wd + wb + (t == 0 ? 0 : NX + (long long)(t - 1) * NW);
    };
    auto zxo = [&](int t) -> double* { return a.zx ? a.zx + (li.gx + t) * NX : nullptr; };
    auto zlo = [&](int t) -> double* { return a.zl ? a.zl + (li.gx + t) * NX : nullptr; };
    auto zwo = [&](int t) -> double* {
        return a.zw ? a.zw + wb + (t == 0 ? 0 : NX + (long long)(t - 1) * NW) : nullptr;
    };
    sweep<W::down_depth>(
        ring, W::down_slot, cd.len,
        [&](int i, T* sl) {
            const int t = cd.t0 + i;
            const long long g = cd.g0 + i;
            if (!UPPER && t == 0) {
                const StageRef<T> st = Addr<T, NX, NW>::arrival(a, b);
                async_block<T, NX, NX, NX>(sl + F0::oK, a.Kst0 + (long long)b * NX * NX);
                if (!last) async_block<T, NX, NX, NX>(sl + F0::oL, a.Lst0 + (long long)b * NX * NX);
                async_vec<T, NX>(sl + F0::ok, a.kst0 + (long long)b * NX);
                async_vec<T, NX>(sl + F0::oa, st.a);
            } else {
                const StageRef<T> st = UPPER ? Addr<T, NX, NW>::upper(a, g) : Addr<T, NX, NW>::leaf_at(a, b, si + t, sr + t);
                async_block<T, NX, NX, NX>(sl + F::oA, st.A);
                async_block<T, NX, MT, NX>(sl + F::oB, st.B);
                async_block<T, MT, NX, MT>(sl + F::oK, a.Kst + g * MT * NX);
                if (!last) async_block<T, MT, NX, MT>(sl + F::oL, a.Lst + g * MT * NX);
                async_vec<T, MT>(sl + F::ok, a.kst + g * MT);
                async_vec<T, NX>(sl + F::oa, st.a);
            }
        },
        [&](int i, const T* sl) {
            const int t = cd.t0 + i;
            if (!UPPER && t == 0) down_fwd_stage<T, NX, NX, KIND_ARRIVAL>(sl, s_x, s_z, s_t, s_wh, !last, xo(t), wo(t));
            else down_fwd_stage<T, NX, MT, KIND>(sl, s_x, s_z, s_t, s_wh, !last, xo(t), wo(t));
        });
    const int t1 = cd.t0 + cd.len;
    float dzm = 0.f;   // this lane's largest |value| added into z (the size of a correction)
    if (last) {
        // lambda_N = Q_{x,N} x_N + l_N (Q_{x,N} = 0 at level 0)
        const T* QN = UPPER ? a.QNk + (long long)b * NX * NX : nullptr;
        const T* lN = UPPER ? (a.lNk ? a.lNk + (long long)b * NX : nullptr)
                            : (a.lN ? a.lN + (long long)b * NX : nullptr);
        wfor(NX, [&](int i) {
            T acc = lN ? lN[i] : (T)0;
            if (QN) {
#pragma unroll 8
                for (int j = 0; j < NX; ++j) acc += QN[i + j * NX] * s_x[j];
            }
            s_l[i] = acc;
            xo(t1)[i] = s_x[i];
            lo(t1)[i] = acc;
            if (a.zx) {
                zxo(t1)[i] += f64_of(s_x[i]);
                zlo(t1)[i] += f64_of(acc);
                dzm = fmaxf(dzm, fmaxf(absf_of(s_x[i]), absf_of(acc)));
            }
        });
    }
    // bytes the starts of l_t = (l_x, l_w) and of w_t are multiples of
    constexpr int gl = piece_of((UPPER ? NX : NX + NW) * (int)sizeof(T));
    constexpr int gw = UPPER ? piece_of(NX * (int)sizeof(T))
                             : min_int(piece_of(NX * (int)sizeof(T)), piece_of(NW * (int)sizeof(T)));
    sweep<W::down_depth>(
        ring, W::down_slot, cd.len,
        [&](int i, T* sl) {
            const int t = cd.t0 + cd.len - 1 - i;
            const long long g = cd.g0 + cd.len - 1 - i;
            if (!UPPER && t == 0) {
                const StageRef<T> st = Addr<T, NX, NW>::arrival(a, b);
                async_vec<T, NX>(sl + S0::ox, xo(t));
                async_vec<T, NX, gw>(sl + S0::ow, wo(t));
                async_vec<T, NX>(sl + S0::ol, st.l);
                if (a.zx) {
                    double* z = reinterpret_cast<double*>(sl + S0::oz);
                    async_vec<double, NX>(z, zlo(t));
                    async_vec<double, NX>(z + NX, zxo(t));
                    async_vec<double, NX>(z + 2 * NX, zwo(t));
                }
            } else {
                const StageRef<T> st = UPPER ? Addr<T, NX, NW>::upper(a, g) : Addr<T, NX, NW>::leaf_at(a, b, si + t, sr + t);
                async_block<T, NX, NX, S::ldA>(sl + S::oA, st.A);
                if constexpr (UPPER) async_block<T, NX, NX, NX>(sl + S::oQ, st.Qx);
                else async_block<T, NX, NX + NW, NX, NX + NW>(sl + S::oQ, st.Q);
                async_vec<T, NX>(sl + S::ox, xo(t));
                async_vec<T, MT, gw>(sl + S::ow, wo(t));
                async_vec<T, NX, gl>(sl + S::ol, st.l);
                if (a.zx) {
                    double* z = reinterpret_cast<double*>(sl + S::oz);
                    async_vec<double, NX>(z, zlo(t));
                    async_vec<double, NX>(z + NX, zxo(t));
                    async_vec<double, MT>(z + 2 * NX, zwo(t));
                }
            }
        },
        [&](int i, const T* sl) {
            const int t = cd.t0 + cd.len - 1 - i;
            if (!UPPER && t == 0)
                down_bwd_stage<T, NX, NX, KIND_ARRIVAL>(sl, s_l, s_z, lo(t), zxo(t), zwo(t), zlo(t), dzm);
            else
                down_bwd_stage<T, NX, MT, KIND>(sl, s_l, s_z, lo(t), zxo(t), zwo(t), zlo(t), dzm);
        });
    // the instance's largest |correction entry| (non-negative floats order like their bit patterns)
    if (a.zx && a.dznorm) wlanes([&](int) {
        if (dzm > 0.f) atomicMax(a.dznorm + b, __float_as_uint(dzm));
    });
}

MHE_TEAM_NS_END
}  // namespace mhe
