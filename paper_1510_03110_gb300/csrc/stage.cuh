// stage.cuh -- what every pass over a chunk's stages shares: where a stage's data lie
// (the caller's arrays, the arrival stage, a master problem's stage) and the index
// checks of the bounds-checked build.
#pragma once
#include <stdint.h>

#include "common.h"
#include "warp.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

enum { KIND_LEAF = 0, KIND_ARRIVAL = 1, KIND_UPPER = 2 };

// Leading dimension of the workspace matrices: a multiple of the 16-byte
// vector (V elements) so every column starts 16-byte aligned, with an odd
// number of vectors per column so neighbouring columns start in different
// bank groups.
constexpr int pick_ld(int n, int v)
{
    int l = n;
    while (l % v != 0 || (l / v) % 2 == 0) ++l;
    return l;
}

// Data of one stage.  LEAF: the caller's stage arrays (Q is (n+m)^2).
// ARRIVAL: A = B = I, Q = diag(0, P~0^{-1}).  UPPER: a master-problem stage in
// square-root form: A = A^, B = R^T, Q = blkdiag(Q^_x, I), l = (l^_x, 0),
// where R^T R = Q^_w is the Cholesky factorisation of the T-form Q^_w = B^.
template <typename T>
struct StageRef {
    const T *A, *B, *Q, *Qx, *Qw0, *l, *a;
};

template <typename T, int KIND, int NX, int MT>
struct Acc {
    static MHE_DEV T A(const StageRef<T>& s, int i, int j)
    {
        return KIND == KIND_ARRIVAL ? (T)(i == j ? 1 : 0) : s.A[i + j * NX];
    }
    static MHE_DEV T B(const StageRef<T>& s, int i, int j)
    {
        return KIND == KIND_ARRIVAL ? (T)(i == j ? 1 : 0) : s.B[i + j * NX];
    }
    static MHE_DEV T qx(const StageRef<T>& s, int i, int j)
    {
        if (KIND == KIND_LEAF) return s.Q[i + j * (NX + MT)];
        if (KIND == KIND_UPPER) return s.Qx[i + j * NX];
        return (T)0;
    }
    static MHE_DEV T qxw(const StageRef<T>& s, int i, int j)
    {
        return KIND == KIND_LEAF ? s.Q[i + (NX + j) * (NX + MT)] : (T)0;
    }
    static MHE_DEV T qw(const StageRef<T>& s, int i, int j)
    {
        if (KIND == KIND_LEAF) return s.Q[(NX + i) + (NX + j) * (NX + MT)];
        if (KIND == KIND_UPPER) return (T)(i == j ? 1 : 0);   // square-root master stage
        return s.Qw0[i + j * NX];
    }
    // entry (i, j) of the stage Hessian [[Q_x, Q_xw], [Q_xw^T, Q_w]], i, j < n + m
    static MHE_DEV T q(const StageRef<T>& s, int i, int j)
    {
        if (KIND == KIND_LEAF) return s.Q[i + j * (NX + MT)];
        if (i < NX && j < NX) return qx(s, i, j);
        if (i >= NX && j >= NX) return qw(s, i - NX, j - NX);
        return (T)0;   // Q_xw = 0 at the arrival and master stages
    }
    static MHE_DEV T lx(const StageRef<T>& s, int i) { return s.l ? s.l[i] : (T)0; }
    static MHE_DEV T lw(const StageRef<T>& s, int j)
    {
        return (KIND != KIND_UPPER && s.l) ? s.l[NX + j] : (T)0;
    }
    static MHE_DEV T a(const StageRef<T>& s, int i) { return s.a ? s.a[i] : (T)0; }
};

// ---- bounds-checked build -----------------------------------------------------
// Compiled with MHE_BOUNDS_CHECK (libmhe_bounds.so), the tree passes check each
// chunk descriptor against the extents of the level's arrays before the chunk is
// processed, and each caller-stage index before it is used: an index outside its
// array records MHE_E_BOUNDS for the instance with (level, chunk, index), and the
// chunk is skipped or the index replaced by 0, so that no access leaves its
// array.  Extents < 0 are not checked (serving rings).  The regular build
// compiles none of it.
constexpr int kBoundsCode = -10;   // MHE_E_BOUNDS

MHE_DEV bool in_ext(long long i, long long ext) { return ext < 0 || (i >= 0 && i < ext); }

template <typename T>
MHE_DEV long long bounds_index(const LevelArgs<T>& a, int b, long long i, long long ext)
{
#ifdef MHE_BOUNDS_CHECK
    if (!in_ext(i, ext)) {
        if (b >= 0 && b < a.ext_batch) record_error(a.status, a.where, b, kBoundsCode, a.level, -1, (int)i);
        return 0;
    }
#else
    (void)a; (void)b; (void)ext;
#endif
    return i;
}

// the descriptor of chunk ci within the level's extents (always true in the regular build)
template <typename T>
MHE_DEV bool chunk_in_bounds(const LevelArgs<T>& a, int ci)
{
#ifdef MHE_BOUNDS_CHECK
    const ChunkDesc cd = a.chunks[ci];
    if (cd.inst < 0 || cd.inst >= a.ext_batch) return false;   // no instance to report to
    const LevelInst li = a.li[cd.inst];
    bool out = true;
    long long bad = 0;   // the offending index, reported in the stage field of where
    if (cd.t0 < 0 || cd.len < 1 || cd.t0 + cd.len > li.N) bad = cd.t0;
    else if (!in_ext(cd.g0, a.ext_S) || !in_ext(cd.g0 + cd.len - 1, a.ext_S)) bad = cd.g0;
    else if (!in_ext(li.gx, a.ext_X) || !in_ext(li.gx + li.N, a.ext_X)) bad = li.gx;
    else if (cd.parent >= 0 && (!in_ext(cd.parent, a.ext_S_up) || !in_ext(cd.pw, a.ext_S_up))) bad = cd.parent;
    else if (cd.parent2 >= 0 && !in_ext(cd.parent2, a.ext_S_up)) bad = cd.parent2;
    else if (cd.px >= 0 && !in_ext(cd.px, a.ext_X_up)) bad = cd.px;
    else out = false;
    if (out) {
        if (lane_id() == 0) record_error(a.status, a.where, cd.inst, kBoundsCode, a.level, ci, (int)bad);
        return false;
    }
#else
    (void)a; (void)ci;
#endif
    return true;
}

// ---- stage addressing -------------------------------------------------------

template <typename T, int NX, int NW>
struct Addr {
    // level-0 stage t >= 1 of instance b
    static MHE_DEV StageRef<T> leaf(const LevelArgs<T>& a, int b, int t)
    {
        return leaf_at(a, b, a.in_off[b] + t - 1, a.rhs_off[b] + t - 1);
    }
    // the same at caller stage si, right-hand side stage sri
    static MHE_DEV StageRef<T> leaf_at(const LevelArgs<T>& a, int b, long long si, long long sri)
    {
        const long long s = bounds_index(a, b, si, a.ext_S_in);
        const long long sr = bounds_index(a, b, sri, a.ext_S_in);
        StageRef<T> r;
        r.A = a.A + s * NX * NX;
        r.B = a.B + s * NX * NW;
        r.Q = a.Q + s * (NX + NW) * (NX + NW);
        r.Qx = nullptr;
        r.Qw0 = nullptr;
        r.l = a.l ? a.l + sr * (NX + NW) : nullptr;
        r.a = a.a ? a.a + sr * NX : nullptr;
        return r;
    }
    static MHE_DEV StageRef<T> arrival(const LevelArgs<T>& a, int b)
    {
        StageRef<T> r;
        r.A = r.B = r.Q = r.Qx = nullptr;
        r.Qw0 = a.P0inv + (long long)b * NX * NX;
        r.l = a.l0 ? a.l0 + (long long)b * 2 * NX : nullptr;
        r.a = a.a0 ? a.a0 + (long long)b * NX : nullptr;
        return r;
    }
    static MHE_DEV StageRef<T> upper(const LevelArgs<T>& a, long long g)
    {
        StageRef<T> r;
        r.A = a.Ah + g * NX * NX;
        r.B = a.Bh + g * NX * NX;
        r.Q = nullptr;
        r.Qx = a.Qxh + g * NX * NX;
        r.Qw0 = nullptr;
        r.l = a.lxh ? a.lxh + g * NX : nullptr;
        r.a = a.ah ? a.ah + g * NX : nullptr;
        return r;
    }
};

// L2 prefetch of A, B, Q, l and a of level-0 stage t of instance b (t >= 1)
template <typename T, int NX, int NW>
MHE_DEV void prefetch_leaf(const LevelArgs<T>& a, int b, int t)
{
    if (t < 1) return;
#ifdef MHE_BOUNDS_CHECK
    if (!in_ext(a.in_off[b] + t - 1, a.ext_S_in) || !in_ext(a.rhs_off[b] + t - 1, a.ext_S_in)) return;
#endif
    const long long s = a.in_off[b] + t - 1;
    prefetch_l2(a.A + s * NX * NX, (int)(sizeof(T) * NX * NX));
    prefetch_l2(a.B + s * NX * NW, (int)(sizeof(T) * NX * NW));
    prefetch_l2(a.Q + s * (NX + NW) * (NX + NW), (int)(sizeof(T) * (NX + NW) * (NX + NW)));
    if (a.l) prefetch_l2(a.l + (a.rhs_off[b] + t - 1) * (NX + NW), (int)(sizeof(T) * (NX + NW)));
    if (a.a) prefetch_l2(a.a + (a.rhs_off[b] + t - 1) * NX, (int)(sizeof(T) * NX));
}

MHE_TEAM_NS_END
}  // namespace mhe
