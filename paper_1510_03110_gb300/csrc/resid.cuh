// resid.cuh -- FP64 KKT residual of one stage, and the MHE stage assembly.
//
// KKT rows of Eq. org_eqc_problem (Lagrangian with +lambda_{t+1}^T (A x + B w
// + a - x_{t+1}) + lambda_0^T (x~0 - x_0)):
//   x_0                                          = x~0
//   Q_x x_t + Q_xw w_t + A^T lambda_{t+1} - lambda_t = -l_x,t
//   Q_xw^T x_t + Q_w w_t + B^T lambda_{t+1}          = -l_w,t
//   A x_t + B w_t - x_{t+1}                          = -a_t
//   Q_{x,N} x_N - lambda_N                           = -l_N   (Q_{x,N} = 0 here)
// The residual r = b - K z is written back as the right-hand side of the
// correction problem K dz = r in UFTOC form (x~0' = r_0, l' = -r_l,
// a' = -r_a, l_N' = -r_N), so a right-hand-side-only solve gives dz.
#pragma once
#include "common.h"
#include "f32conv.h"
#include "reduce.cuh"
#include "vec.cuh"
#include "warp.cuh"
#include "wgemm.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// a residual entry in the precision of the correction solve
template <typename TR>
MHE_DEV TR to_tr(double v)
{
    if constexpr (sizeof(TR) == 4) return f32_rn(v);
    else return v;
}

MHE_DEV int stage_instance(const long long* gs0, int batch, long long gstage)
{
    int lo = 0, hi = batch;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if (gs0[mid] <= gstage) lo = mid; else hi = mid;
    }
    return lo;
}

template <int NX, int NW, int NY = 0>
struct ResidSmem {
    static constexpr int rows = 5 * NX + NW;
    static constexpr int q_form = 3 * rows + 4;                      // resid_rows
    // pieces of a length-n product in resid_mhe: length-nw pieces when nw divides
    // n and nw >= 3 (every task of the first phase then has one length)
    static constexpr int sp = (NX % NW == 0 && NW >= 3) ? NX / NW : 1;
    static constexpr int mhe_form = 4 * NX + 3 * NW + 3 * NY + 5 + sp * (2 * NX + NY + NW);   // resid_mhe
    static constexpr int count = q_form > mhe_form ? q_form : mhe_form;   // 8-byte entries
};

// One stage t of instance b: rows of stationarity in x_t and w_t, dynamics
// t -> t+1, plus the initial rows (t = 0) and the terminal rows (t = N-1).
// The FP64 work is the products of the rows alone; the maxima of |r|, |z|,
// |b| are taken on bit patterns (integer operations).
template <int NX, int NW, int KIND, typename TR>
MHE_DEV void resid_rows(const ResidArgs<TR>& r, int b, int t, int N, unsigned long long* sm)
{
    constexpr int MT = (KIND == 1) ? NX : NW;   // the arrival stage has width n
    constexpr int NQ = NX + MT;
    constexpr int ROWS = ResidSmem<NX, NW>::rows;
    const long long gx = r.gs0[b] + b;
    const double* xt = r.x + (gx + t) * NX;
    const double* xn = xt + NX;
    const double* lt = r.lam + (gx + t) * NX;
    const double* ln = lt + NX;
    const double* wt = r.w + r.w_off[b] + (t == 0 ? 0 : NX + (long long)(t - 1) * NW);
    const long long s = r.in_off[b] + t - 1;
    const double* A = (KIND == 1) ? nullptr : r.A + s * NX * NX;
    const double* B = (KIND == 1) ? nullptr : r.B + s * NX * NW;
    const double* Q = (KIND == 1) ? nullptr : r.Q + s * (NX + NW) * (NX + NW);
    const double* P0 = r.P0inv + (long long)b * NX * NX;
    const double* l = (KIND == 1) ? nullptr : (r.l ? r.l + s * (NX + NW) : nullptr);
    const double* a = (KIND == 1) ? nullptr : (r.a ? r.a + s * NX : nullptr);
    const long long so = r.out_off[b] + t - 1;
    TR* rl = (KIND == 1) ? r.rl0 + (long long)b * 2 * NX : r.rl + so * (NX + NW);
    TR* ra = (KIND == 1) ? r.ra0 + (long long)b * NX : r.ra + so * NX;
    const bool first = (t == 0), lastst = (t == N - 1);
    const int nrow = NQ + NX + (first ? NX : 0) + (lastst ? NX : 0);
    unsigned long long* sr = sm;
    unsigned long long* sz = sm + ROWS;
    unsigned long long* sb = sm + 2 * ROWS;
    wfor(nrow, [&](int i) {
        double res;
        unsigned long long zz = 0, bb = 0;
        if (i < NQ) {
            // stationarity rows of stage t
            double acc;
            if (KIND == 1) {
                // arrival: Q_0 = diag(0, P~0^{-1}), A_0 = B_0 = I
                if (i < NX) {
                    acc = ln[i] - lt[i];
                } else {
                    acc = ln[i - NX];
                    for (int j = 0; j < NX; ++j) acc = fma(P0[(i - NX) + j * NX], wt[j], acc);
                }
            } else {
                acc = 0.0;
                for (int j = 0; j < NX; ++j) acc = fma(Q[i + j * NQ], xt[j], acc);
                for (int j = 0; j < MT; ++j) acc = fma(Q[i + (NX + j) * NQ], wt[j], acc);
                if (i < NX) {
                    for (int j = 0; j < NX; ++j) acc = fma(A[j + i * NX], ln[j], acc);
                    acc -= lt[i];
                } else {
                    for (int j = 0; j < NX; ++j) acc = fma(B[j + (i - NX) * NX], ln[j], acc);
                }
            }
            const double li = l ? l[i] : 0.0;
            res = -li - acc;
            rl[i] = to_tr<TR>(li + acc);
            zz = (i < NX) ? (abs_bits(xt[i]) > abs_bits(lt[i]) ? abs_bits(xt[i]) : abs_bits(lt[i]))
                          : abs_bits(wt[i - NX]);
            bb = abs_bits(li);
        } else if (i < NQ + NX) {
            const int ii = i - NQ;
            double acc = -xn[ii];
            if (KIND == 1) {
                acc += xt[ii] + wt[ii];
            } else {
                for (int j = 0; j < NX; ++j) acc = fma(A[ii + j * NX], xt[j], acc);
                for (int j = 0; j < MT; ++j) acc = fma(B[ii + j * NX], wt[j], acc);
            }
            const double ai = a ? a[ii] : 0.0;
            res = -ai - acc;
            ra[ii] = to_tr<TR>(ai + acc);
            bb = abs_bits(ai);
        } else if (first && i < NQ + 2 * NX) {
            const int ii = i - NQ - NX;
            const double x0i = r.x0[(long long)b * NX + ii];
            res = x0i - xt[ii];
            r.rx0[(long long)b * NX + ii] = to_tr<TR>(res);
            bb = abs_bits(x0i);
        } else {
            // terminal rows with Q_{x,N} = 0, l_N = 0:  -(0 - lambda_N)
            const int ii = i - NQ - NX - (first ? NX : 0);
            const double* xN = r.x + (gx + N) * NX;
            const double* lamN = r.lam + (gx + N) * NX;
            res = lamN[ii];
            r.rlN[(long long)b * NX + ii] = to_tr<TR>(-res);
            zz = abs_bits(xN[ii]) > abs_bits(lamN[ii]) ? abs_bits(xN[ii]) : abs_bits(lamN[ii]);
        }
        sr[i] = abs_bits(res);
        sz[i] = zz;
        sb[i] = bb;
    });
    wone([&](int) {
        unsigned long long m0 = 0, m1 = 0, m2 = 0;
        for (int i = 0; i < nrow; ++i) {
            m0 = sr[i] > m0 ? sr[i] : m0;
            m1 = sz[i] > m1 ? sz[i] : m1;
            m2 = sb[i] > m2 ? sb[i] : m2;
        }
        atomic_max_u64(r.norms + 3LL * b + 0, m0);
        atomic_max_u64(r.norms + 3LL * b + 1, m1);
        atomic_max_u64(r.norms + 3LL * b + 2, m2);
    });
}

// Stage t >= 1 in the MHE form (Section II): Q z from C and R,
//   u = C x_t,  e = V u - S^T w_t,  [Q z]_x = C^T e,  [Q z]_w = W w_t - S u,
// the same rows as resid_rows.  The FP64 work is cut into dot products dealt
// round-robin to the lanes; a lane only selects the pointers, stride and length
// of its dot product, and all lanes then run one predicated FMA loop, so the
// FP64 instructions (the pipe that bounds this kernel) issue without branch
// divergence:
//   1. length n : A x, u = C x, A^T lam_{t+1}, B^T lam_{t+1};
//      length nw: B w, W w, S^T w
//   2. e = V u - S^T w, S u          3. C^T e
//   4. the rows  p1 + p2 - p3 + p4:  C^T e + A^T lam - lam_t + l_x;
//      W w + B^T lam - S u + l_w;  A x + B w - x_{t+1} + a;  terminal rows
// Each lane keeps its maxima of |r|, |z|, |b| and merges them once.
template <int KMAX>
MHE_DEV double dot_pred(const double* m, int sm, const double* v, int k, double acc)
{
#pragma unroll
    for (int j = 0; j < KMAX; ++j)
        if (j < k) acc = fma(m[j * sm], v[j], acc);
    return acc;
}

template <int NX, int NW, int NY, typename TR>
MHE_DEV void resid_mhe(const ResidArgs<TR>& r, int b, int t, int N, unsigned long long* sm)
{
    constexpr int NR = NW + NY, NQ = NX + NW;
    const long long gx = r.gs0[b] + b;
    const double* xt = r.x + (gx + t) * NX;
    const double* xn = xt + NX;
    const double* lt = r.lam + (gx + t) * NX;
    const double* ln = lt + NX;
    const double* wt = r.w + r.w_off[b] + NX + (long long)(t - 1) * NW;
    const long long s = r.in_off[b] + t - 1;
    const double* A = r.A + s * NX * NX;
    const double* B = r.B + s * NX * NW;
    const double* C = r.C + s * NY * NX;
    const double* R = r.R + s * NR * NR;
    const double* l = r.l ? r.l + s * NQ : nullptr;
    const double* a = r.a ? r.a + s * NX : nullptr;
    const long long so = r.out_off[b] + t - 1;
    TR* rl = r.rl + so * NQ;
    TR* ra = r.ra + so * NX;
    const bool lastst = (t == N - 1);
    double* dA = reinterpret_cast<double*>(sm);   // A x
    double* dB = dA + NX;                         // B w
    double* atl = dB + NX;                        // A^T lam_{t+1}
    double* cte = atl + NX;                       // C^T e
    double* u = cte + NX;                         // C x
    double* sw = u + NY;                          // S^T w
    double* e = sw + NY;                          // V u - S^T w
    double* btl = e + NY;                         // B^T lam_{t+1}
    double* ww = btl + NW;                        // W w
    double* su = ww + NW;                         // S u
    double* zero = su + NW;
    unsigned long long* mx = reinterpret_cast<unsigned long long*>(zero + 1);
    wone([&](int) {
        zero[0] = 0.0;
        mx[0] = mx[1] = mx[2] = 0ULL;
    });
    // V(p,q) = R[NW+p + (NW+q) NR], S(k,p) = R[k + (NW+p) NR], W(k,j) = R[k + j NR]
    // The length-n dot products (A x, C x, A^T lam, B^T lam) are cut into SP pieces of
    // length n / SP = nw when nw divides n and nw >= 3, so every task of the phase has
    // one length (measured on the batched workload: the step 83.5 -> 82.1 ms when the
    // nx = 6 and 12 shapes split too).
    constexpr int T1 = NX + NY + NX + NW;                  // length-n dot products
    constexpr int SP = ResidSmem<NX, NW, NY>::sp;          // pieces per length-n product
    constexpr int LP = NX / SP;                            // piece length
    constexpr int KM = LP > NW ? LP : NW;
    double* part = zero + 4;                               // SP x T1 partial sums (past mx[3])
    wfor(T1 * SP + NX + NW + NY, [&](int k) {
        const double* m;
        const double* v;
        double* o;
        int st, len = LP;
        if (k < T1 * SP) {
            const int r = k % T1, c = k / T1, j0 = c * LP;
            o = part + c * T1 + r;
            if (r < NX) { m = A + r + j0 * NX; st = NX; v = xt + j0; }
            else if (r < NX + NY) { m = C + (r - NX) + j0 * NY; st = NY; v = xt + j0; }
            else if (r < 2 * NX + NY) { m = A + (r - NX - NY) * NX + j0; st = 1; v = ln + j0; }
            else { m = B + (r - 2 * NX - NY) * NX + j0; st = 1; v = ln + j0; }
        } else {
            const int q = k - T1 * SP;
            len = NW;
            if (q < NX) { m = B + q; st = NX; v = wt; o = dB + q; }
            else if (q < NX + NW) { m = R + (q - NX); st = NR; v = wt; o = ww + (q - NX); }
            else { m = R + (NW + q - NX - NW) * NR; st = 1; v = wt; o = sw + (q - NX - NW); }
        }
        *o = dot_pred<KM>(m, st, v, len, 0.0);
    });
    // the length-n products from their pieces
    wfor(T1, [&](int r) {
        double s = part[r];
#pragma unroll
        for (int c = 1; c < SP; ++c) s += part[c * T1 + r];
        if (r < NX) dA[r] = s;
        else if (r < NX + NY) u[r - NX] = s;
        else if (r < 2 * NX + NY) atl[r - NX - NY] = s;
        else btl[r - 2 * NX - NY] = s;
    });
    wfor(NY + NW, [&](int k) {
        const double* m;
        double* o;
        double init;
        if (k < NY) { m = R + NW + k + NW * NR; o = e + k; init = -sw[k]; }
        else { m = R + (k - NY) + NW * NR; o = su + (k - NY); init = 0.0; }
        *o = dot_pred<NY>(m, NR, u, NY, init);
    });
    wfor(NX, [&](int i) { cte[i] = dot_pred<NY>(C + i * NY, 1, e, NY, 0.0); });
    unsigned long long m0 = 0, m1 = 0, m2 = 0;
    const int nrow = NQ + NX + (lastst ? NX : 0);
    const double* xN = r.x + (gx + N) * NX;
    const double* lamN = r.lam + (gx + N) * NX;
    wfor(nrow, [&](int i) {
        const double *p1, *p2, *p3, *p4, *z1, *z2;
        TR* dst;
        if (i < NX) {
            p1 = cte + i; p2 = atl + i; p3 = lt + i; p4 = l ? l + i : zero;
            z1 = xt + i; z2 = lt + i; dst = rl + i;
        } else if (i < NQ) {
            const int q = i - NX;
            p1 = ww + q; p2 = btl + q; p3 = su + q; p4 = l ? l + i : zero;
            z1 = wt + q; z2 = zero; dst = rl + i;
        } else if (i < NQ + NX) {
            const int ii = i - NQ;
            p1 = dA + ii; p2 = dB + ii; p3 = xn + ii; p4 = a ? a + ii : zero;
            z1 = zero; z2 = zero; dst = ra + ii;
        } else {
            // terminal rows with Q_{x,N} = 0, l_N = 0: r = lambda_N
            const int ii = i - NQ - NX;
            p1 = zero; p2 = zero; p3 = lamN + ii; p4 = zero;
            z1 = xN + ii; z2 = lamN + ii; dst = r.rlN + (long long)b * NX + ii;
        }
        const double sum = *p4 + ((*p1 + *p2) - *p3);   // r = -(l + K z) for the stationarity and dynamics rows
        *dst = to_tr<TR>(sum);
        const unsigned long long rr = abs_bits(sum), bb = abs_bits(*p4);
        const unsigned long long za = abs_bits(*z1), zb = abs_bits(*z2);
        const unsigned long long zz = za > zb ? za : zb;
        m0 = rr > m0 ? rr : m0;
        m1 = zz > m1 ? zz : m1;
        m2 = bb > m2 ? bb : m2;
    });
    atomic_max_u64(mx + 0, m0);
    atomic_max_u64(mx + 1, m1);
    atomic_max_u64(mx + 2, m2);
    wsync();
    wone([&](int) {
        atomic_max_u64(r.norms + 3LL * b + 0, mx[0]);
        atomic_max_u64(r.norms + 3LL * b + 1, mx[1]);
        atomic_max_u64(r.norms + 3LL * b + 2, mx[2]);
    });
}

// ---- the MHE-form residual in double-float arithmetic ------------------------
//
// The residual r = b - K z needs about FP64 accuracy (the refinement drives it to
// 1e-12 of ||K|| ||z||), but GB300 issues FP64 at a small fraction of its FP32
// rate.  Every FP64 input is carried as a float pair hi + lo (48 bits): the stage
// matrices as the pairs the preparation pass wrote, the vectors split here in
// integer arithmetic (f32_rn, f32_lo).  A product of two pairs keeps ah bh exactly
// (its rounding error by an FMA) and the cross terms ah bl + al bh in float; a dot
// product sums the exact ah bh in float with each addition's error recovered
// (two-sum) into a float compensation, which also takes the product errors and
// cross terms (compensated dot product in the manner of Ogita, Rump and Oishi's
// Dot2, extended to pair inputs).  The result is about as accurate as if computed
// with 48-bit significands, ample for relres 1e-12 at the refinement's ~1e-13
// floor of FP64 summation order differences.  Only the FP32 pipes are used.

// s + c += (ah + al)(bh + bl)
MHE_DEV void df_acc(float& s, float& c, float ah, float al, float bh, float bl)
{
    const float p = ah * bh;
    const float pe = fmaf(ah, bh, -p);          // ah bh - p, exactly
    const float t = s + p;
    const float z = t - s;
    const float se = (s - (t - z)) + (p - z);   // s + p - t, exactly
    s = t;
    c += se + (pe + fmaf(ah, bl, al * bh));
}

// (s, c) += (s2, c2)
MHE_DEV void df_add(float& s, float& c, float s2, float c2)
{
    const float t = s + s2;
    const float z = t - s;
    const float se = (s - (t - z)) + (s2 - z);
    s = t;
    c += se + c2;
}

// the pair (s, c) as a normalised pair (hi, lo), |lo| <= ulp(hi) / 2
MHE_DEV float2 df_norm(float s, float c)
{
    const float h = s + c;
    return make_float2(h, c - (h - s));
}

MHE_DEV float2 df_split(double v)
{
    const float h = f32_rn(v);
    return make_float2(h, f32_lo(v, h));
}

// Two double-float accumulators side by side in packed FP32 instructions: the even and the odd
// terms of a dot product, half the issue slots.
MHE_DEV F2 sub2(F2 a, F2 b) { return fma2(b, pack2(-1.f, -1.f), a); }   // exact product: one rounding, as a - b

// the sums s and their compensations: rounding errors of the sums (c) and the products' parts (d)
struct Df2 {
    F2 s, c, d;
    MHE_DEV Df2() : s(0ULL), c(0ULL), d(0ULL) {}
    // += (ah + al)(bh + bl), nb = -bh: df_acc on both halves
    MHE_DEV void acc(F2 ah, F2 al, F2 bh, F2 bl, F2 nb)
    {
        const F2 p = mul2(ah, bh);
        const F2 q = fma2(ah, nb, p);   // p - ah bh, exactly
        const F2 t = add2(s, p);
        const F2 z = sub2(t, s);
        const F2 x = sub2(s, sub2(t, z)), y = sub2(p, z);   // x + y = s + p - t, exactly
        s = t;
        c = add2(add2(c, x), y);
        d = sub2(fma2(al, bh, fma2(ah, bl, d)), q);
    }
    MHE_DEV void result(float& so, float& co) const
    {
        const float2 a = unpack2(s), e = unpack2(c), f = unpack2(d);
        so = a.x;
        co = e.x + f.x;
        df_add(so, co, a.y, e.y + f.y);
    }
};

// A vector in shared memory split for the products: hi, lo and -hi parts of n entries each, the parts
// `pitch` apart
struct DfVec {
    const float* p;
    int pitch;
};

// sum_{j < L} (mh + ml)[j sm] * v[j] as (s, c); the low parts LO floats behind the high ones.  v starts on
// an even entry when L is even (pairs are loaded at once)
template <int L, int LO>
MHE_DEV float2 dot_df(const float* m, int sm, const DfVec& v)
{
    Df2 a;
    float s, c;
#pragma unroll
    for (int j = 0; j + 1 < L; j += 2) {
        const F2 ah = pack2(m[j * sm], m[(j + 1) * sm]), al = pack2(m[j * sm + LO], m[(j + 1) * sm + LO]);
        F2 bh, bl, nb;
        if constexpr (L % 2 == 0) {
            bh = *reinterpret_cast<const F2*>(v.p + j);
            bl = *reinterpret_cast<const F2*>(v.p + v.pitch + j);
            nb = *reinterpret_cast<const F2*>(v.p + 2 * v.pitch + j);
        } else {
            bh = pack2(v.p[j], v.p[j + 1]);
            bl = pack2(v.p[v.pitch + j], v.p[v.pitch + j + 1]);
            nb = pack2(v.p[2 * v.pitch + j], v.p[2 * v.pitch + j + 1]);
        }
        a.acc(ah, al, bh, bl, nb);
    }
    a.result(s, c);
    if constexpr (L % 2 != 0)
        df_acc(s, c, m[(L - 1) * sm], m[(L - 1) * sm + LO], v.p[L - 1], v.p[v.pitch + L - 1]);
    return make_float2(s, c);
}

// the same over a contiguous segment whose start lies a multiple of the bank count (or near it) from the
// neighbouring lane's: lane q begins at entry q mod L and wraps, so the lanes' loads fall in different banks
template <int L, int LO>
MHE_DEV float2 dot_df_turn(const float* m, int q, const DfVec& v)
{
    Df2 a;
    float s, c;
    int j = q % L;
    auto next = [&]() {
        const int i = j;
        j = j + 1 == L ? 0 : j + 1;
        return i;
    };
#pragma unroll 4
    for (int k = 0; k + 1 < L; k += 2) {
        const int i0 = next(), i1 = next();
        a.acc(pack2(m[i0], m[i1]), pack2(m[i0 + LO], m[i1 + LO]), pack2(v.p[i0], v.p[i1]),
              pack2(v.p[v.pitch + i0], v.p[v.pitch + i1]), pack2(v.p[2 * v.pitch + i0], v.p[2 * v.pitch + i1]));
    }
    a.result(s, c);
    if constexpr (L % 2 != 0) {
        const int i = next();
        df_acc(s, c, m[i], m[i + LO], v.p[i], v.p[v.pitch + i]);
    }
    return make_float2(s, c);
}

// the same over a contiguous segment, in loads of VW floats (m aligned to VW floats)
template <int L, int LO, int VW>
MHE_DEV float2 dot_df_col(const float* m, const DfVec& v)
{
    if constexpr (VW == 1) {
        return dot_df<L, LO>(m, 1, v);
    } else {
        static_assert(L % VW == 0 && LO % VW == 0, "whole vectors");
        Df2 a;
#pragma unroll
        for (int j = 0; j < L; j += VW) {
            float h[VW], l[VW];
            ldv(m + j, h);
            ldv(m + LO + j, l);
#pragma unroll
            for (int q = 0; q < VW; q += 2)
                a.acc(pack2(h[q], h[q + 1]), pack2(l[q], l[q + 1]), *reinterpret_cast<const F2*>(v.p + j + q),
                      *reinterpret_cast<const F2*>(v.p + v.pitch + j + q),
                      *reinterpret_cast<const F2*>(v.p + 2 * v.pitch + j + q));
        }
        float s, c;
        a.result(s, c);
        return make_float2(s, c);
    }
}

// f(idx) for lo <= idx < hi, lanes round-robin in rounds that are not unrolled (bodies of a hundred
// instructions and more: the instruction cache), no barrier
template <class F>
MHE_DEV void rounds(int lo, int hi, F&& f)
{
#pragma unroll 1
    for (int i = lo + lane_id(); i < hi; i += MHE_TEAM) f(i);
}

// Shared memory of one team of the double-float residual (bytes).  A stage's float
// pairs come in two halves through a slot each: C and R (the products u = C x, W w,
// S^T w, then [S; V] u and C^T e) and A and B ([A | B]^T lambda, A x + B w); while one half
// is worked on the other's copies, of this stage or the team's next, are in flight.
// The FP64 vectors read to the end of a stage have a pair of slots of their own.
template <int NX, int NW, int NY>
struct DfWs {
    static constexpr int NR = NW + NY, NQ = NX + NW;
    // the length-n products are cut into SP segments of length LP (= nw when it divides n), so
    // that the tasks of a phase have about one length
    static constexpr int SP = NX % NW == 0 ? NX / NW : 1, LP = NX / SP;
    static constexpr int ldA = pick_ld(NX, vec_of<float>(NX)), ldC = pick_ld(NY, vec_of<float>(NY));
    static constexpr int vA = LP % vec_of<float>(NX) == 0 ? vec_of<float>(NX) : (LP % 2 == 0 && ldA % 2 == 0 ? 2 : 1);
    // floats: [A | B] hi, then lo
    static constexpr int oB = ldA * NX, abl = round_to(ldA * NQ, 4), ab = 2 * abl;
    // floats: C and R hi, then lo
    static constexpr int oR = round_to(ldC * NX, 4), crl = oR + round_to(NR * NR, 4), cr = 2 * crl;
    // doubles: x_t, w_t, lambda_{t+1}, split at once; lambda_t, x_{t+1}, l, a, read at the end (two slots)
    static constexpr int vec1 = round_to(NQ + NX, 2);
    static constexpr int oxn = NX, ol = oxn + NX, oa = ol + NQ, vec2 = round_to(oa + NX, 2);
    // split vectors (floats, three parts each): (x, w) and lambda_{t+1}; u and e (in col's place: they are
    // done with before col is begun).  w follows x at once when it makes the products' last segment
    static constexpr int sw0 = LP == NW ? NX : round_to(NX, 2);
    static constexpr int olam = round_to(sw0 + NW, 4), pz = olam + round_to(NX, 4), py = round_to(NY, 4), split = 3 * pz;
    // float2: partial sums and products (cx, ww, sw are done with before row is begun)
    static constexpr int row = 0, cx = 0, ww = row + (SP + 1) * NX, sw = cx + SP * NY, col = ww + NW,
                         su = col + max_int(SP * NQ, 3 * py),
                         cte = su + NW, pairs = round_to(cte + NX, 2);
    static_assert(SP * NY + NY <= (SP + 1) * NX, "cx and sw fit row");
    static constexpr int bytes = (4 * (ab + cr + split) + 8 * (vec1 + 2 * vec2) + 8 * pairs + 15) / 16 * 16;
};

// the stages of a team's share, next(b, t, N) one after another (false: no more): blocks of
// stages dealt round-robin over all teams, instances that no longer refine left out
struct StageBlocks {
    const long long* gs0;
    const int* active;
    int batch, len, b = 0;
    long long blk, stride, total, g = 0, end = 0, g0 = 0, g1 = 0;
    template <typename TR>
    MHE_DEV StageBlocks(const ResidArgs<TR>& r, long long team, long long teams)
        : gs0(r.gs0), active(r.active), batch(r.batch), blk(team - teams), stride(teams), total(r.nstages)
    {
        // eight stages a block (an instance's offsets are looked up once a block), fewer when that
        // would leave teams without a block
        const long long most = (total + teams - 1) / teams;
        len = most < 8 ? (int)most : 8;
    }
    MHE_DEV bool next(int& bo, int& t, int& N)
    {
        for (;;) {
            if (g >= end) {
                blk += stride;
                g = blk * len;
                if (g >= total) return false;
                end = g + len < total ? g + len : total;
                b = stage_instance(gs0, batch, g);
                g0 = gs0[b];
                g1 = gs0[b + 1];
            }
            while (g >= g1) {
                ++b;
                g0 = g1;
                g1 = gs0[b + 1];
            }
            if (active && !active[b]) {
                g = g1;
                continue;
            }
            bo = b;
            t = (int)(g - g0);
            N = (int)(g1 - g0);
            ++g;
            return true;
        }
    }
};

// the stages team, team + teams, .. of one instance
struct StageStride {
    int b, t, teams, N;
    MHE_DEV bool next(int& bo, int& to, int& No)
    {
        if (t >= N) return false;
        bo = b;
        to = t;
        No = N;
        t += teams;
        return true;
    }
};

// running maxima of |r| (float bits of the double-float rows, double bits of the FP64 ones), |z|, |b| (double bits)
// of one instance, merged into its norms at once
struct NormMax {
    unsigned r = 0;
    unsigned long long rd = 0, z = 0, b = 0;
    MHE_DEV void see_rd(double v) { const unsigned long long u = abs_bits(v); rd = u > rd ? u : rd; }
    MHE_DEV void see_r(float v) { const unsigned u = __float_as_uint(v) & 0x7fffffffu; r = u > r ? u : r; }
    MHE_DEV void see_z(double v) { const unsigned long long u = abs_bits(v); z = u > z ? u : z; }
    MHE_DEV void see_b(double v) { const unsigned long long u = abs_bits(v); b = u > b ? u : b; }
    MHE_DEV void flush(unsigned long long* norms)
    {
        constexpr int CW = MHE_TEAM < 32 ? MHE_TEAM : 32;
        const unsigned mask =
            CW == 32 ? 0xffffffffu : (((1u << CW) - 1u) << ((threadIdx.x & 31) & ~(CW - 1)));
        const unsigned long long rf = abs_bits(f64_of(__uint_as_float(r)));
        unsigned long long m[3] = {rf > rd ? rf : rd, z, b};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
#pragma unroll
            for (int d = CW / 2; d > 0; d /= 2) {
                const unsigned long long o = __shfl_xor_sync(mask, m[k], d, CW);
                m[k] = o > m[k] ? o : m[k];
            }
            if ((lane_id() & (CW - 1)) == 0 && m[k]) atomic_max_u64(norms + k, m[k]);
        }
        r = 0;
        rd = z = b = 0;
    }
};

// The arrival stage t = 0 (A_0 = B_0 = I, Q_0 = diag(0, P~0^{-1}), l_0 = a_0 = 0) in FP64, and the initial rows
template <int NX>
MHE_DEV void resid_arrival(const ResidArgs<float>& r, int b, int N, NormMax& mx)
{
    const long long gx = r.gs0[b] + b;
    const double *xt = r.x + gx * NX, *lt = r.lam + gx * NX, *wt = r.w + r.w_off[b];
    const double* P0 = r.P0inv + (long long)b * NX * NX;
    each<NX>([&](int i) {
        const double x = xt[i], xn = xt[NX + i], l = lt[i], ln = lt[NX + i], w = wt[i], x0 = r.x0[(long long)b * NX + i];
        double q = ln;
#pragma unroll 4
        for (int j = 0; j < NX; ++j) q = fma(P0[i + j * NX], wt[j], q);
        const double rx = ln - l, rd = x + w - xn, ri = x0 - x;
        r.rl0[(long long)b * 2 * NX + i] = f32_rn(rx);
        r.rl0[(long long)b * 2 * NX + NX + i] = f32_rn(q);
        r.ra0[(long long)b * NX + i] = f32_rn(rd);
        r.rx0[(long long)b * NX + i] = f32_rn(ri);
        mx.see_rd(rx); mx.see_rd(q); mx.see_rd(rd); mx.see_rd(ri);
        mx.see_z(x); mx.see_z(l); mx.see_z(w);
        mx.see_b(x0);
        if (N == 1) {   // terminal rows: -(0 - lambda_N)
            r.rlN[(long long)b * NX + i] = f32_rn(-ln);
            mx.see_rd(ln);
            mx.see_z(xn); mx.see_z(ln);
        }
    });
}

// The MHE-form residual with FP32 correction solves over the stages `it` yields.
// Per stage t >= 1 (the tasks of resid_mhe, each a double-float dot product):
//   C and R:  u = C x,  W w,  S^T w;   then  S u,  e = V u - S^T w;   then  C^T e;
//   A and B:  A x + B w,  A^T lambda_{t+1},  B^T lambda_{t+1};   then the rows.
// What bounds it: HBM has 15.4 KB a stage to deliver at nx = 24 (1.2 ms for 535k stages); the products are
// 2880 double-float terms of 12 packed instructions for two, so the nine to ten teams an SM holds
// are now bound by the latency of their dependent sums (ncu: 46% issue, 51% DRAM).  Full pass, before
// (a stage's tasks read straight from global memory, scalar instructions) and after: nx = 24, 535k
// stages, 2.63 -> 1.95 ms; nx = 12, 1.05M stages, 2.13 -> 1.21 ms; nx = 6, 1.10M stages, 0.97 -> 0.54 ms; nx = 64,
// 131k stages, 4.09 -> 3.17 ms (3.97 before S^T w took its columns turned: 32-way bank conflicts).
template <int NX, int NW, int NY, class IT>
MHE_DEV void resid_df_run(const ResidArgs<float>& r, IT& it, unsigned char* smem)
{
    using S = DfWs<NX, NW, NY>;
    constexpr int NR = S::NR, NQ = S::NQ, SP = S::SP, LP = S::LP, ldA = S::ldA, ldC = S::ldC;
    constexpr int aB = piece_of(4 * S::oB), aR = piece_of(4 * NR * NR);
    float* cr = reinterpret_cast<float*>(smem);
    float* ab = cr + S::cr;
    float* sz = ab + S::ab;           // split (x, w), lambda
    double* vi = reinterpret_cast<double*>(sz + S::split);
    double* vec0 = vi + S::vec1;
    float2* pr = reinterpret_cast<float2*>(vec0 + 2 * S::vec2);
    float* su = reinterpret_cast<float*>(pr + S::col);   // split u, e
    auto put = [](float* p, int pitch, int k, const float2& v) {
        p[k] = v.x;
        p[pitch + k] = v.y;
        p[2 * pitch + k] = -v.x;
    };
    auto zv = [&](int k) { return DfVec{sz + k, S::pz}; };
    auto yv = [&](int e) { return DfVec{su + e * 3 * S::py, S::py}; };
    NormMax mx;
    int b = 0, t = 0, N = 0;
    bool have;
    // the team's next stage t >= 1; arrival stages are evaluated on the way
    auto advance = [&]() {
        for (;;) {
            have = it.next(b, t, N);
            if (!have || t > 0) return;
            NormMax am;
            resid_arrival<NX>(r, b, N, am);
            am.flush(r.norms + 3LL * b);
        }
    };
    auto load_cr = [&](double* v) {
        const long long s = r.in_off[b] + t - 1, gx = r.gs0[b] + b + t;
        async_block<float, NY, NX, ldC>(cr, r.Chi + s * NY * NX);
        async_block<float, NR, NR, NR, NR, aR>(cr + S::oR, r.Rhi + s * NR * NR);
        async_block<float, NY, NX, ldC>(cr + S::crl, r.Clo + s * NY * NX);
        async_block<float, NR, NR, NR, NR, aR>(cr + S::crl + S::oR, r.Rlo + s * NR * NR);
        async_vec<double, NX>(vi, r.x + gx * NX);
        async_vec<double, NW>(vi + NX, r.w + r.w_off[b] + NX + (long long)(t - 1) * NW);
        async_vec<double, NX>(vi + NQ, r.lam + (gx + 1) * NX);
        async_vec<double, NX>(v, r.lam + gx * NX);
        async_vec<double, NX>(v + S::oxn, r.x + (gx + 1) * NX);
        async_vec<double, NQ>(v + S::ol, r.l ? r.l + s * NQ : nullptr);
        async_vec<double, NX>(v + S::oa, r.a ? r.a + s * NX : nullptr);
    };
    auto load_ab = [&]() {
        const long long s = r.in_off[b] + t - 1;
        async_block<float, NX, NX, ldA>(ab, r.Ahi + s * NX * NX);
        async_block<float, NX, NW, ldA, NX, aB>(ab + S::oB, r.Bhi + s * NX * NW);
        async_block<float, NX, NX, ldA>(ab + S::abl, r.Alo + s * NX * NX);
        async_block<float, NX, NW, ldA, NX, aB>(ab + S::abl + S::oB, r.Blo + s * NX * NW);
    };
    advance();
    int par = 0;
    if (have) load_cr(vec0);
    cp_commit();
    while (have) {
        const double* v = vec0 + par * S::vec2;
        load_ab();
        cp_commit();
        const int sb = b, st = t;
        const bool lastst = t == N - 1;
        cp_wait<1>();
        wsync();
        // ---- C and R
        rounds(0, NQ + NX, [&](int k) {
            const double z = vi[k];
            put(sz, S::pz, k < NX ? k : (k < NQ ? S::sw0 + k - NX : S::olam + k - NQ), df_split(z));
            if (k < NQ || lastst) mx.see_z(z);
        });
        wsync();
        // segments of C x, then W w and S^T w (the first nw entries of column nw + k of R)
        // (at nx >= 48 a column of R is a multiple of the banks long: S^T w goes apart, turned)
        constexpr bool turn = NR % 32 == 0;
        if constexpr (turn)
            rounds(0, NY, [&](int k) {
                pr[S::sw + k] = dot_df_turn<NW, S::crl>(cr + S::oR + (NW + k) * NR, k, zv(S::sw0));
            });
        if constexpr (LP == NW) {
            rounds(0, NY * SP + NW + (turn ? 0 : NY), [&](int k) {
                const float* m;
                int sm, j0, o;
                if (k < NY * SP) {
                    j0 = (k / NY) * LP;
                    m = cr + k % NY + j0 * ldC;
                    sm = ldC;
                    o = S::cx + k;
                } else if (k < NY * SP + NW) {
                    const int q = k - NY * SP;
                    m = cr + S::oR + q;
                    sm = NR;
                    j0 = NX;
                    o = S::ww + q;
                } else {
                    const int q = k - NY * SP - NW;
                    m = cr + S::oR + (NW + q) * NR;
                    sm = 1;
                    j0 = NX;
                    o = S::sw + q;
                }
                pr[o] = dot_df<LP, S::crl>(m, sm, zv(j0));
            });
        } else {
            rounds(0, NY * SP, [&](int k) {
                const int j0 = (k / NY) * LP;
                pr[S::cx + k] = dot_df<LP, S::crl>(cr + k % NY + j0 * ldC, ldC, zv(j0));
            });
            rounds(0, turn ? NW : NR, [&](int k) {
                const bool w = k < NW;
                pr[w ? S::ww + k : S::sw + k - NW] =
                    dot_df<NW, S::crl>(cr + S::oR + (w ? k : k * NR), w ? NR : 1, zv(S::sw0));
            });
        }
        wsync();
        rounds(0, NY, [&](int k) {
            float s = pr[S::cx + k].x, c = pr[S::cx + k].y;
#pragma unroll
            for (int q = 1; q < SP; ++q) df_add(s, c, pr[S::cx + q * NY + k].x, pr[S::cx + q * NY + k].y);
            put(su, S::py, k, df_norm(s, c));
        });
        wsync();
        rounds(0, NR, [&](int k) {   // row k of [S; V] u;  e = V u - S^T w
            const float2 d = dot_df<NY, S::crl>(cr + S::oR + k + NW * NR, NR, yv(0));
            if (k < NW) {
                pr[S::su + k] = d;
            } else {
                float s = d.x, c = d.y;
                df_add(s, c, -pr[S::sw + k - NW].x, -pr[S::sw + k - NW].y);
                put(su + 3 * S::py, S::py, k - NW, df_norm(s, c));
            }
        });
        wsync();
        rounds(0, NX, [&](int i) {   // C^T e
            pr[S::cte + i] = dot_df_col<NY, S::crl, NY % 2 == 0 ? vec_of<float>(NY) : 1>(cr + i * ldC, yv(1));
        });
        wsync();   // the C and R slot is free
        advance();
        par ^= 1;
        if (have) load_cr(vec0 + par * S::vec2);
        cp_commit();
        cp_wait<1>();
        wsync();
        // ---- A and B: row i of [A | B] with (x, w), in segments (the last one B w)
        constexpr int nrow = NX * (SP + 1), ncol = NQ * SP, T = MHE_TEAM;
        // whole rounds of either kind, then the rest of both in one round with the stride chosen per lane
        constexpr bool mixed = LP == NW && nrow % T + ncol % T <= T && nrow % T > 0 && ncol % T > 0;
        constexpr int row1 = mixed ? nrow / T * T : nrow, col1 = mixed ? ncol / T * T : ncol;
        rounds(0, row1, [&](int k) {
            const int i = k % NX, j0 = (k / NX) * LP;
            if constexpr (LP == NW) {
                pr[S::row + k] = dot_df<LP, S::abl>(ab + i + j0 * ldA, ldA, zv(j0));
            } else {
                if (k < NX * SP) pr[S::row + k] = dot_df<LP, S::abl>(ab + i + j0 * ldA, ldA, zv(j0));
                else pr[S::row + k] = dot_df<NW, S::abl>(ab + S::oB + i, ldA, zv(S::sw0));
            }
        });
        // column i of [A | B] with lambda_{t+1}, in segments
        rounds(0, col1, [&](int k) {
            const int i = k % NQ, j0 = (k / NQ) * LP;
            pr[S::col + k] = dot_df_col<LP, S::abl, LP % 2 == 0 ? S::vA : 1>(ab + i * ldA + j0, zv(S::olam + j0));
        });
        if constexpr (mixed) {
            rounds(0, nrow - row1 + ncol - col1, [&](int k) {
                const bool rw = k < nrow - row1;
                const int q = rw ? row1 + k : col1 + k - (nrow - row1);
                const int i = rw ? q % NX : q % NQ, j0 = (rw ? q / NX : q / NQ) * LP;
                pr[rw ? S::row + q : S::col + q] = dot_df<LP, S::abl>(ab + (rw ? i + j0 * ldA : i * ldA + j0),
                                                                     rw ? ldA : 1, zv(rw ? j0 : S::olam + j0));
            });
        }
        wsync();
        // ---- the rows: r = -(l + K z)
        const long long so = r.out_off[sb] + st - 1;
        float *rl = r.rl + so * NQ, *ra = r.ra + so * NX;
        rounds(0, NX, [&](int i) {   // C^T e + A^T lambda_{t+1} - lambda_t + l_x
            const double l = v[S::ol + i], lt = v[i];
            const float2 v4 = df_split(l - lt);
            float s = v4.x, c = v4.y;
            df_add(s, c, pr[S::cte + i].x, pr[S::cte + i].y);
#pragma unroll
            for (int q = 0; q < SP; ++q) df_add(s, c, pr[S::col + q * NQ + i].x, pr[S::col + q * NQ + i].y);
            rl[i] = s + c;
            mx.see_r(s + c);
            mx.see_z(lt);
            mx.see_b(l);
        });
        rounds(0, NW, [&](int i) {   // W w - S u + B^T lambda_{t+1} + l_w
            const double l = v[S::ol + NX + i];
            const float2 v4 = df_split(l);
            float s = v4.x, c = v4.y;
            df_add(s, c, pr[S::ww + i].x, pr[S::ww + i].y);
#pragma unroll
            for (int q = 0; q < SP; ++q) df_add(s, c, pr[S::col + q * NQ + NX + i].x, pr[S::col + q * NQ + NX + i].y);
            df_add(s, c, -pr[S::su + i].x, -pr[S::su + i].y);
            rl[NX + i] = s + c;
            mx.see_r(s + c);
            mx.see_b(l);
        });
        rounds(0, NX, [&](int i) {   // A x + B w - x_{t+1} + a
            const double a = v[S::oa + i], xn = v[S::oxn + i];
            const float2 v4 = df_split(a - xn);
            float s = v4.x, c = v4.y;
#pragma unroll
            for (int q = 0; q <= SP; ++q) df_add(s, c, pr[S::row + q * NX + i].x, pr[S::row + q * NX + i].y);
            ra[i] = s + c;
            mx.see_r(s + c);
            mx.see_b(a);
            if (lastst) {   // terminal rows with Q_{x,N} = 0, l_N = 0: r = lambda_N
                const float ln = sz[S::olam + i] + sz[S::pz + S::olam + i];
                r.rlN[(long long)sb * NX + i] = -ln;
                mx.see_r(ln);
                mx.see_z(xn);
            }
        });
        if (!have || b != sb) mx.flush(r.norms + 3LL * sb);
        wsync();   // the A and B slot and the products are free
    }
    cp_wait<0>();
}

// Stage t >= 1 with the assembled Q: the same rows as resid_rows, as dot
// products of length n or nw dealt round-robin to the lanes (each Q row is
// split into its x and w halves) and one predicated FMA loop, then the rows
//   Q_x x + Q_xw w + A^T lam_{t+1} - lam_t + l_x,  Q_xw^T x + Q_w w + B^T lam_{t+1} + l_w,
//   A x + B w + a - x_{t+1}  (and the terminal rows at t = N - 1).
template <int NX, int NW, typename TR>
MHE_DEV void resid_q(const ResidArgs<TR>& r, int b, int t, int N, unsigned long long* sm)
{
    constexpr int NQ = NX + NW;
    const long long gx = r.gs0[b] + b;
    const double* xt = r.x + (gx + t) * NX;
    const double* xn = xt + NX;
    const double* lt = r.lam + (gx + t) * NX;
    const double* ln = lt + NX;
    const double* wt = r.w + r.w_off[b] + NX + (long long)(t - 1) * NW;
    const long long s = r.in_off[b] + t - 1;
    const double* A = r.A + s * NX * NX;
    const double* B = r.B + s * NX * NW;
    const double* Q = r.Q + s * NQ * NQ;
    const double* l = r.l ? r.l + s * NQ : nullptr;
    const double* a = r.a ? r.a + s * NX : nullptr;
    const long long so = r.out_off[b] + t - 1;
    TR* rl = r.rl + so * NQ;
    TR* ra = r.ra + so * NX;
    const bool lastst = (t == N - 1);
    double* qx = reinterpret_cast<double*>(sm);   // Q[:, 0:n] x      (NQ)
    double* qw = qx + NQ;                         // Q[:, n:n+nw] w   (NQ)
    double* atl = qw + NQ;                        // A^T lam_{t+1}    (NX)
    double* btl = atl + NX;                       // B^T lam_{t+1}    (NW)
    double* dA = btl + NW;                        // A x              (NX)
    double* dB = dA + NX;                         // B w              (NX)
    double* zero = dB + NX;
    unsigned long long* mx = reinterpret_cast<unsigned long long*>(zero + 1);
    wone([&](int) {
        zero[0] = 0.0;
        mx[0] = mx[1] = mx[2] = 0ULL;
    });
    constexpr int T1 = NQ + NX + NW + NX;   // length-n tasks, then length-nw tasks
    wfor(T1 + NQ + NX, [&](int k) {
        const double* m;
        const double* v;
        double* o;
        int st, len = NX;
        if (k < NQ) { m = Q + k; st = NQ; v = xt; o = qx + k; }
        else if (k < NQ + NX) { m = A + (k - NQ) * NX; st = 1; v = ln; o = atl + (k - NQ); }
        else if (k < NQ + NX + NW) { m = B + (k - NQ - NX) * NX; st = 1; v = ln; o = btl + (k - NQ - NX); }
        else if (k < T1) { m = A + (k - NQ - NX - NW); st = NX; v = xt; o = dA + (k - NQ - NX - NW); }
        else if (k < T1 + NQ) { m = Q + (k - T1) + NX * NQ; st = NQ; v = wt; o = qw + (k - T1); len = NW; }
        else { m = B + (k - T1 - NQ); st = NX; v = wt; o = dB + (k - T1 - NQ); len = NW; }
        *o = dot_pred<(NX > NW ? NX : NW)>(m, st, v, len, 0.0);
    });
    unsigned long long m0 = 0, m1 = 0, m2 = 0;
    const int nrow = NQ + NX + (lastst ? NX : 0);
    const double* xN = r.x + (gx + N) * NX;
    const double* lamN = r.lam + (gx + N) * NX;
    wfor(nrow, [&](int i) {
        const double *p1, *p2, *p3, *p4, *p5, *z1, *z2;
        TR* dst;
        if (i < NX) {
            p1 = qx + i; p2 = qw + i; p3 = atl + i; p4 = lt + i; p5 = l ? l + i : zero;
            z1 = xt + i; z2 = lt + i; dst = rl + i;
        } else if (i < NQ) {
            p1 = qx + i; p2 = qw + i; p3 = btl + (i - NX); p4 = zero; p5 = l ? l + i : zero;
            z1 = wt + (i - NX); z2 = zero; dst = rl + i;
        } else if (i < NQ + NX) {
            const int ii = i - NQ;
            p1 = dA + ii; p2 = dB + ii; p3 = zero; p4 = xn + ii; p5 = a ? a + ii : zero;
            z1 = zero; z2 = zero; dst = ra + ii;
        } else {
            // terminal rows with Q_{x,N} = 0, l_N = 0: r = lambda_N
            const int ii = i - NQ - NX;
            p1 = zero; p2 = zero; p3 = zero; p4 = lamN + ii; p5 = zero;
            z1 = xN + ii; z2 = lamN + ii; dst = r.rlN + (long long)b * NX + ii;
        }
        const double sum = *p5 + (((*p1 + *p2) + *p3) - *p4);   // r = -(l + K z)
        *dst = to_tr<TR>(sum);
        const unsigned long long rr = abs_bits(sum), bb = abs_bits(*p5);
        const unsigned long long za = abs_bits(*z1), zb = abs_bits(*z2);
        const unsigned long long zz = za > zb ? za : zb;
        m0 = rr > m0 ? rr : m0;
        m1 = zz > m1 ? zz : m1;
        m2 = bb > m2 ? bb : m2;
    });
    atomic_max_u64(mx + 0, m0);
    atomic_max_u64(mx + 1, m1);
    atomic_max_u64(mx + 2, m2);
    wsync();
    wone([&](int) {
        atomic_max_u64(r.norms + 3LL * b + 0, mx[0]);
        atomic_max_u64(r.norms + 3LL * b + 1, mx[1]);
        atomic_max_u64(r.norms + 3LL * b + 2, mx[2]);
    });
}

template <int NX, int NW, typename TR, int NY = 0>
MHE_DEV void resid_stage(const ResidArgs<TR>& r, long long gstage, unsigned long long* sm)
{
    const int b = stage_instance(r.gs0, r.batch, gstage);
    if (r.active && !r.active[b]) return;
    const int t = (int)(gstage - r.gs0[b]);
    const int N = (int)(r.gs0[b + 1] - r.gs0[b]);
    if (t == 0) {
        resid_rows<NX, NW, 1, TR>(r, b, t, N, sm);
    } else {
        if constexpr (NY > 0) {
            resid_mhe<NX, NW, NY, TR>(r, b, t, N, sm);
        } else {
            resid_q<NX, NW, TR>(r, b, t, N, sm);
        }
    }
}

// ||K||_inf contribution of one stage: absolute row sums (in float) of the KKT
// rows the residual above evaluates; one atomic max per stage.
template <int NX, int NW>
MHE_DEV void knorm_stage(const KnormArgs& r, long long gstage, float* sm)
{
    const int b = stage_instance(r.gs0, r.batch, gstage);
    const int t = (int)(gstage - r.gs0[b]);
    constexpr int NQ = NX + NW;
    if (t == 0) {
        // arrival stage: x rows 1 + 1, w rows |P~0^{-1} row| + 1, dynamics rows 3, initial row 1
        const double* P0 = r.P0inv + (long long)b * NX * NX;
        wfor(NX, [&](int i) {
            float rs = 1.f;
            for (int j = 0; j < NX; ++j) rs += abs_to_float(P0[i + j * NX]);
            sm[i] = rs > 3.f ? rs : 3.f;
        });
        wone([&](int) {
            float m = 0.f;
            for (int i = 0; i < NX; ++i) m = sm[i] > m ? sm[i] : m;
            atomic_max_u32(r.kinf + b, float_bits(m));
        });
        return;
    }
    const long long s = r.in_off[b] + t - 1;
    const double* A = r.A + s * NX * NX;
    const double* B = r.B + s * NX * NW;
    const double* Q = r.Q + s * NQ * NQ;
    wfor(NQ + NX, [&](int i) {
        float rs;
        if (i < NQ) {
            rs = (i < NX) ? 1.f : 0.f;
            for (int j = 0; j < NQ; ++j) rs += abs_to_float(Q[i + j * NQ]);
            if (i < NX) for (int j = 0; j < NX; ++j) rs += abs_to_float(A[j + i * NX]);
            else for (int j = 0; j < NX; ++j) rs += abs_to_float(B[j + (i - NX) * NX]);
        } else {
            const int ii = i - NQ;
            rs = 1.f;
            for (int j = 0; j < NX; ++j) rs += abs_to_float(A[ii + j * NX]);
            for (int j = 0; j < NW; ++j) rs += abs_to_float(B[ii + j * NX]);
        }
        sm[i] = rs;
    });
    wone([&](int) {
        float m = 1.f;
        for (int i = 0; i < NQ + NX; ++i) m = sm[i] > m ? sm[i] : m;
        atomic_max_u32(r.kinf + b, float_bits(m));
    });
}

// ---- Section II: MHE stage weights -> UFTOC Q_t, l_t, c_t ---------------------
// R = [[W, S], [S^T, V]] ((nw+ny)^2), S the nw x ny block:
//   Q = [[C^T V C, -C^T S^T], [-S C, W]],  l = [C^T (S^T w~ - V y~); S y~ - W w~],
//   c = 1/2 w~^T W w~ - y~^T S^T w~ + 1/2 y~^T V y~.
template <int NX, int NW, int NY>
struct AsmSmem {
    static constexpr int NR = NW + NY;
    static constexpr int count = NY * NX + NR * NR + NY * NX + NW * NX + NY + NW + NY + NW + 8;
};

template <int NX, int NW, int NY>
MHE_DEV void assemble_stage(const double* C, const double* R, const double* yt, const double* wt,
                            double* Q, double* l, double* c, double* sm)
{
    constexpr int NR = NW + NY, NQ = NX + NW;
    double* sC = sm;
    double* sR = sC + NY * NX;
    double* sVC = sR + NR * NR;
    double* sSC = sVC + NY * NX;
    double* sy = sSC + NW * NX;
    double* sw = sy + NY;
    double* st = sw + NW;   // NY + NW
    wfor(NY * NX + NR * NR + NY + NW, [&](int idx) {
        if (idx < NY * NX) sC[idx] = C[idx];
        else if (idx < NY * NX + NR * NR) sR[idx - NY * NX] = R[idx - NY * NX];
        else if (idx < NY * NX + NR * NR + NY) sy[idx - NY * NX - NR * NR] = yt[idx - NY * NX - NR * NR];
        else sw[idx - NY * NX - NR * NR - NY] = wt[idx - NY * NX - NR * NR - NY];
    });
    // V(p,r) = R[NW+p + (NW+r) NR], S(i,r) = R[i + (NW+r) NR], W(i,j) = R[i + j NR]
    wfor(NY * NX + NW * NX + NY + NW, [&](int idx) {
        if (idx < NY * NX) {
            int p = idx % NY, j = idx / NY;
            double acc = 0;
            for (int q = 0; q < NY; ++q) acc += sR[NW + p + (NW + q) * NR] * sC[q + j * NY];
            sVC[p + j * NY] = acc;
        } else if (idx < NY * NX + NW * NX) {
            int r = idx - NY * NX, i = r % NW, j = r / NW;
            double acc = 0;
            for (int q = 0; q < NY; ++q) acc += sR[i + (NW + q) * NR] * sC[q + j * NY];
            sSC[i + j * NW] = acc;
        } else if (idx < NY * NX + NW * NX + NY) {
            int p = idx - NY * NX - NW * NX;
            double acc = 0;
            for (int q = 0; q < NW; ++q) acc += sR[q + (NW + p) * NR] * sw[q];        // S^T w~
            for (int q = 0; q < NY; ++q) acc -= sR[NW + p + (NW + q) * NR] * sy[q];   // V y~
            st[p] = acc;
        } else {
            int i = idx - NY * NX - NW * NX - NY;
            double acc = 0;
            for (int q = 0; q < NY; ++q) acc += sR[i + (NW + q) * NR] * sy[q];        // S y~
            for (int q = 0; q < NW; ++q) acc -= sR[i + q * NR] * sw[q];               // W w~
            st[NY + i] = acc;
        }
    });
    wfor(NQ * NQ + NQ + (c ? 1 : 0), [&](int idx) {
        if (idx < NQ * NQ) {
            int i = idx % NQ, j = idx / NQ;
            double v;
            if (i < NX && j < NX) {
                v = 0;
                for (int p = 0; p < NY; ++p) v += sC[p + i * NY] * sVC[p + j * NY];
            } else if (i < NX) v = -sSC[(j - NX) + i * NW];
            else if (j < NX) v = -sSC[(i - NX) + j * NW];
            else v = sR[(i - NX) + (j - NX) * NR];
            Q[idx] = v;
        } else if (idx < NQ * NQ + NQ) {
            int i = idx - NQ * NQ;
            double v;
            if (i < NX) {
                v = 0;
                for (int p = 0; p < NY; ++p) v += sC[p + i * NY] * st[p];
            } else v = st[NY + (i - NX)];
            l[i] = v;
        } else {
            double ww = 0, ys = 0, yy = 0;
            for (int i = 0; i < NW; ++i)
                for (int j = 0; j < NW; ++j) ww += sw[i] * sR[i + j * NR] * sw[j];
            for (int i = 0; i < NW; ++i)
                for (int p = 0; p < NY; ++p) ys += sw[i] * sR[i + (NW + p) * NR] * sy[p];
            for (int p = 0; p < NY; ++p)
                for (int q = 0; q < NY; ++q) yy += sy[p] * sR[NW + p + (NW + q) * NR] * sy[q];
            *c = 0.5 * ww - ys + 0.5 * yy;
        }
    });
}

// ---- Section II in one pass: MHE data -> FP32 working copies -----------------
// Per stage t >= 1: A, B, a rounded to FP32; Q of the stage assembled in FP32
// from FP32 copies of C and R (it only feeds the FP32 factorisation, whose
// error the FP64 refinement removes); the linear term l in FP64 (it is part of
// the right-hand side the residual is measured against) and its FP32 copy; the
// stage's rows of ||K||_inf.  Per arrival stage: FP32 copies of P~0^{-1} and
// x~0 and their rows of ||K||_inf.  The constant c is not formed.
// One batched load of every input block, register-tiled FP32 products, and the
// FP64 dot products of l dealt to lanes without branch divergence.
template <int NX, int NW, int NY>
struct PrepSmem {
    static constexpr int NR = NW + NY, NQ = NX + NW;
    static constexpr int nd = NY + NW + NY;   // doubles: y~, w~, t = S^T w~ - V y~
    // floats: C and V C by columns, R by rows (its rows are the products' contiguous operand); A and B
    // (odd leading dimension: read along rows and columns) for their row sums, then Q in their place
    static constexpr int ldC = pick_ld(NY, vec_of<float>(NY)), ldR = pick_ld(NR, vec_of<float>(NR)), ldA = NX | 1;
    static constexpr int oC = round_to(nd, 2) * 2, oVC = oC + round_to(ldC * NX, 4), oR = oVC + round_to(ldC * NX, 4),
                         oQ = oR + round_to(ldR * NR, 4), oB = oQ + ldA * NX;
    static constexpr int nq = max_int(NQ * NQ, ldA * NQ);
    static constexpr int count = (oQ + round_to(nq, 4)) / 2;   // 8-byte words
    static_assert(NW % vec_of<float>(NY) == 0, "the S and V parts of a row of R start on a whole vector");
};

// f(i, src[i]) for i < COUNT, lanes round-robin, the next loads of a lane (MOST of them) in flight while it works
// on as many.  The rounds are not unrolled: a preparation stage unrolled in full outgrows the instruction cache
// (at nx = 64 ten of thirteen warp cycles per instruction went into waiting for instructions).  MOST: nx = 24,
// 535k stages, 4.09 ms with 4, 3.51 with 6, 4.01 with 12; nx = 64, 131k stages, 11.42 with 2, 9.82 with 4, 10.94 with
// 6, 11.86 with 12.
template <int COUNT, class F>
MHE_DEV void stream_in(const double* src, F&& f)
{
    constexpr int PER = (COUNT + MHE_TEAM - 1) / MHE_TEAM, MOST = MHE_TEAM >= 128 ? 4 : 6, CH = PER < MOST ? PER : MOST, NB = (PER + CH - 1) / CH;
    double cur[CH], nxt[CH];
    auto load = [&](double (&v)[CH], int k0) {
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int i = lane_id() + MHE_TEAM * (k0 + k);
            v[k] = i < COUNT ? src[i] : 0.0;
        }
    };
    load(cur, 0);
#pragma unroll 1
    for (int c = 0; c < NB; ++c) {
        if (c + 1 < NB) load(nxt, (c + 1) * CH);
#pragma unroll
        for (int k = 0; k < CH; ++k) {
            const int i = lane_id() + MHE_TEAM * (c * CH + k);
            if (i < COUNT) f(i, cur[k]);
            cur[k] = nxt[k];
        }
    }
}

template <int NX, int NW, int NY>
MHE_DEV void prep_stage(const PrepArgs& p, long long gstage, double* sm)
{
    using PS = PrepSmem<NX, NW, NY>;
    constexpr int NR = NW + NY, NQ = NX + NW;
    constexpr int ldC = PS::ldC, ldR = PS::ldR, ldA = PS::ldA;
    const int b = stage_instance(p.gs0, p.batch, gstage);
    const int t = (int)(gstage - p.gs0[b]);
    double* dy = sm;
    double* dw = dy + NY;
    double* dt = dw + NW;
    float* sf = reinterpret_cast<float*>(sm);
    float *fC = sf + PS::oC, *fVC = sf + PS::oVC, *fR = sf + PS::oR, *fQ = sf + PS::oQ;
    float *fA = fQ, *fB = sf + PS::oB;
    // the largest row sum of this lane, merged over the team into the instance's ||K||_inf
    auto merge = [&](float m) {
        constexpr int CW = MHE_TEAM < 32 ? MHE_TEAM : 32;
        const unsigned mask =
            CW == 32 ? 0xffffffffu : (((1u << CW) - 1u) << ((threadIdx.x & 31) & ~(CW - 1)));
        unsigned u = float_bits(m);
#pragma unroll
        for (int d = CW / 2; d > 0; d /= 2) {
            const unsigned o = __shfl_xor_sync(mask, u, d, CW);
            u = o > u ? o : u;
        }
        if ((lane_id() & (CW - 1)) == 0) atomic_max_u32(p.kinf + b, u);
    };
    if (t == 0) {
        // arrival stage: x rows 1 + 1, w rows |P~0^{-1} row| + 1, dynamics rows 3, initial row 1
        const double* P0 = p.P0inv + (long long)b * NX * NX;
        float* P0f = p.P0_32 + (long long)b * NX * NX;
        wcopy<NX * NX>([&](int i) { return P0[i]; }, [&](int i, double v) {
            const float f = f32_rn(v);
            P0f[i] = f;
            fA[i % NX + (i / NX) * ldA] = f;
        });
        float m = 3.f;
        each<NX>([&](int i) {
            p.x0_32[(long long)b * NX + i] = f32_rn(p.x0[(long long)b * NX + i]);
            float rs = 1.f;
            for (int j = 0; j < NX; ++j) rs += mabs(fA[i + j * ldA]);
            m = rs > m ? rs : m;
        });
        wsync();
        merge(m);
        return;
    }
    const long long s = p.in_off[b] + t - 1;
    const double *A = p.A + s * NX * NX, *B = p.B + s * NX * NW, *C = p.C + s * NY * NX, *R = p.R + s * NR * NR;
    const double *yt = p.yt + s * NY, *wt = p.wt + s * NW, *av = p.a + s * NX;
    float *A32 = p.A32 + s * NX * NX, *B32 = p.B32 + s * NX * NW, *a32 = p.a32 + s * NX;
    // the double-float pairs of the residual (when asked for): hi = the FP32 rounding, lo = the rest
    const bool pairs = p.A_lo != nullptr;
    float* Qo = p.Q32 + s * NQ * NQ;
    double* lo = p.l + s * NQ;
    float* lo32 = p.l32 + s * NQ;
    // every block of the stage on its way to L2 before the first is read
    prefetch_l2(C, 8 * NY * NX);
    prefetch_l2(R, 8 * NR * NR);
    prefetch_l2(A, 8 * NX * NX);
    prefetch_l2(B, 8 * NX * NW);
    each<NY>([&](int i) { dy[i] = yt[i]; });
    each<NW>([&](int i) { dw[i] = wt[i]; });
    each<NX>([&](int i) { a32[i] = f32_rn(av[i]); });
    auto pair_out = [&](float* ho, float* lo_, int i, double v) -> float {
        float h, l;
        f32_pair(v, h, l);
        if (ho) ho[i] = h;
        if (lo_) lo_[i] = l;
        return h;
    };
    float *Ch = pairs ? p.C_hi + s * NY * NX : nullptr, *Cl = pairs ? p.C_lo + s * NY * NX : nullptr;
    float *Rh = pairs ? p.R_hi + s * NR * NR : nullptr, *Rl = pairs ? p.R_lo + s * NR * NR : nullptr;
    float *Al = pairs ? p.A_lo + s * NX * NX : nullptr, *Bl = pairs ? p.B_lo + s * NX * NW : nullptr;
    stream_in<NY * NX>(C, [&](int i, double v) { fC[i % NY + (i / NY) * ldC] = pair_out(Ch, Cl, i, v); });
    stream_in<NR * NR>(R, [&](int i, double v) { fR[i / NR + (i % NR) * ldR] = pair_out(Rh, Rl, i, v); });
    stream_in<NX * NX>(A, [&](int i, double v) { fA[i % NX + (i / NX) * ldA] = pair_out(A32, Al, i, v); });
    stream_in<NX * NW>(B, [&](int i, double v) { fB[i % NX + (i / NX) * ldA] = pair_out(B32, Bl, i, v); });
    wsync();
    // rows of ||K||_inf, the A and B parts: stationarity rows (a column of A or B, and -lambda_t; the Q part
    // follows) and dynamics rows (a row of A and of B, and -x_{t+1})
    constexpr int RS = (NQ + MHE_TEAM - 1) / MHE_TEAM;
    float rs[RS], m = 1.f;
#pragma unroll
    for (int k = 0; k < RS; ++k) {
        const int i = lane_id() + k * MHE_TEAM;
        rs[k] = i < NX ? 1.f : 0.f;
        if (i < NQ) {
#pragma unroll 8
            for (int j = 0; j < NX; ++j) rs[k] += mabs(fA[j + i * ldA]);   // (B follows A)
        }
    }
    each<NX>([&](int i) {
        float r = 1.f;
#pragma unroll 8
        for (int j = 0; j < NQ; ++j) r += mabs(fA[i + j * ldA]);
        m = r > m ? r : m;
    });
    // FP64: t = S^T w~ - V y~ (ny) and l_w = S y~ - W w~ (nw): two dot products per lane
    each<NY + NW>([&](int k) {
        const double *m1, *v1, *m2, *v2;
        int s1, k1, s2, k2;
        if (k < NY) {
            m1 = R + (NW + k) * NR; s1 = 1; v1 = dw; k1 = NW;          // S^T w~
            m2 = R + NW + k + NW * NR; s2 = NR; v2 = dy; k2 = NY;      // V y~
        } else {
            const int q = k - NY;
            m1 = R + q + NW * NR; s1 = NR; v1 = dy; k1 = NY;           // S y~
            m2 = R + q; s2 = NR; v2 = dw; k2 = NW;                     // W w~
        }
        const double d = dot_pred<(NW > NY ? NW : NY)>(m1, s1, v1, k1, 0.0) -
                         dot_pred<(NW > NY ? NW : NY)>(m2, s2, v2, k2, 0.0);
        if (k < NY) {
            dt[k] = d;
        } else {
            lo[NX + k - NY] = d;
            lo32[NX + k - NY] = f32_rn(d);
        }
    });
    wsync();   // A and B are done with: Q takes their place
    // FP32: [S; V] C (row k of R is contiguous): Q_xw = -(S C)^T and its mirror, V C
    auto none = [](int, int) { return None(); };
    auto put = [&](int k, int j, float v) {
        if (k < NW) fQ[j + (NX + k) * NQ] = fQ[(NX + k) + j * NQ] = -v;
        else fVC[k - NW + j * ldC] = v;
    };
    if constexpr (NX < 48) {
        prod<float, NR, NX, NY, ldR, ldC, false, 0, MHE_TEAM>(fR + NW, fC, none,
                                                              [&](int k, int j, float v, None) { put(k, j, v); });
    } else {
        // One term after another: with the packed sums' rounding of Q (no larger, but another) more short instances of
        // nx = 64 meet the tolerance one correction early.  Of 1200 of 2 to 12 stages refined to relres 1e-12, 86 then end
        // more than 1e-7 off, against 56 with these sums; refined to 1e-13 none does either way
        wgemm<float, NR, NX, NY>([](int, int) { return 0.f; }, [&](int k, int q) { return fR[NW + q + k * ldR]; },
                                 [&](int q, int j) { return fC[q + j * ldC]; }, put);
    }
    each<NW * NW>([&](int i) { fQ[NX + i % NW + (NX + i / NW) * NQ] = fR[i / NW + (i % NW) * ldR]; });
    wsync();
    // Q_x = C^T (V C) (one triangle, mirrored);  FP64: l_x = C^T t
    auto putx = [&](int i, int j, float v) { fQ[i + j * NQ] = fQ[j + i * NQ] = v; };
    if constexpr (NX < 48) {
        prod<float, NX, NX, NY, ldC, ldC, true, 0, MHE_TEAM>(fC, fVC, none,
                                                             [&](int i, int j, float v, None) { putx(i, j, v); });
    } else {
        wgemm<float, NX, NX, NY, true>([](int, int) { return 0.f; }, [&](int i, int q) { return fC[q + i * ldC]; },
                                       [&](int q, int j) { return fVC[q + j * ldC]; }, putx);
    }
    each<NX>([&](int i) {
        const double d = dot_pred<NY>(C + i * NY, 1, dt, NY, 0.0);
        lo[i] = d;
        lo32[i] = f32_rn(d);
    });
    wsync();
    if constexpr (NQ % 4 == 0) {
        each<NQ * NQ / 4>([&](int u) { st16(Qo + 4 * u, ld16g(fQ + 4 * u)); });
    } else {
        each<NQ * NQ>([&](int i) { Qo[i] = fQ[i]; });
    }
#pragma unroll
    for (int k = 0; k < RS; ++k) {
        const int i = lane_id() + k * MHE_TEAM;
        if (i < NQ) {
#pragma unroll 8
            for (int j = 0; j < NQ; ++j) rs[k] += mabs(fQ[i + j * NQ]);
            m = rs[k] > m ? rs[k] : m;
        }
    }
    wsync();
    merge(m);
}

MHE_TEAM_NS_END
}  // namespace mhe
