// kernels.cuh -- __global__ wrappers and launchers of the level passes.
//
// Launch shape: one team (MHE_TEAM lanes) per chunk, W teams per CTA (at most 256
// threads) by the shared memory their workspaces take; the tensor-core reductions
// take one four-warp team per CTA.
#pragma once
#include <cuda_runtime.h>

#include "device.h"
#include "engine.h"
#include "reduce_tc.cuh"
#include "resid.cuh"
#include "solve.cuh"
#include "tree.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// OP_REDUCE_TC / OP_REDUCE_BF: the reduction with the stage products on the
// tensor cores, TF32 or BF16 operands
// OP_DOWN_LIT: Algorithm 6 as printed (every subproblem solved again), the reduction's workspace
enum { OP_REDUCE = 0, OP_RHS = 1, OP_DOWN = 2, OP_REDUCE_TC = 3, OP_REDUCE_BF = 4, OP_DOWN_LIT = 5 };

// floats past the workspace of a tensor-core reduction: a 32 KB operand tile,
// the mbarrier and the TMEM address
constexpr int kTcExtra = 8192 + 4;

// shapes whose reduction runs reduce_chunk_small (pivot blocks of at most 32 rows)
template <int NX>
constexpr bool small_shape() { return NX <= 32; }

// shared-memory workspace (elements of T) one team of a pass needs
template <typename T, int NX, int NW, int UPPER, int OP>
constexpr int op_count()
{
    if (OP == OP_REDUCE && small_shape<NX>()) return team_stride<T>(RedWs<T, NX, NW, UPPER != 0>::count);
    return (OP == OP_REDUCE || OP == OP_DOWN_LIT)
               ? Ws<T, NX>::count
               : (OP == OP_RHS ? team_stride<T>(VecWs<T, NX, NW, UPPER != 0>::rhs_count)
                               : (OP == OP_DOWN ? team_stride<T>(VecWs<T, NX, NW, UPPER != 0>::down_count)
                                                : Ws<T, NX>::count + kTcExtra));   // both tensor-core reductions
}

// CTAs of the residual kernel per SM its register budget is sized for
// (measured on the batched workload: 4 -> 5 CTAs took the n = 24 pass from
// 23.6 to 18.6 ms, 6 the same, 8 spilled and doubled it)
constexpr int kResidBlocks = 5;

// teams per CTA of at most 256 threads: at most 256 / MHE_TEAM
constexpr int kMaxTeams = 256 / MHE_TEAM;

// shared memory the level kernels give their teams' workspaces per CTA
constexpr int kLevelSmem = 224 * 1024;

// the vector passes run in CTAs of 128 threads (one team, when it is wider): their workspaces are
// rings of stage slots, and small CTAs fill an SM's shared memory closely
template <int OP>
constexpr bool vector_op() { return OP == OP_RHS || OP == OP_DOWN; }
template <int OP>
constexpr int op_max_teams()
{
    return vector_op<OP>() ? (MHE_TEAM >= 128 ? 1 : 128 / MHE_TEAM) : kMaxTeams;
}

// CTAs of w teams of `bytes` each that fit an SM (228 KB, of which a CTA takes 1 KB beside its own)
constexpr int ctas_per_sm(int w, int bytes) { return 228 * 1024 / (w * bytes + 1024); }
// teams per CTA that leave the least shared memory unused, whole warps, at most 256 threads
constexpr int best_teams(int bytes)
{
    const int step = MHE_TEAM >= 32 ? 1 : 32 / MHE_TEAM;
    int best = step, most = 0;
    for (int w = step; w <= kMaxTeams; w += step) {
        if (w * bytes > kLevelSmem) break;
        const int n = w * ctas_per_sm(w, bytes);
        if (n > most || (n == most && w * MHE_TEAM <= 128)) { most = n; best = w; }
    }
    return best;
}

// teams per CTA: as many per-team workspaces as fit in kLevelSmem, at most the op's
template <typename T, int NX, int NW, int UPPER, int OP>
constexpr int level_warps()
{
    if (OP == OP_REDUCE && small_shape<NX>()) return best_teams((int)(op_count<T, NX, NW, UPPER, OP>() * sizeof(T)));
    constexpr int fit = kLevelSmem / (int)(op_count<T, NX, NW, UPPER, OP>() * sizeof(T));
    return fit >= op_max_teams<OP>() ? op_max_teams<OP>() : (fit < 1 ? 1 : fit);
}

// a workspace the shared memory of one SM can hold (227 KB per CTA)
template <typename T, int NX, int NW, int UPPER, int OP>
constexpr bool level_fits()
{
    return (long long)op_count<T, NX, NW, UPPER, OP>() * (long long)sizeof(T) <= 227LL * 1024;
}

template <typename T, int NX, int NW, int UPPER, int OP>
constexpr int level_threads()
{
    return vector_op<OP>() ? 128 : (OP == OP_REDUCE && small_shape<NX>() ? level_warps<T, NX, NW, UPPER, OP>() * MHE_TEAM : 256);
}

// CTAs per SM the register allocation is sized for.  The literal Algorithm 6 pass (nx <= 32, 256 threads, the
// general workspace): 64 or 80 registers a thread keep 32 or 24 warps per SM of the small shapes, nx = 20 and
// 24 keep 255 (shared memory allows one CTA anyway); the nx = 64 passes of four-warp teams take 255.
template <typename T, int NX, int NW, int UPPER, int OP>
constexpr int level_min_blocks()
{
    if (vector_op<OP>()) {
        // as many CTAs as shared memory holds, with at least 64 registers a thread
        constexpr int bytes = level_warps<T, NX, NW, UPPER, OP>() * op_count<T, NX, NW, UPPER, OP>() * (int)sizeof(T);
        constexpr int fit = 228 * 1024 / (bytes + 1024);
        return fit > 8 ? 8 : (fit < 1 ? 1 : fit);
    }
    if (OP == OP_REDUCE && small_shape<NX>()) {
        // what shared memory holds, with at least 96 registers a thread
        constexpr int w = level_warps<T, NX, NW, UPPER, OP>();
        constexpr int fit = ctas_per_sm(w, op_count<T, NX, NW, UPPER, OP>() * (int)sizeof(T));
        constexpr int regs = 65536 / (w * MHE_TEAM * 96);
        return fit < regs ? (fit < 1 ? 1 : fit) : (regs < 1 ? 1 : regs);
    }
    return NX > 12 ? 1 : (sizeof(T) == 8 ? 2 : (NX <= 8 ? 4 : 3));
}

// shapes whose stage products run on the tensor cores: a team of four warps,
// one team per CTA, M = 128 >= n + m and 2n rows, K = n a multiple of 16,
// a 128-row operand tile of at most 32 KB
template <int NX, int NW>
constexpr bool tc_shape()
{
    return MHE_TEAM == 128 && NX % 16 == 0 && NW % 16 == 0 && NX + NW <= 128 && 2 * NX <= 128 &&
           128 * NX * 4 <= 32 * 1024 && level_warps<float, NX, NW, 0, OP_REDUCE_TC>() == 1 &&
           (long long)op_count<float, NX, NW, 0, OP_REDUCE_TC>() * 4 <= 227LL * 1024;
}

// Team slots of a global-memory workspace a context provides: two CTAs of one
// team per SM of a 152-SM GB300 (the register budget of a 128-thread team at 255
// registers a thread allows two per SM).  A launch takes at most this many CTAs
// and each CTA walks the chunks blockIdx.x, blockIdx.x + gridDim.x, ...
constexpr int kGwsTeams = 2 * 152;

template <typename T, int NX, int NW, int UPPER, int OP>
__global__ void __launch_bounds__(level_threads<T, NX, NW, UPPER, OP>(), level_min_blocks<T, NX, NW, UPPER, OP>()) k_level(LevelArgs<T> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int W = level_warps<T, NX, NW, UPPER, OP>();
    if constexpr (!level_fits<T, NX, NW, UPPER, OP>()) {
        // the workspace of one subproblem exceeds an SM's shared memory (FP64 at
        // nx = 64): one team per CTA, its workspace in the CTA's slot of the
        // context's global workspace (L2-resident; the FP64 pipe, at about two
        // DFMAs per clock per SM, hides the L2 latency of the products)
        static_assert(W == 1 && (OP == OP_REDUCE || OP == OP_RHS || OP == OP_DOWN), "one CUDA-core team per CTA");
        if (a.any_active && *a.any_active == 0) return;
        T* ws = a.gws + (size_t)blockIdx.x * op_count<T, NX, NW, UPPER, OP>();
        for (int ci = blockIdx.x; ci < a.nchunks; ci += gridDim.x) {
            if (!chunk_in_bounds(a, ci)) continue;
            if constexpr (OP == OP_REDUCE) reduce_chunk<T, NX, NW, UPPER != 0>(a, ci, ws);
            else if constexpr (OP == OP_RHS) rhs_chunk<T, NX, NW, UPPER != 0>(a, ci, ws);
            else down_chunk<T, NX, NW, UPPER != 0>(a, ci, ws);
        }
        return;
    }
    const int team = team_id();
    const int ci = blockIdx.x * W + team;
    if (ci >= a.nchunks) return;   // the whole team leaves together
    if (a.any_active && *a.any_active == 0) return;   // a refinement pass with every instance converged
    T* sm = reinterpret_cast<T*>(smem_raw) + (size_t)team * op_count<T, NX, NW, UPPER, OP>();
    if constexpr (OP == OP_REDUCE_TC || OP == OP_REDUCE_BF) {
        // one team per CTA: TMEM (all 512 columns; one CTA fits an SM) and the mbarrier are the CTA's
        static_assert(W == 1 && sizeof(T) == 4, "one FP32 tensor-core team per CTA");
        float* xbuf = reinterpret_cast<float*>(smem_raw) + Ws<float, NX>::count;
        uint64_t* mbar = reinterpret_cast<uint64_t*>(xbuf + 8192);
        uint32_t* slot = reinterpret_cast<uint32_t*>(mbar + 1);
        if (threadIdx.x < 32) tc::tmem_alloc(slot, 512);
        if (threadIdx.x == 0) tc::mbar_init(mbar, 1);
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        TcState tcs{*slot, mbar, xbuf, 0u, 1};
        if (chunk_in_bounds(a, ci)) reduce_chunk<T, NX, NW, UPPER != 0, OP == OP_REDUCE_TC ? 1 : 2>(a, ci, sm, &tcs);
        // a wait that ran out: give the MMAs of that phase another bounded wait before freeing TMEM
        if (!tcs.ok) tc::mbar_wait(mbar, tcs.phase, tc::kWaitLimit);
        tc::fence_before();
        __syncthreads();
        tc::fence_after();
        if (threadIdx.x < 32) tc::tmem_dealloc(tcs.tbase, 512);
    } else {
        if (!chunk_in_bounds(a, ci)) return;
        if constexpr (OP == OP_REDUCE && small_shape<NX>()) reduce_chunk_small<T, NX, NW, UPPER != 0>(a, ci, sm);
        else if constexpr (OP == OP_REDUCE) reduce_chunk<T, NX, NW, UPPER != 0>(a, ci, sm);
        else if constexpr (OP == OP_RHS) rhs_chunk<T, NX, NW, UPPER != 0>(a, ci, sm);
        else if constexpr (OP == OP_DOWN_LIT) down_chunk_literal<T, NX, NW, UPPER != 0>(a, ci, sm);
        else down_chunk<T, NX, NW, UPPER != 0>(a, ci, sm);
    }
}

template <typename T, int NX, int NW, int UPPER, int OP>
void launch_level_v(const LevelArgs<T>& a, void* stream)
{
    constexpr int W = level_warps<T, NX, NW, UPPER, OP>();
    if constexpr (!level_fits<T, NX, NW, UPPER, OP>()) {
        // global-memory workspace: at most gws_teams CTAs of one team, no dynamic shared memory
        if (!a.gws || a.gws_teams < 1) return;   // the context holds no workspace slots: nothing is launched
        const int grid = a.nchunks < a.gws_teams ? a.nchunks : a.gws_teams;
        k_level<T, NX, NW, UPPER, OP><<<grid, MHE_TEAM, 0, (cudaStream_t)stream>>>(a);
        return;
    }
    const size_t smem = (size_t)W * op_count<T, NX, NW, UPPER, OP>() * sizeof(T);
    static OncePerDevice attr;
    attr([&] {
        cudaFuncSetAttribute(k_level<T, NX, NW, UPPER, OP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    });
    const int grid = (a.nchunks + W - 1) / W;
    k_level<T, NX, NW, UPPER, OP><<<grid, MHE_TEAM * W, smem, (cudaStream_t)stream>>>(a);
}

template <typename T, int NX, int NW, int OP>
void launch_level(const LevelArgs<T>& a, int upper, void* stream)
{
    if (a.nchunks <= 0) return;
    if (upper) launch_level_v<T, NX, NW, 1, OP>(a, stream);
    else launch_level_v<T, NX, NW, 0, OP>(a, stream);
}

// Whole instances (plans of one level), TF32 products: two CTAs of one team per SM.  Measured (nx = 64, 256
// instances of 512 stages): 18.04 -> 9.9 ms, the estimate 45.7 -> 37.5 ms.  Plans of several levels keep the general
// workspace: their other chunks' stages form V.
constexpr int kTcLastCols = 256;   // TMEM columns of a team: half of an SM's

template <int NX, int NW>
__global__ void __launch_bounds__(MHE_TEAM, 2) k_reduce_last(LevelArgs<float> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (a.any_active && *a.any_active == 0) return;
    float* sm = reinterpret_cast<float*>(smem_raw);
    uint64_t* mbar = reinterpret_cast<uint64_t*>(sm + TcWs<NX, NW>::count);
    uint32_t* slot = reinterpret_cast<uint32_t*>(mbar + 1);
    static_assert(2 * (NX + NW) <= kTcLastCols && TcWs<NX, NW>::count % 4 == 0, "accumulators, alignment");
    if (threadIdx.x < 32) tc::tmem_alloc(slot, kTcLastCols);
    if (threadIdx.x == 0) tc::mbar_init(mbar, 1);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    TcState tcs{*slot, mbar, nullptr, 0u, 1};
    if (chunk_in_bounds(a, blockIdx.x)) reduce_last_tc<NX, NW>(a, blockIdx.x, sm, tcs);
    // a wait that ran out: give the MMAs of that phase another bounded wait before freeing TMEM
    if (!tcs.ok) tc::mbar_wait(mbar, tcs.phase, tc::kWaitLimit);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (threadIdx.x < 32) tc::tmem_dealloc(tcs.tbase, kTcLastCols);
}

template <int NX, int NW>
void launch_reduce_last(const LevelArgs<float>& a, int, void* stream)
{
    if (a.nchunks <= 0) return;
    constexpr size_t smem = (size_t)TcWs<NX, NW>::count * sizeof(float) + 16;
    static_assert(2 * (smem + 1024) <= 228 * 1024, "two CTAs per SM");
    static OncePerDevice attr;
    attr([&] {
        cudaFuncSetAttribute(k_reduce_last<NX, NW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    k_reduce_last<NX, NW><<<a.nchunks, MHE_TEAM, smem, (cudaStream_t)stream>>>(a);
}

// The residual waits on its FP64 loads from HBM; five CTAs of 256 threads per SM
// (48 registers a thread, a few spilled) hide that latency better than four.
template <int NX, int NW, typename TR, int NY>
__global__ void __launch_bounds__(256, kResidBlocks) k_resid(ResidArgs<TR> r)
{
    __shared__ unsigned long long sm[kMaxTeams][ResidSmem<NX, NW, NY>::count];
    const int team = team_id();
    const long long g = (long long)blockIdx.x * kMaxTeams + team;
    if (g >= r.nstages) return;
    if (r.any_active && *r.any_active == 0) return;
    resid_stage<NX, NW, TR, NY>(r, g, sm[team]);
}

// The double-float residual (MHE form, FP32 correction solves): one resident grid, whose teams walk the
// stages, in CTAs that leave the least of an SM's shared memory unused (at most 64 threads a CTA before: nx = 24,
// 535k stages, 2.05 -> 1.94 ms; nx = 12, 1.05M stages, 1.27 -> 1.21 ms).
template <int NX, int NW, int NY>
constexpr int resid_df_teams() { return best_teams(DfWs<NX, NW, NY>::bytes); }
template <int NX, int NW, int NY>
constexpr int resid_df_blocks()
{
    // what shared memory holds, with at least 64 registers a thread
    constexpr int w = resid_df_teams<NX, NW, NY>();
    constexpr int fit = ctas_per_sm(w, DfWs<NX, NW, NY>::bytes), regs = 65536 / (w * MHE_TEAM * 64);
    return fit < regs ? (fit < 1 ? 1 : fit) : (regs < 1 ? 1 : regs);
}

template <int NX, int NW, int NY>
__global__ void __launch_bounds__(resid_df_teams<NX, NW, NY>() * MHE_TEAM, resid_df_blocks<NX, NW, NY>())
    k_resid_df(ResidArgs<float> r)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    if (r.any_active && *r.any_active == 0) return;
    constexpr int W = resid_df_teams<NX, NW, NY>();
    StageBlocks it(r, (long long)blockIdx.x * W + team_id(), (long long)gridDim.x * W);
    resid_df_run<NX, NW, NY>(r, it, smem_raw + (size_t)team_id() * DfWs<NX, NW, NY>::bytes);
}

// NY = 0: Q form; NY > 0: MHE form (C, R)
template <int NX, int NW, typename TR, int NY = 0>
void launch_resid(const ResidArgs<TR>& r, void* stream)
{
    if (r.nstages <= 0) return;
    if constexpr (NY > 0 && sizeof(TR) == 4) {
        if (r.Ahi) {
            constexpr int W = resid_df_teams<NX, NW, NY>();
            constexpr size_t smem = (size_t)W * DfWs<NX, NW, NY>::bytes;
            static OncePerDevice attr;
            attr([&] {
                cudaFuncSetAttribute(k_resid_df<NX, NW, NY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            });
            const long long blocks = (r.nstages + W - 1) / W;
            const long long room = (long long)device_sms() * resid_df_blocks<NX, NW, NY>();
            k_resid_df<NX, NW, NY><<<(unsigned)(blocks < room ? blocks : room), W * MHE_TEAM, smem,
                                     (cudaStream_t)stream>>>(r);
            return;
        }
    }
    const long long grid = (r.nstages + kMaxTeams - 1) / kMaxTeams;
    k_resid<NX, NW, TR, NY><<<(unsigned)grid, 256, 0, (cudaStream_t)stream>>>(r);
}

// teams per block of the one-pass MHE preparation: <= 40 KB of shared memory
// per CTA (several CTAs per SM), at least one team
template <int NX, int NW, int NY>
constexpr int prep_warps()
{
    constexpr int fit = 40 * 1024 / (PrepSmem<NX, NW, NY>::count * 8);
    return fit >= kMaxTeams ? kMaxTeams : (fit < 1 ? 1 : fit);
}

template <int NX, int NW, int NY>
__global__ void __launch_bounds__(256) k_prep(PrepArgs p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int W = prep_warps<NX, NW, NY>();
    const int team = team_id();
    const long long g = (long long)blockIdx.x * W + team;
    if (g >= p.nstages) return;
    prep_stage<NX, NW, NY>(p, g, reinterpret_cast<double*>(smem_raw) + (size_t)team * PrepSmem<NX, NW, NY>::count);
}

template <int NX, int NW, int NY>
void launch_prep(const PrepArgs& p, void* stream)
{
    if (p.nstages <= 0) return;
    constexpr int W = prep_warps<NX, NW, NY>();
    const size_t smem = (size_t)W * PrepSmem<NX, NW, NY>::count * 8;
    static OncePerDevice attr;
    attr([&] {
        cudaFuncSetAttribute(k_prep<NX, NW, NY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    const long long grid = (p.nstages + W - 1) / W;
    k_prep<NX, NW, NY><<<(unsigned)grid, MHE_TEAM * W, smem, (cudaStream_t)stream>>>(p);
}

template <int NX, int NW>
__global__ void __launch_bounds__(256) k_knorm(KnormArgs r)
{
    __shared__ float sm[kMaxTeams][2 * NX + NW + 4];
    const int team = team_id();
    const long long g = (long long)blockIdx.x * kMaxTeams + team;
    if (g >= r.nstages) return;
    knorm_stage<NX, NW>(r, g, sm[team]);
}

template <int NX, int NW>
void launch_knorm(const KnormArgs& r, void* stream)
{
    if (r.nstages <= 0) return;
    const long long grid = (r.nstages + kMaxTeams - 1) / kMaxTeams;
    k_knorm<NX, NW><<<(unsigned)grid, 256, 0, (cudaStream_t)stream>>>(r);
}

template <int NX, int NW, int NY>
constexpr int asm_warps()
{
    return (40 * 1024) / (int)(AsmSmem<NX, NW, NY>::count * 8) >= kMaxTeams
               ? kMaxTeams
               : ((40 * 1024) / (int)(AsmSmem<NX, NW, NY>::count * 8) < 1
                      ? 1
                      : (40 * 1024) / (int)(AsmSmem<NX, NW, NY>::count * 8));
}

template <int NX, int NW, int NY>
__global__ void __launch_bounds__(256) k_assemble(long long S, const double* C, const double* R,
                                                   const double* yt, const double* wt, double* Q, double* l,
                                                   double* c)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int W = asm_warps<NX, NW, NY>();
    const int team = team_id();
    const long long s = (long long)blockIdx.x * W + team;
    if (s >= S) return;
    constexpr int NR = NW + NY, NQ = NX + NW;
    assemble_stage<NX, NW, NY>(C + s * NY * NX, R + s * NR * NR, yt + s * NY, wt + s * NW, Q + s * NQ * NQ,
                               l + s * NQ, c ? c + s : nullptr,
                               reinterpret_cast<double*>(smem_raw) + (size_t)team * AsmSmem<NX, NW, NY>::count);
}

template <int NX, int NW, int NY>
void launch_assemble(long long S, const double* C, const double* R, const double* yt, const double* wt,
                     double* Q, double* l, double* c, void* stream)
{
    if (S <= 0) return;
    constexpr int W = asm_warps<NX, NW, NY>();
    const size_t smem = (size_t)W * AsmSmem<NX, NW, NY>::count * 8;
    static OncePerDevice attr;
    attr([&] {
        cudaFuncSetAttribute(k_assemble<NX, NW, NY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    });
    const long long grid = (S + W - 1) / W;
    k_assemble<NX, NW, NY><<<(unsigned)grid, MHE_TEAM * W, smem, (cudaStream_t)stream>>>(S, C, R, yt, wt, Q, l, c);
}

template <int NX, int NW, int NY>
ShapeEntry make_shape()
{
    ShapeEntry e;
    e.ops.nx = NX;
    e.ops.nw = NW;
    e.ops.team = MHE_TEAM;
    if constexpr (level_fits<double, NX, NW, 0, OP_REDUCE>()) {
        e.ops.reduce64 = &launch_level<double, NX, NW, OP_REDUCE>;
        e.ops.rhs64 = &launch_level<double, NX, NW, OP_RHS>;
        e.ops.down64 = &launch_level<double, NX, NW, OP_DOWN>;
    } else {   // the FP64 workspace of one subproblem exceeds an SM's shared memory: a translation
               // unit of its own adds the global-memory variant (set_fp64_global_ops)
        e.ops.reduce64 = nullptr;
        e.ops.rhs64 = nullptr;
        e.ops.down64 = nullptr;
    }
    e.ops.reduce32 = &launch_level<float, NX, NW, OP_REDUCE>;
    if constexpr (tc_shape<NX, NW>()) {
        e.ops.reduce32tc = &launch_level<float, NX, NW, OP_REDUCE_TC>;
        e.ops.reduce32bf = &launch_level<float, NX, NW, OP_REDUCE_BF>;
    } else {
        e.ops.reduce32tc = nullptr;
        e.ops.reduce32bf = nullptr;
    }
    if constexpr (tc_shape<NX, NW>() && tc_last_shape<NX, NW>()) e.ops.reduce32tc1 = &launch_reduce_last<NX, NW>;
    else e.ops.reduce32tc1 = nullptr;
    e.ops.rhs32 = &launch_level<float, NX, NW, OP_RHS>;
    e.ops.down32 = &launch_level<float, NX, NW, OP_DOWN>;
    // the literal Algorithm 6 down pass, for the shapes whose reduction workspace fits an SM
    if constexpr (level_fits<double, NX, NW, 0, OP_REDUCE>() && NX <= 32) {
        e.ops.down64lit = &launch_level<double, NX, NW, OP_DOWN_LIT>;
        e.ops.down32lit = &launch_level<float, NX, NW, OP_DOWN_LIT>;
    } else {
        e.ops.down64lit = nullptr;
        e.ops.down32lit = nullptr;
    }
    e.ops.resid64 = &launch_resid<NX, NW, double>;
    e.ops.resid32 = &launch_resid<NX, NW, float>;
    e.ops.knorm = &launch_knorm<NX, NW>;
    e.ops.ny = NY;
    e.ops.assemble = &launch_assemble<NX, NW, NY>;
    e.ops.prep32 = &launch_prep<NX, NW, NY>;
    e.ops.resid_mhe32 = &launch_resid<NX, NW, float, NY>;
    e.ops.gws64 = 0;
    e.ops.gws_teams = 0;
    e.ops.reduce64w = nullptr;
    e.ops.reduce32w = nullptr;
    e.ops.wide64 = e.ops.wide32 = 0;
    if constexpr (NX <= 32) {
        e.ops.solve64 = &launch_solve<double, NX, NW, 0>;
        e.ops.solve32 = &launch_solve<float, NX, NW, 0>;
        e.ops.solve_mhe32 = &launch_solve<float, NX, NW, NY>;
        e.ops.solve_cluster = &solve_cluster<NX, NW, NY>;
        e.ops.resume_cluster = &resume_cluster<NX, NW, NY>;
    } else {
        e.ops.solve64 = nullptr;
        e.ops.solve32 = e.ops.solve_mhe32 = nullptr;
        e.ops.solve_cluster = e.ops.resume_cluster = nullptr;
    }
    e.ny = NY;
    e.assemble = &launch_assemble<NX, NW, NY>;
    return e;
}

// A level's reduction with this unit's wider team, for levels of few chunks: there the length of one chunk's chain is
// the time.  The limits are four (eight) chunks for each of the GPU's 152 SMs.  Measured (GB300, a level's reduction, own
// team and wider one, ratio of the times; leaf levels of 16 stages and master levels of four, 19 to 6080 chunks):
//             up to 152    304          608          760          912          1216
//   FP64 n=4  0.70-0.97    0.70-0.97    0.71-0.80    0.71-0.80    0.70-0.80    0.80-1.35
//   FP64 n=6  0.50-0.74    0.50-0.72    0.51-0.60    0.51-0.59    0.51-0.59    0.89-1.07
//   FP64 12   0.27-0.40    0.32-0.48    0.54-0.59    0.91-0.92    1.06-1.07    0.87-0.94
//   FP64 20   0.33-0.47    0.48-0.59    0.87-0.88    1.22-1.31    0.94-1.32    0.76-0.84
//   FP64 24   0.32-0.44    0.47-0.57    0.68-0.88    0.77-1.30    0.78-0.88    0.73-0.85
//   FP32 4, 6 0.67-0.89    0.68-0.85    0.66-0.74    0.66-0.71    0.67-0.74    0.67-0.78
//   FP32 12   0.53-0.88    0.53-0.85    0.58-0.75    1.04-1.23    1.04-1.24    0.92-1.15
//   FP32 20   0.62-0.81    0.66-0.83    0.82-0.94    1.14-1.21    1.20-1.28    1.25-1.37
//   FP32 24   0.60-0.73    0.62-0.79    0.70-0.83    1.00-1.03    1.16-1.22    0.74-1.17
// (nx = nw = 20 as nx = 20.)  Up to 608 the wider team wins for every shape; beyond it depends on how the chunks fill the
// last wave, and only FP64 nx = 12 keeps it further, where it loses at most 7% and wins 13%.
template <int NX, int NW>
WideEntry make_wide()
{
    WideEntry w;
    w.nx = NX;
    w.nw = NW;
    w.reduce64 = &launch_level<double, NX, NW, OP_REDUCE>;
    w.reduce32 = &launch_level<float, NX, NW, OP_REDUCE>;
    w.chunks64 = NX <= 12 && MHE_TEAM == 128 ? 1216 : 608;
    w.chunks32 = 608;
    return w;
}

// The FP64 passes of a shape whose FP64 reduction workspace exceeds an SM's
// shared memory: the reduction keeps it in global memory (k_level's global
// variant); the right-hand-side and down passes need less and stay in shared memory.
template <int NX, int NW>
void set_fp64_global_ops(ShapeOps& o)
{
    static_assert(!level_fits<double, NX, NW, 0, OP_REDUCE>(), "shapes whose FP64 workspace fits use make_shape");
    o.reduce64 = &launch_level<double, NX, NW, OP_REDUCE>;
    o.rhs64 = &launch_level<double, NX, NW, OP_RHS>;
    o.down64 = &launch_level<double, NX, NW, OP_DOWN>;
    o.gws64 = op_count<double, NX, NW, 0, OP_REDUCE>();
    o.gws_teams = kGwsTeams;
}

MHE_TEAM_NS_END
}  // namespace mhe
