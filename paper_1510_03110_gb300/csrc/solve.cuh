// solve.cuh -- a whole solve with stored factors, and its refinement, in one launch.
//
// One cluster of CTAs per instance: its teams share the chunks of every level of
// that instance (vector part of Algorithm 4 level by level up, Algorithm 6 down),
// then the stages of the residual, and repeat the correction until the instance's
// residual meets the tolerance.  The steps that depend on one another are
// separated by the cluster's hardware barrier; nothing waits across clusters, so
// instances converge and finish independently of each other.
//
// Why: with one launch per level and pass a correction is about a dozen launches,
// each a couple of microseconds of latency, and every allowed correction is
// launched whether an instance still needs it or not.  For a batch of few or small
// instances that is most of the solve: one estimate of nx = 12, N = 200 with 16 corrections
// allowed took 213 launches and 0.81 ms; this launch brought it to 12 launches and 0.41 ms, and to 0.29 ms
// with the reductions that came after it.
#pragma once
#include <cuda_runtime.h>
#include <string.h>

#include "device.h"
#include "resid.cuh"
#include "solve_rule.h"
#include "tree.cuh"

namespace mhe {
MHE_TEAM_NS_BEGIN

// 8-byte words of shared memory one team needs: the larger of the vector passes' workspaces and the residual's
template <typename T, int NX, int NW, int NY>
constexpr int solve_words()
{
    using V0 = VecWs<T, NX, NW, false>;
    using V1 = VecWs<T, NX, NW, true>;
    constexpr int v = max_int(max_int(V0::rhs_count, V0::down_count), max_int(V1::rhs_count, V1::down_count));
    constexpr int r = (v * (int)sizeof(T) + 7) / 8;
    constexpr int q = NY > 0 ? DfWs<NX, NW, NY == 0 ? 1 : NY>::bytes / 8 : ResidSmem<NX, NW, 0>::count;
    constexpr int n = ((r > q ? r : q) + 1) / 2 * 2;
    return team_stride<T>(n * (8 / (int)sizeof(T))) * (int)sizeof(T) / 8;
}

// teams per CTA: 256 threads, fewer (a power of two) where their workspaces do not fit
template <typename T, int NX, int NW, int NY>
constexpr int solve_teams()
{
    int w = 256 / MHE_TEAM;
    while (w > 1 && w * solve_words<T, NX, NW, NY>() * 8 > 222 * 1024) w /= 2;
    return w;
}
template <typename T, int NX, int NW, int NY>
constexpr int solve_threads() { return solve_teams<T, NX, NW, NY>() * MHE_TEAM; }

MHE_DEV int cluster_rank()
{
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}

// every thread of the instance's cluster; orders global memory among them
MHE_DEV void instance_sync(int cluster)
{
    __syncwarp();   // the teams of a warp meet first
    if (cluster == 1) {
        __syncthreads();
    } else {
        asm volatile("barrier.cluster.arrive.release;" ::: "memory");
        asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    }
}

template <typename T, int NX, int NW, int NY>
MHE_DEV void solve_residual(const ResidArgs<T>& r, int b, int N, int team, int teams, unsigned long long* sm)
{
    if constexpr (NY > 0) {
        StageStride it{b, team, teams, N};
        resid_df_run<NX, NW, NY>(r, it, reinterpret_cast<unsigned char*>(sm));
        wsync();
    } else {
        for (int t = team; t < N; t += teams) {
            if (t == 0) resid_rows<NX, NW, 1, T>(r, b, 0, N, sm);
            else resid_q<NX, NW, T>(r, b, t, N, sm);
            wsync();
        }
    }
}

template <typename T, int NX, int NW, int NY>
__global__ void __launch_bounds__(solve_threads<T, NX, NW, NY>(), 2) k_solve(const __grid_constant__ SolveArgs<T> p)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int kThreads = solve_threads<T, NX, NW, NY>(), kTeams = solve_teams<T, NX, NW, NY>();
    const int C = p.cluster;
    const int rank = C == 1 ? 0 : cluster_rank();
    const int b = blockIdx.x / C;
    const int team = rank * kTeams + team_id(), teams = C * kTeams;
    const bool lead = rank == 0 && threadIdx.x == 0;
    unsigned long long* sm =
        reinterpret_cast<unsigned long long*>(smem_raw) + (size_t)team_id() * solve_words<T, NX, NW, NY>();
    T* ws = reinterpret_cast<T*>(sm);
    if (p.resume && !p.active[b]) return;   // the whole cluster
    const LevelInst li = p.lv[0].li[b];
    const int N = li.N;
    unsigned long long* norms = p.r.norms + 3LL * b;
    if (p.zx) {
        // the accumulated solution of this instance starts from zero
        const int tid = rank * kThreads + threadIdx.x, nt = C * kThreads;
        const long long nxl = (long long)(N + 1) * NX, nwl = NX + (long long)(N - 1) * NW;
        for (long long i = tid; i < nxl; i += nt) p.zx[li.gx * NX + i] = p.zl[li.gx * NX + i] = 0.0;
        for (long long i = tid; i < nwl; i += nt) p.zw[p.lv[0].w_off[b] + i] = 0.0;
    }
    if (lead) {
        norms[0] = norms[1] = norms[2] = 0ULL;
        p.dznorm[b] = 0u;
    }
    // resumed: the check that left the instance active counted the correction that comes now
    int iters = p.resume ? p.iters[b] : 0;
    double relres = 0.0, est = 0.0;
    for (int it = p.resume ? 0 : -1;; ++it) {
        const int v0 = it < 0 ? 0 : kSolveLevels;
        if (it >= 0 || !p.fused_rhs) {
#pragma unroll 1
            for (int k = 0; k < p.nlev; ++k) {
                const LevelInst lk = p.lv[k].li[b];
#pragma unroll 1
                for (int ci = lk.c0 + team; ci < lk.c1; ci += teams) {
                    if (!chunk_in_bounds(p.lv[v0 + k], ci)) continue;
                    if (k == 0) rhs_chunk<T, NX, NW, false>(p.lv[v0 + k], ci, ws);
                    else rhs_chunk<T, NX, NW, true>(p.lv[v0 + k], ci, ws);
                    wsync();
                }
                if (lk.top) break;
                instance_sync(C);
            }
        }
        instance_sync(C);
        if (lead && it >= 0) {
            norms[0] = norms[1] = norms[2] = 0ULL;   // every thread has read the last check's
            p.dznorm[b] = 0u;                        // this correction is measured afresh
        }
        int top = 0;
        while (top + 1 < p.nlev && !p.lv[top].li[b].top) ++top;
        if (top == 0) instance_sync(C);   // dznorm is cleared before level 0's down pass
#pragma unroll 1
        for (int k = top; k >= 0; --k) {
            const int c0 = p.lv[k].li[b].c0, c1 = p.lv[k].li[b].c1;
#pragma unroll 1
            for (int ci = c0 + team; ci < c1; ci += teams) {
                if (!chunk_in_bounds(p.lv[v0 + k], ci)) continue;
                if (k == 0) down_chunk<T, NX, NW, false>(p.lv[v0 + k], ci, ws);
                else down_chunk<T, NX, NW, true>(p.lv[v0 + k], ci, ws);
                wsync();
            }
            instance_sync(C);
        }
        solve_residual<T, NX, NW, NY>(p.r, b, N, team, teams, sm);
        instance_sync(C);
        // the check: every thread of the cluster reads the same norms and decides the same
        const double r = __longlong_as_double((long long)__ldcg(norms));
        const double z = __longlong_as_double((long long)__ldcg(norms + 1));
        const double bb = __longlong_as_double((long long)__ldcg(norms + 2));
        const double den = (double)__uint_as_float(p.kinf[b]) * z + bb;
        relres = den > 0 ? r / den : r;
        est = (iters > 0 && z > 0) ? (double)__uint_as_float(__ldcg(p.dznorm + b)) / z : 0.0;
        const bool act = p.lv[0].status[b] == 0 && isfinite(relres) && !(relres <= p.tol);
        if (!act || iters >= p.max_refine) break;
        ++iters;
    }
    if (lead) {
        const int* where = p.lv[0].where + 3LL * b;
        mhe_info_rec o;
        o.status = p.lv[0].status[b];
        if (o.status == 0 && !isfinite(relres)) o.status = -4;                                   // MHE_E_NONFINITE
        else if (o.status == 0 && p.max_refine > 0 && !(relres <= p.tol)) o.status = -6;         // MHE_E_NO_CONVERGE
        o.level = where[0];
        o.chunk = where[1];
        o.stage = where[2];
        o.refine_iters = iters;
        o.pad = 0;
        o.relres = relres;
        o.est_relerr = est;
        p.info[b] = o;
        p.iters[b] = iters;
        p.active[b] = 0;
    }
}

template <typename T, int NX, int NW, int NY>
constexpr size_t solve_smem()
{
    return (size_t)solve_teams<T, NX, NW, NY>() * solve_words<T, NX, NW, NY>() * 8;
}

// clusters of more than eight CTAs and the shared memory, allowed once per kernel and GPU
template <typename T, int NX, int NW, int NY>
void solve_attributes()
{
    static OncePerDevice attr;
    attr([] {
        cudaFuncSetAttribute(k_solve<T, NX, NW, NY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)solve_smem<T, NX, NW, NY>());
        cudaFuncSetAttribute(k_solve<T, NX, NW, NY>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    });
}

template <typename T, int NX, int NW, int NY>
void launch_solve(const SolveArgs<T>& p, void* stream)
{
    if (p.batch <= 0) return;
    solve_attributes<T, NX, NW, NY>();
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3((unsigned)p.batch * p.cluster);
    cfg.blockDim = dim3(solve_threads<T, NX, NW, NY>());
    cfg.dynamicSmemBytes = solve_smem<T, NX, NW, NY>();
    cfg.stream = (cudaStream_t)stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)p.cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.cluster > 1 ? 1 : 0;
    cudaLaunchKernelEx(&cfg, k_solve<T, NX, NW, NY>, p);
}

inline int device_sms()
{
    static PerDevice sms;
    return sms([] {
        int dev = 0, v = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
            cudaGetLastError();
            v = 152;
        }
        return v;
    });
}

// Clusters of 1 << i CTAs of the kernel the current GPU holds at a time, 0 for a size it cannot schedule
template <typename T, int NX, int NW, int NY>
int solve_resident(int i)
{
    static PerDevice most[kSolveSizes];
    return most[i]([i] {
        solve_attributes<T, NX, NW, NY>();
        cudaLaunchConfig_t cfg;
        memset(&cfg, 0, sizeof(cfg));
        cfg.gridDim = dim3((unsigned)(device_sms() * kSolveMaxCluster));
        cfg.blockDim = dim3(solve_threads<T, NX, NW, NY>());
        cfg.dynamicSmemBytes = solve_smem<T, NX, NW, NY>();
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1u << i;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, k_solve<T, NX, NW, NY>, &cfg) != cudaSuccess) {
            cudaGetLastError();
            n = 0;
        }
        return n;
    });
}

template <typename T, int NX, int NW, int NY>
SolveRoom solve_room()
{
    SolveRoom r;
    r.teams = solve_teams<T, NX, NW, NY>();
    r.sms = device_sms();
    for (int i = 0; i < kSolveSizes; ++i) r.resident[i] = solve_resident<T, NX, NW, NY>(i);
    return r;
}

// the kernel a solve takes; mhe: the residual is the double-float MHE form's
template <int NX, int NW, int NY>
SolveRoom solve_room_of(int fp64, int mhe)
{
    if (fp64) return solve_room<double, NX, NW, 0>();
    return mhe ? solve_room<float, NX, NW, NY>() : solve_room<float, NX, NW, 0>();
}

// CTAs per instance of a whole solve, and of a larger batch's last corrections, or 0 (solve_rule.h)
template <int NX, int NW, int NY>
int solve_cluster(int fp64, int mhe, int batch, int max_N)
{
    return fused_cluster(NX, solve_room_of<NX, NW, NY>(fp64, mhe), batch, max_N);
}
template <int NX, int NW, int NY>
int resume_cluster(int fp64, int mhe, int batch, int max_N)
{
    return resumed_cluster(solve_room_of<NX, NW, NY>(fp64, mhe), batch, max_N);
}

MHE_TEAM_NS_END
}  // namespace mhe
