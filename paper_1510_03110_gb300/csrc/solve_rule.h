// solve_rule.h -- when a solve and its corrections run as one launch (solve.cuh), and with how many CTAs an
// instance.  Plain arithmetic of the shape, the batch and the GPU, so that it can be checked without one.
//
// All times: GB300 (152 SMs), milliseconds; "passes" is one launch per level and pass.
#pragma once

namespace mhe {

constexpr int kSolveMaxCluster = 16;   // CTAs per instance: 1, 2, 4, 8 or 16
constexpr int kSolveSizes = 5;

// What one kernel of solve.cuh has on one GPU: its teams per CTA, and how many clusters of 1 << i CTAs the GPU
// holds at a time (0: that size cannot be scheduled)
struct SolveRoom {
    int teams = 0, sms = 0;
    int resident[kSolveSizes] = {};
};

// stages of the residual a team may walk: above nx = 12 the stages are longer.  Beyond it the passes, which spread
// every stage over the whole GPU, are faster even though they launch the corrections nobody needs
constexpr int solve_stages(int nx) { return nx <= 12 ? 16 : 6; }

// CTAs per instance of a whole solve, or 0 for a launch per level pass.  A team has at least about one stage of the
// residual, the clusters together about fill the GPU once, and every cluster is resident at once: a second wave
// doubles the time (FP32, three corrections: 8 instances of nx = 12, N = 800, clusters of 8 and of 16: 0.60 and
// 0.98, passes 0.63; 20 of nx = 24, N = 100, clusters of 4 and of 8: 0.48 and 0.78, passes 0.49).
// Above solve_stages a team the passes are faster.  Measured with every allowed correction used (the launch's
// worst case, three of them), one launch and passes: nx = 12, N = 1000, 16 CTAs (4 stages a team), 0.51 and 0.53;
// N = 3000 (12) 0.90 and 0.65; nx = 20, N = 400 (3) 0.51 and 0.48; nx = 24, N = 600 (5) 0.67 and 0.55.  A correction
// that is allowed and not needed costs the passes another 0.04, one launch nothing, so the line lies above the
// point where they meet: with 16 allowed, one of nx = 12, N = 200 0.29 and 0.36, one of nx = 24, N = 1000 (8
// stages a team) 0.96 and 0.85.
inline int fused_cluster(int nx, const SolveRoom& r, int batch, int max_N)
{
    const int room = r.sms * 11 / 10;
    if (batch > room || batch > r.resident[0]) return 0;
    int c = 1, i = 0;
    while (i + 1 < kSolveSizes && batch <= r.resident[i + 1] && batch * c * 2 <= room &&
           (long long)c * 2 * r.teams * 10 <= (long long)max_N * 13) {
        c *= 2;
        ++i;
    }
    return max_N <= solve_stages(nx) * c * r.teams ? c : 0;
}

}  // namespace mhe
