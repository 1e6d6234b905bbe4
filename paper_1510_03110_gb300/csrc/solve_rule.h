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

// CTAs per instance of the corrections after the first four, in one launch, or 0 to go on with a launch per pass.  A solve
// that has converged by then (the usual one) saves the empty passes of every correction still allowed, 0.04 each: 0.5
// with 16 allowed.  One that has not should not pay much for it, whether one instance works on or all do.  So few
// instances take clusters that fill the GPU, many take one CTA, more (up to four) where a single instance of the
// longest horizon would leave a team more than 64 stages; beyond 64 a team (32 with eight CTAs and more, which only few
// instances take and then leave most of the GPU idle) the passes go on.  Measured (nx, batch, N; passes and this rule's
// cluster), 16 corrections allowed, converged after four or before, and all 16 used:
//   24, 1, 1000             1.46  0.94 (16 CTAs);    2.73  3.08    (four CTAs: 5.91)
//   24, 1, 2000             1.57  1.03 (16);         2.97  4.25    (four: 10.2)
//   12, 1, 6000             1.45  0.86 (16);         2.94  4.28    (four: 11.0)
//   24, 8, 1000             1.94  1.34 (8);          3.91  4.84
//   20, 30, <= 512          1.50  0.98 (4);          3.37  4.61
//   24, 60, <= 600          2.56  2.04 (2);          5.91  7.95
//   24, 512, <= 2048        26.9  26.4 (4);          83.5  163     (one CTA: 106)
//   12, 1024, <= 2048       12.2  11.7 (2);          47.5  80.8    (four: 127)
//   12, 1024, <= 512        4.75  4.15 (1);          16.0  23.0
//   6, 1024, <= 2048        5.56  5.01 (1);          20.8  25.3
//   4, 2000, <= 60          0.97  0.53 (1);          2.21  4.41    (four: 16.2)
// Left to the passes: 20, 1, 16384 (2.46 and 1.80 converged, but 5.2 and 17.5 with 16 CTAs, 59 with four).
inline int resumed_cluster(const SolveRoom& r, int batch, int max_N)
{
    const int room = r.sms * 11 / 10;
    int c = 1, i = 0;
    if (r.resident[0] < 1) return 0;
    while (i + 1 < kSolveSizes && batch <= r.resident[i + 1] && batch * c * 2 <= room) {
        c *= 2;
        ++i;
    }
    while (c < 4 && r.resident[i + 1] > 0 && max_N > 64 * c * r.teams) {
        c *= 2;
        ++i;
    }
    return max_N <= (c >= 8 ? 32 : 64) * c * r.teams ? c : 0;
}

}  // namespace mhe
