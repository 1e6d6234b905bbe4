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

// CTAs per instance of a larger batch's corrections after the first four, in one launch, or 0 to go on with a launch
// per pass.  A solve that has converged by then (the usual one) saves the empty passes of every correction still
// allowed; one that has not should not pay much for it, whether one instance works on or all do: one CTA, or two,
// which is as far as the few chunks of an instance keep the teams busy.  Measured, twelve corrections allowed,
// passes and clusters of 1, 2, 4, with none, a few and all instances working on after the fourth:
//   MHE form, 1024 of nx = 6, N <= 2048:  4.11  3.74 3.74 3.75;  7.43  6.76 6.69 6.70;  16.2  19.0 20.7 28.8
//   MHE form, 200 of nx = 12, N <= 300:   1.03  0.73 0.73 0.73;  1.50  1.23 1.21 1.21;   2.5   3.5  3.7  5.6
//   Q form, 500 of nx = 4, N <= 512:      1.03  0.65 0.65 0.65;  1.68  1.44 1.38 1.35;   3.0   3.3  4.4  6.5
//   Q form, 256 of nx = 12, N <= 512:     1.31  0.92 0.92 0.93;  2.48  2.23 2.15 2.11;   4.7   7.5  7.4  9.6
// Left to the passes: few instances or long horizons (16 corrections used: one of nx = 20, N = 16384, 5.1 by passes
// and 55 resumed with four CTAs; one of nx = 24, N = 2000 2.8 and 9.6), horizons with fewer chunks than teams (2000
// of nx = 4, N <= 60: all 1.8 and 3.6), and above nx = 8 large batches (1024 of nx = 12, N <= 512: none 3.1 and
// 2.8, all 11.2 and 18.9).
inline int resumed_cluster(int nx, const SolveRoom& r, int batch, int max_N)
{
    if (2 * batch < r.sms || max_N < 4 * r.teams || (nx > 8 && batch > 2 * r.sms)) return 0;
    const int most = (nx <= 8 ? 32 : solve_stages(nx)) * r.teams;   // stages of one CTA
    if (r.resident[0] > 0 && max_N <= most) return 1;
    return r.resident[1] > 0 && max_N <= 2 * most ? 2 : 0;
}

}  // namespace mhe
