// lbmhd_pipe_plan.h -- how a pass of several steps (lbmhd_step_pipe.cu) is cut
// into warps (plain host C++, no CUDA types, so that it can be checked on its
// own).
#pragma once

#include <algorithm>

namespace lbmhd {

// Columns of a strip: a warp computes 64 and stores pipe_useful(S), the rest is
// the halo of S steps (rounded up to even on the left).
constexpr int pipe_halo(int S) { return (S + 1) / 2 * 2; }
constexpr int pipe_useful(int S) { return (64 - pipe_halo(S) - S) / 2 * 2; }

// Warps per scheduler that the registers are cut for (65536 / 128 / warps);
// `bytes` of a stored value.  4 bytes: 128 registers at S = 2, 168 at S = 3, 255
// at S = 4 (three warps spill there: 72 G); 2 bytes, whose history is packed,
// 128 at every S.
constexpr int pipe_warps(int bytes, int S) { return bytes == 2 || S == 2 ? 4 : (S == 3 ? 3 : 2); }
// An ensemble's run rates are read by every lane into registers.
constexpr int batch_pipe_warps(int bytes) { return bytes == 2 ? 3 : 2; }

struct PipePlan {
    int seglen;  // rows of a segment
    double us;   // expected time of the pass
};

// Rows per segment, at most 96 (longer ones let neighbouring strips drift
// apart and their shared columns leave L2: 8192^2, S = 4, 96 rows 127.9 G,
// 192 rows 124 G).  Two estimates of a pass, in microseconds at 152 SMs:
//
// The mean over the schedulers, which is what counts when other work fills the
// rest of them: rounds of resident warps at a + b w a row for w of them on a
// scheduler, a part of a warp as that part.
//
// The busiest scheduler, which is what one run on its own takes: whole warps,
// w = ceil(units / schedulers), `warps` at a time (measured on GB300, S = 4,
// either format: 1.4, 2.25, 3.2, 4.15 a row at 1 to 4) times the rows of a
// segment and S - 1/2 for those around it, most of whose steps are not taken.
//
// The length is the best by the mean unless that leaves the busiest scheduler
// more than 1/6 above the least, as where a few schedulers get one warp more:
// then it is the best by the busiest.  FP32, us per step, the mean's length /
// the busiest's: 1024 x 585 10.1 / 8.0, 256 x 2343 11.2 / 8.4; within the 1/6,
// 1024^2 (19 / 16 rows) 12.3 / 11.0 for one run but 10.20 / 10.38 for two at once.
template <class Units>
PipePlan pipe_plan(int S, int warps, int most, int sm_count, Units units_of) {
    const int longest = std::min(most, 96);
    const long long sched = 4LL * sm_count, resident = sched * warps;
    auto mean = [&](int len) {
        const double a = S == 2 ? 0.8 : (S == 3 ? 0.56 : 0.45), b = S == 2 ? 0.6 : (S == 3 ? 0.61 : 0.8);
        const long long units = units_of(len), rest = units % resident;
        double t = (double)(units / resident) * (a + b * warps);
        if (rest) t += a + b * (rest > sched ? (double)rest / (double)sched : 1.0);
        return t * (len + 2 * S - 1);
    };
    auto busiest = [&](int len) {
        const double a = S == 2 ? 0.8 : (S == 3 ? 0.56 : 0.48), b = S == 2 ? 0.6 : (S == 3 ? 0.61 : 0.9);
        const long long w = (units_of(len) + sched - 1) / sched, rest = w % warps;
        return ((double)(w / warps) * (a + b * warps) + (rest ? a + b * (double)rest : 0.0)) * (len + S - 0.5);
    };
    int by_mean = 1, by_busiest = 1;
    double least_mean = 1e300, least = 1e300;
    for (int len = 1; len <= longest; ++len) {
        if (const double t = mean(len); t < least_mean) {
            least_mean = t;
            by_mean = len;
        }
        if (const double t = busiest(len); t < least) {
            least = t;
            by_busiest = len;
        }
    }
    const double t = busiest(by_mean);
    return t > least * (7.0 / 6.0) ? PipePlan{by_busiest, least} : PipePlan{by_mean, t};
}

}  // namespace lbmhd
