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
// `bytes` of a stored value.  4 bytes: 116 registers at S = 2, 156 at S = 3, 208
// at S = 4 (242 with odd rows; three warps spill there: 72 G); 2 bytes, whose
// history is packed, at most 128 at every S.
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
// the busiest's: 1024 x 585 10.1 / 7.7, 256 x 2343 11.2 / 7.6; within the 1/6,
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

// ---- the lattices and ensembles that passes are for --------------------------
// Both state buffers together beyond 80 MB, about where they stop fitting in L2
// and the one-step kernel falls to the rate of HBM; or up to 32768 nodes, where
// a launch is mostly latency and one for four steps takes less than four.
// Between them the rows that segments share cost as much as the passes save
// (FP32, us per step, one-step / pass: 512^2 5.2 / 6.3).
constexpr long long kPipeBytes = 80LL << 20;
constexpr long long kPipeSmall = 32768;

// Microseconds of one step by the one-step kernels on GB300: picoseconds
// per node while the state fits in L2, beyond it, and where it is many times that,
// by `bytes` of a value.  An odd nx costs them a third (2 bytes; 4 bytes: a
// tenth), an even one that is no multiple of their widest vector a tenth.
// align: the largest power of two up to 8 that divides every nx.
inline double one_step_us(int bytes, long long nodes, int align, bool ensemble) {
    const double mb = 2.0 * 19.0 * bytes * (double)nodes * 1e-6;
    const double fit = ensemble ? (bytes == 2 ? 14.5 : 25.5) : (bytes == 2 ? 11.6 : 16.3);
    const double mid = ensemble ? (bytes == 2 ? 16.2 : 25.5) : (bytes == 2 ? 15.2 : 23.4);
    const double big = ensemble ? (bytes == 2 ? 14.2 : 25.5) : (bytes == 2 ? 12.9 : 23.2);
    const double x = std::min(std::max((mb - 84.0) / 63.0, 0.0), 1.0);
    const double y = std::min(std::max((mb - 300.0) / 900.0, 0.0), 1.0);
    double ps = fit + (mid - fit) * x + (big - mid) * y;
    if (align == 1) ps *= bytes == 2 ? 1.3 : 1.1;
    else if (bytes == 2 && align < (ensemble ? 4 : 8)) ps *= 1.08 + 0.09 * y;
    return ps * 1e-6 * (double)nodes;
}

// Whether passes of four steps are the faster way for these lattices (les 0, 1;
// one, or the runs of an ensemble).  A strip computes 64 columns whatever the
// lattice has, and rows around a segment whatever its rows, so this depends on
// the shape, not on the nodes alone (GB300, us per step, one-step / pass, FP32
// 2^21 nodes in rows of 8, 16, 24, 64 and 256: 48 / 122, 48 / 60, 48 / 40,
// 48 / 31, 48 / 20; in 1, 2 and 4 rows 48 / 70, 47 / 44, 47 / 32).
//
// Large: by the plan's time and that of four single steps.  Of 430 lattices
// and ensembles timed, none takes a pass that is more than 2% slower and none
// misses one that is more than 11% faster.
//
// Small lattices: while one warp per scheduler does with segments of a row --
// or of two rows where FP16 steps four nodes at a time, which is slower at such
// sizes -- (FP32 128^2 2.15 / 1.86, 16 x 1024 2.1 / 2.4, 64 x 512 2.0 / 2.3, 256 x
// 128 2.1 / 2.2, 1024 x 32 2.1 / 2.0; FP16 256 x 128 2.6 / 2.2), and not in rows
// so short that warps of different SMs write one sector (4 x 512 1.8 / 2.6).
// Odd rows of FP16, which are not fetched ahead, lose a tenth (99^2 2.2 / 2.4).
// Small ensembles, whose one-step launch takes 3.8 us: up to 14 warps per SM in
// segments of a row (128 runs of 16 x 16 3.9 / 3.3, of 8 x 32 3.9 / 5.2).
inline bool pipe_pays(int bytes, int nruns, const int* nx, const int* ny, bool ensemble, int sm_count) {
    constexpr int S = 4;
    auto strips = [&](int r) { return (long long)((nx[r] + pipe_useful(S) - 1) / pipe_useful(S)); };
    auto units_of = [&](int len) {
        long long u = 0;
        for (int r = 0; r < nruns; ++r) u += strips(r) * ((ny[r] + len - 1) / len);
        return u;
    };
    long long nodes = 0;
    int most = 1, align = 8;
    for (int r = 0; r < nruns; ++r) {
        nodes += (long long)nx[r] * ny[r];
        most = std::max(most, ny[r]);
        while (nx[r] % align) align /= 2;
    }
    if (2 * 19 * bytes * nodes >= kPipeBytes) {
        const int warps = ensemble ? batch_pipe_warps(bytes) : pipe_warps(bytes, S);
        return pipe_plan(S, warps, most, sm_count, units_of).us <= S * one_step_us(bytes, nodes, align, ensemble);
    }
    if (nodes > kPipeSmall) return false;
    if (ensemble) return units_of(1) <= 14LL * sm_count;
    const int rows = bytes == 2 && align >= 4 ? 2 : 1;
    return (nx[0] >= 8 || ny[0] <= 8) && units_of(rows) <= 4LL * sm_count;
}

// The kinetic closures, two steps per pass: only the large ones (les 2 FP32, us
// per step, one-step / pass: 128^2 3.0 / 3.6, 512^2 11.6 / 12.2, 1024^2 36.1 /
// 26.3).  Their one-step kernel sweeps strips of 256 columns, so narrow lattices
// gain the most (2^21 nodes in rows of 2, 16, 57, 113 and 256: 2015 / 1868, 347 /
// 131, 126 / 84, 86 / 65, 67 / 44); rows fewer than four are slower in a pass
// (1, 2, 3 rows: 76 / 143, 68 / 93, 69 / 76).
inline bool kin_pipe_pays(int bytes, int nx, int ny) {
    return 2LL * 19 * bytes * nx * ny >= kPipeBytes;
}

}  // namespace lbmhd
