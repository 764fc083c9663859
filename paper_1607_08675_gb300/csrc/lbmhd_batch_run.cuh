// lbmhd_batch_run.cuh -- one run of an ensemble as the device sees it
// (shared by the ensemble step kernel and the ensemble kinetic kernels).
#pragma once

#include "lbmhd_device.cuh"

namespace lbmhd {

template <class R>
struct RunDev {
    long long off;   // element offset of the run's 19 planes in each state buffer
    long long moff;  // element offset of its 5 moment planes (les 2, 3)
    long long ps;    // plane stride (elements)
    int nx, ny;
    unsigned total;  // live threads of the run (nx / V * ny)
    unsigned unit0;  // first work unit of the run
    int kstrips;     // fused kinetic kernel: column strips of the run
    int kseglen;     // ... and rows per segment (units = strips x segments)
    Coll<R> c;
};

static_assert(sizeof(Coll<float>) == 68 && sizeof(RunDev<float>) == 120,
              "read by every thread of the step kernels: what only some of them use goes elsewhere");

// A run's share of a pass of several steps: its first unit, column strips and
// rows per segment.  Not part of RunDev, which every thread of the other
// kernels reads: three words more there cost the fused kinetic kernels up to 5%
// (12 runs of 128^2, us per step: les 2 FP16 115.0 / 119.6, les 3 FP32 122.4 /
// 128.1).
struct RunPass {
    unsigned unit0;
    int strips, seglen;
};

}  // namespace lbmhd
