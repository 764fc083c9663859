"""Which lattices take passes of several steps and how these are cut into warps
(csrc/lbmhd_pipe_plan.h), on the host: the header is plain C++, compiled here with g++ into a small driver.

The segment length must leave the busiest scheduler at most 1/6 above the least.
Measured on GB300 (152 SMs, us per step, a length that gives a few schedulers
one warp more / this): FP32 1024 x 585 10.1 / 7.7, 256 x 2343 11.2 / 7.6.
"""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

DRIVER = r"""
#include <cstdio>
#include <vector>
#include "lbmhd_pipe_plan.h"
using namespace lbmhd;
int main() {
    int S, bytes, nx, ny, sms;
    while (std::scanf("%d %d %d %d %d", &S, &bytes, &nx, &ny, &sms) == 5) {
        if (S <= 1) {  // S = 0: the lattice; S < 0: an ensemble of -S such runs
            const std::vector<int> w(S ? -S : 1, nx), h(S ? -S : 1, ny);
            std::printf("%d\n", (int)pipe_pays(bytes, (int)w.size(), w.data(), h.data(), S < 0, sms));
            continue;
        }
        const int strips = (nx + pipe_useful(S) - 1) / pipe_useful(S);
        const PipePlan p = pipe_plan(S, pipe_warps(bytes, S), ny, sms,
                                     [&](int len) { return (long long)strips * ((ny + len - 1) / len); });
        std::printf("%d %.17g %d %d\n", p.seglen, p.us, strips, pipe_warps(bytes, S));
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("pipe_plan")
    src, exe = d / "plan.cpp", d / "plan"
    src.write_text(DRIVER)
    inc = os.path.join(ROOT, "paper_1607_08675_gb300", "csrc")
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", inc, str(src), "-o", str(exe)], check=True)

    def ask(*rows):
        text = "".join(" ".join(map(str, r)) + "\n" for r in rows)
        out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
        return [tuple(float(v) for v in line.split()) for line in out.splitlines()]

    return ask


SHAPES = [(1024, 585), (256, 2343), (512, 1171), (1024, 1024), (256, 128), (774, 775), (8192, 8192),
          (57, 3), (1, 1), (300, 2001), (1 << 24, 3), (5, 1 << 20)]


@pytest.mark.parametrize("S", [2, 3, 4])
@pytest.mark.parametrize("bytes_", [4, 2])
@pytest.mark.parametrize("sms", [152, 76])
def test_the_busiest_scheduler_has_little_more_than_the_least_work(driver, S, bytes_, sms):
    """Counting part of a warp as that part of its time took 15 rows for FP32
    1024 x 585: 741 units, two warps on some schedulers and one on most, 1.37
    times the least."""
    for (nx, ny), (length, us, strips, warps) in zip(SHAPES, driver(*[(S, bytes_, *s, sms) for s in SHAPES])):
        a, b = {2: (0.8, 0.6), 3: (0.56, 0.61), 4: (0.48, 0.9)}[S]

        def cost(n):
            w = -(-int(strips) * -(-ny // n) // (4 * sms))  # warps of the busiest scheduler
            full, rest = divmod(w, int(warps))
            return (full * (a + b * warps) + (a + b * rest if rest else 0)) * (n + S - 0.5)

        assert 1 <= length <= min(ny, 96)
        assert us == pytest.approx(cost(int(length)))
        assert us <= (7 / 6 + 1e-9) * min(cost(n) for n in range(1, min(ny, 96) + 1))



# us per step on GB300: one-step / pass (bytes of a value, nx, ny)
LATTICES = [
    # narrow: the rest of 64 columns is computed for nothing
    (4, 8, 262144, 48.5, 121.7), (4, 16, 131072, 48.5, 60.4), (4, 28, 74898, 48.6, 36.9),
    (4, 64, 32768, 48.3, 33.0), (4, 57, 36792, 60.6, 39.8), (4, 12, 1398101, 364, 606),
    (2, 16, 131072, 33.0, 59.1), (2, 24, 87381, 33.1, 40.8), (2, 60, 25000, 23.5, 25.2),
    (2, 64, 23437, 21.1, 23.9), (2, 48, 43690, 33.1, 22.2), (2, 57, 294337, 351, 273),
    # flat: the rows around a segment
    (4, 2097152, 1, 48.3, 69.8), (4, 524288, 4, 47.1, 32.3), (2, 1048576, 2, 29.3, 40.0),
    (2, 262144, 8, 32.1, 23.1), (4, 300000, 2, 11.0, 13.3),
    # ordinary ones on both sides of L2
    (4, 1024, 585, 10.4, 8.0), (4, 1024, 1024, 26.0, 12.3), (4, 8192, 8192, 1463, 526),
    (2, 2048, 2048, 60, 37), (2, 1024, 1131, 13.8, 13.9), (4, 512, 512, 5.8, 6.3),
    # small
    (4, 64, 64, 2.15, 1.76), (4, 128, 128, 2.15, 1.86), (4, 256, 128, 2.09, 2.62), (4, 64, 512, 2.0, 2.33),
    (4, 32, 1024, 2.0, 2.29), (4, 1024, 32, 2.1, 2.0), (4, 16, 1024, 2.14, 2.38), (4, 4, 8192, 2.0, 10.2),
    (4, 1, 1024, 1.8, 7.4), (4, 4, 512, 1.81, 2.57), (2, 256, 128, 2.6, 2.2), (2, 16, 2048, 2.6, 3.0),
    (2, 113, 289, 2.3, 2.9), (2, 18, 251, 2.1, 1.9),
]
ENSEMBLES = [  # bytes, runs, nx, ny
    (4, 256, 8, 512, 28.8, 68.2), (4, 256, 16, 256, 29.0, 35.4), (4, 256, 64, 64, 28.7, 19.7),
    (4, 16, 256, 256, 28.5, 12.4), (2, 323, 64, 64, 21.0, 29.2), (2, 282, 64, 64, 17.2, 20.8),
    (2, 132, 100, 100, 21.8, 16.8), (2, 80, 32, 512, 20.8, 29.1), (4, 128, 8, 32, 3.9, 5.2),
    (4, 32, 8, 128, 3.9, 4.8), (4, 128, 16, 16, 3.9, 3.3), (4, 8, 64, 64, 3.9, 2.4), (2, 16, 32, 32, 3.8, 2.1),
]


def test_passes_are_taken_where_they_are_faster(driver):
    rows = [(0, b, nx, ny, 152) for b, nx, ny, *_ in LATTICES] + [(-k, b, nx, ny, 152) for b, k, nx, ny, *_ in ENSEMBLES]
    for row, (pays,) in zip(LATTICES + ENSEMBLES, driver(*rows)):
        one, many = row[-2:]
        if abs(one / many - 1) > 0.04:  # else either will do
            assert bool(pays) == (many < one), row
