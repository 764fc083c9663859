"""How passes of several steps are cut into warps (csrc/lbmhd_pipe_plan.h), on
the host: the header is plain C++, compiled here with g++ into a small driver.

The segment length must leave the busiest scheduler at most 1/6 above the least.
Measured on GB300 (152 SMs, us per step, a length that gives a few schedulers
one warp more / this): FP32 1024 x 585 10.1 / 8.0, 256 x 2343 11.2 / 8.4.
"""
import os
import shutil
import subprocess

import pytest

from conftest import ROOT

DRIVER = r"""
#include <cstdio>
#include "lbmhd_pipe_plan.h"
using namespace lbmhd;
int main() {
    int S, bytes, nx, ny, sms;
    while (std::scanf("%d %d %d %d %d", &S, &bytes, &nx, &ny, &sms) == 5) {
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

