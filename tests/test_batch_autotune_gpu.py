"""The ensemble autotuner keeps what it found fastest, passes of four steps or
single ones, and a cached entry brings back what it was measured with."""
import json

import pytest

from paper_1607_08675_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def L():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1607_08675_gb300 import build, lbmhd

    build.build()
    return lbmhd


def launches_of_eight_steps(L, sizes, prec, cache):
    nx, ny = [s[0] for s in sizes], [s[1] for s in sizes]
    n = len(sizes)
    b = L.lbmhd_batch_create(nx, ny, [0.6] * n, [0.6] * n, [0.1] * n, L.lbmhd_params_default(precision=prec))
    try:
        rate = L.lbmhd_batch_autotune(b, cache, 8)
        shape = L.lbmhd_batch_get_launch(b)
        for r, s in enumerate(sizes):
            L.lbmhd_batch_init(b, r, *inputs.orszag_tang(*s, seed=1, amp=1e-3))
        before = L.lbmhd_batch_launch_count(b)
        L.lbmhd_batch_step(b, 8)
        return rate, shape, L.lbmhd_batch_launch_count(b) - before
    finally:
        L.lbmhd_batch_destroy(b)


@pytest.mark.parametrize("prec,sizes", [("fp32", [(256, 256)] * 10), ("fp16_dev", [(512, 512)] * 6)])
def test_the_cached_entry_says_whether_its_rate_is_that_of_passes(L, prec, sizes, tmp_path):
    cache = str(tmp_path / "tune.json")
    rate, shape, launches = launches_of_eight_steps(L, sizes, prec, cache)
    (key, entry), = json.load(open(cache)).items()
    assert tuple(entry[:3]) == shape and entry[3] == pytest.approx(rate, abs=0.1)
    assert launches == (2 if entry[4] else -(-8 // shape[2]))

    def again(value):
        json.dump({key: value}, open(cache, "w"))
        return launches_of_eight_steps(L, sizes, prec, cache)

    # a shape that won over passes is used for every step
    assert again([4, 64, 1, 123.0, 0]) == (123.0, (4, 64, 1), 8)
    assert again([4, 128, 8, 124.0, 0]) == (124.0, (4, 128, 8), 1)
    assert again([4, 64, 1, 125.0, 1]) == (125.0, (4, 64, 1), 2)
    # an entry without a word on passes: the rule, by which these ensembles take them
    assert again([4, 64, 1, 126.0]) == (126.0, (4, 64, 1), 2)


def test_an_ensemble_that_is_not_for_passes_never_takes_them(L, tmp_path):
    cache = str(tmp_path / "tune.json")
    sizes = [(8, 512)] * 256
    _, shape, launches = launches_of_eight_steps(L, sizes, "fp32", cache)
    (key, entry), = json.load(open(cache)).items()
    assert entry[4] == 0 and launches == -(-8 // shape[2])
    json.dump({key: [4, 64, 1, 1.0, 1]}, open(cache, "w"))
    assert launches_of_eight_steps(L, sizes, "fp32", cache)[2] == 8
