"""Passes of several steps on lattices and ensembles beyond L2, in every format.

test_pipe_gpu.py compares passes with single steps on small lattices; its large
ones are beyond 80 MB at four bytes per value only.  Here the size follows the
format, odd and even rows are both there, and every case asserts the launches,
so that a case that takes single steps on both sides fails.
"""
import numpy as np
import pytest

from paper_1607_08675_gb300 import inputs

pytestmark = pytest.mark.gpu

RATES = dict(tau_nu=0.6, tau_eta=0.65, C_S=0.1)
# several rounds of warps and a part of one; segments that do not divide the rows
LATTICES = {"fp32": [(1999, 301), (300, 2001), (1024, 1100)],
            "fp16_dev": [(1999, 701), (300, 4001), (301, 6001), (1024, 2200)]}
LATTICES["fp32_dev"] = LATTICES["fp32"]
ENSEMBLES = {"fp32": [[(640, 701), (96, 100), (513, 300)], [(640, 1201), (96, 100), (514, 700)]],
             "fp16_dev": [[(640, 1201), (96, 100), (513, 1300)], [(130, 1201), (96, 100), (1026, 1100)]]}
ENSEMBLES["fp32_dev"] = ENSEMBLES["fp32"]


@pytest.fixture(scope="module")
def L():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1607_08675_gb300 import build, lbmhd

    build.build()
    return lbmhd


def run(L, shape, prec, les, calls, single, state=None, fields=None):
    h = L.lbmhd_create(*shape, L.lbmhd_params_default(precision=prec, les=les, **RATES))
    try:
        if single:
            L.lbmhd_set_launch(h, 1, 64)
        L.lbmhd_init(h, *fields)
        if state is not None:
            L.lbmhd_set_state_raw(h, state)
        for n in calls:
            L.lbmhd_step(h, n)
        return L.lbmhd_get_state_raw(h), L.lbmhd_launch_count(h)
    finally:
        L.lbmhd_destroy(h)


@pytest.mark.parametrize("prec,shape", [(p, s) for p in LATTICES for s in LATTICES[p]])
def test_large_lattices_take_passes_that_equal_single_steps(L, prec, shape):
    fields = inputs.orszag_tang(*shape, seed=3, amp=1e-3)
    for les in (1, 0):
        got, launches = run(L, shape, prec, les, (4, 6, 2), False, fields=fields)
        ref, one = run(L, shape, prec, les, (4, 6, 2), True, fields=fields)
        assert np.array_equal(got, ref), les
        assert (launches, one) == (4, 12)  # 4, 3 + 3 and 2 steps


@pytest.mark.parametrize("prec,sizes", [(p, s) for p in ENSEMBLES for s in ENSEMBLES[p]])
def test_large_ensembles_take_passes_that_equal_single_lattices(L, prec, sizes):
    nx, ny = [s[0] for s in sizes], [s[1] for s in sizes]
    tau, cs = [0.55 + 0.02 * i for i in range(len(sizes))], [0.1 + 0.01 * i for i in range(len(sizes))]
    f = [inputs.orszag_tang(*s, seed=i, amp=1e-3) for i, s in enumerate(sizes)]
    calls = (3, 4, 33, 6)
    b = L.lbmhd_batch_create(nx, ny, tau, tau, cs, L.lbmhd_params_default(precision=prec))
    try:
        for r in range(len(sizes)):
            L.lbmhd_batch_init(b, r, *f[r])
        for n in calls:
            L.lbmhd_batch_step(b, n)
        # a pass per four steps, and the one to three steps that are left in one launch
        assert L.lbmhd_batch_launch_count(b) == 1 + 1 + (8 + 1) + (1 + 1)
        got = [L.lbmhd_batch_get_state(b, r) for r in range(len(sizes))]
    finally:
        L.lbmhd_batch_destroy(b)
    for r, s in enumerate(sizes):
        h = L.lbmhd_create(*s, L.lbmhd_params_default(precision=prec, tau_nu=tau[r], tau_eta=tau[r], C_S=cs[r]))
        try:
            L.lbmhd_set_launch(h, 1, 64)
            L.lbmhd_init(h, *f[r])
            L.lbmhd_step(h, sum(calls))
            assert np.array_equal(L.lbmhd_get_state(h), got[r]), s
        finally:
            L.lbmhd_destroy(h)


@pytest.mark.parametrize("prec,shape", [("fp32", (8, 70000)), ("fp32", (600000, 1)), ("fp16_dev", (16, 80000)),
                                        ("fp32", (256, 128)), ("fp16_dev", (4, 8192))])
def test_narrow_and_flat_lattices_take_single_steps(L, prec, shape):
    fields = inputs.orszag_tang(*shape, seed=3, amp=1e-3)
    got, launches = run(L, shape, prec, 1, (5,), False, fields=fields)
    ref, one = run(L, shape, prec, 1, (5,), True, fields=fields)
    assert np.array_equal(got, ref) and launches == one == 5


@pytest.mark.parametrize("prec", ["fp32", "fp32_dev", "fp16_dev"])
@pytest.mark.parametrize("les,shape", [(1, (128, 64)), (1, (57, 33)), (2, (1200, 1000)), (3, (1200, 1000))])
def test_negative_zeros_change_no_value(L, prec, les, shape):
    """A state with negative zeros, which the packed product does not keep: the
    same values as single steps of one node per thread, and the same bits
    wherever the value is not zero."""
    nx, ny = shape
    g = np.random.default_rng(2)
    dev = np.where(g.random((19, ny, nx)) < 0.5, -0.0, 0.0)
    dev[:, : ny // 2] += np.where(g.random((19, ny // 2, nx)) < 0.3, 0.0, g.normal(0, 0.01, (19, ny // 2, nx)))
    if prec == "fp32":
        dev[:9] += np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)[:, None, None]
    scale, dtype = {"fp32": (1, np.float32), "fp32_dev": (1, np.float32), "fp16_dev": (1024, np.float16)}[prec]
    state = (dev * scale).astype(dtype)
    fields = [np.ones((ny, nx))] + [np.zeros((ny, nx))] * 4
    n = 4 if les == 1 else 2
    got, launches = run(L, shape, prec, les, (n,), False, state, fields)
    ref, one = run(L, shape, prec, les, (n,), True, state, fields)
    assert (launches, one) == (1, n)
    assert np.array_equal(got, ref)
    bits = {2: np.uint16, 4: np.uint32}[got.dtype.itemsize]
    other = np.ascontiguousarray(got).view(bits) != np.ascontiguousarray(ref).view(bits)
    assert not np.any(got[other])
