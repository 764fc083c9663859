"""Several steps per launch (csrc/lbmhd_step_pipe.cu) against single steps.

The kernel performs the operations of the one-step kernel in their order, so
the states must be equal bit for bit (tolerance zero), whatever the lattice:
narrower than a strip's halo, at and around the 60, 56 and 2 x 56 columns that
a strip stores, odd rows, fewer rows than the steps of a launch.
"""
import numpy as np
import pytest

from paper_1607_08675_gb300 import inputs

pytestmark = pytest.mark.gpu

RATES = dict(tau_nu=0.6, tau_eta=0.65, C_S=0.1)
SMALL = [(1, 1), (2, 1), (1, 7), (3, 5), (55, 3), (56, 4), (57, 2), (60, 9), (61, 97), (112, 96),
         (113, 193), (64, 64), (130, 67)]
# beyond 80 MB in two buffers (FP32), odd and even rows, several rounds of warps
LARGE = [(1999, 301), (300, 2001)]


@pytest.fixture(scope="module")
def L():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_1607_08675_gb300 import build, lbmhd

    build.build()
    return lbmhd


def raw(L, shape, fields, prec, les, calls, single):
    p = L.lbmhd_params_default(precision=prec, les=les, **RATES)
    h = L.lbmhd_create(*shape, p)
    try:
        if single:
            L.lbmhd_set_launch(h, 1, 64)
        L.lbmhd_init(h, *fields)
        for n in calls:
            L.lbmhd_step(h, n)
        assert L.lbmhd_step_count(h) == sum(calls)
        return L.lbmhd_get_state_raw(h), L.lbmhd_launch_count(h)
    finally:
        L.lbmhd_destroy(h)


@pytest.mark.parametrize("prec", ["fp32", "fp32_dev", "fp16_dev"])
@pytest.mark.parametrize("shape", SMALL + LARGE)
def test_several_steps_per_launch_equal_single_steps(L, prec, shape):
    fields = inputs.orszag_tang(*shape, seed=3, amp=1e-3)
    # 2, 3 and 4 steps per launch, mixtures of them, and a lone step
    calls = (2, 3, 4, 5, 7, 1) if shape in SMALL else (4, 6)
    for les in (1, 0):
        got, launches = raw(L, shape, fields, prec, les, calls, False)
        ref, one = raw(L, shape, fields, prec, les, calls, True)
        assert np.array_equal(got, ref), (shape, les)
        assert one == sum(calls)
        if shape in SMALL:
            assert launches == 8


# about 1.2 M nodes, where the kinetic closures take two steps per pass: one and
# two nodes wide or high, and around the 56 columns that a strip stores
THIN = [(1, 1200000), (1200000, 1), (2, 600000), (400001, 3), (55, 21819), (57, 21053), (113, 10620)]


@pytest.mark.parametrize("prec", ["fp32", "fp32_dev", "fp16_dev"])
@pytest.mark.parametrize("shape", THIN)
def test_two_steps_of_a_kinetic_closure_equal_single_steps(L, prec, shape):
    """les 2 and 3, two steps per launch, against the one-step fused kernel
    (vec 1) bit for bit."""
    fields = inputs.orszag_tang(*shape, seed=3, amp=1e-3)
    for les in (2, 3):
        got, launches = raw(L, shape, fields, prec, les, (2, 3), False)
        ref, one = raw(L, shape, fields, prec, les, (2, 3), True)
        assert np.array_equal(got, ref), (shape, les)
        assert one == 5 and launches == 3


def test_several_steps_per_launch_with_tied_rates_and_graph_replay(L):
    """Rates s_7, s_8 tied to the local s_nu and a run long enough for graph
    replay, in calls that leave the buffers in either parity."""
    shape = (114, 90)
    fields = inputs.turbulence(*shape, kmin=2, kmax=5, seed=5)
    ref = raw(L, shape, fields, "fp32", 1, (133,), True)[0]
    for calls in ((133,), (3, 130), (64, 1, 68)):
        assert np.array_equal(raw(L, shape, fields, "fp32", 1, calls, False)[0], ref)


def test_finiteness_check_between_launches(L):
    """check_finite_every counts steps, not launches: the check after step 3
    of a ten-step call sees the state of step 3."""
    shape = (48, 40)
    fields = inputs.orszag_tang(*shape, seed=1)
    p = L.lbmhd_params_default(precision="fp32", check_finite_every=3, **RATES)
    h = L.lbmhd_create(*shape, p)
    try:
        L.lbmhd_init(h, *fields)
        L.lbmhd_step(h, 10)
        L.lbmhd_sync(h)
        got = L.lbmhd_get_state_raw(h)
        assert L.lbmhd_launch_count(h) == 4  # 3 + 3 + 3 + 1 steps
    finally:
        L.lbmhd_destroy(h)
    assert np.array_equal(got, raw(L, shape, fields, "fp32", 1, (10,), True)[0])


@pytest.mark.parametrize("prec", ["fp32", "fp32_dev", "fp16_dev"])
@pytest.mark.parametrize("sizes", [[(64, 40), (57, 3), (8, 8)], [(112, 9), (56, 33), (2, 1), (130, 64)],
                                   [(640, 701), (96, 100), (513, 300)]])
def test_ensemble_passes_equal_single_lattices(L, prec, sizes):
    """Runs of uneven sizes, odd and even, one below and one above the size
    from which an ensemble leaves L2; calls that mix passes of four steps,
    graph replay and single steps."""
    nx, ny = [s[0] for s in sizes], [s[1] for s in sizes]
    tau, cs = [0.55 + 0.02 * i for i in range(len(sizes))], [0.1 + 0.01 * i for i in range(len(sizes))]
    rates = dict(s5=1.2, s6=1.2, s7=1.3, s8=1.3)
    calls = (3, 4, 33, 6)
    f = [inputs.orszag_tang(*s, seed=i, amp=1e-3) for i, s in enumerate(sizes)]
    b = L.lbmhd_batch_create(nx, ny, tau, tau, cs, L.lbmhd_params_default(precision=prec, **rates))
    try:
        for r in range(len(sizes)):
            L.lbmhd_batch_init(b, r, *f[r])
        for n in calls:
            L.lbmhd_batch_step(b, n)
        assert L.lbmhd_batch_step_count(b) == sum(calls)
        got = [L.lbmhd_batch_get_state(b, r) for r in range(len(sizes))]
    finally:
        L.lbmhd_batch_destroy(b)
    for r, s in enumerate(sizes):
        h = L.lbmhd_create(*s, L.lbmhd_params_default(precision=prec, tau_nu=tau[r], tau_eta=tau[r],
                                                      C_S=cs[r], **rates))
        try:
            L.lbmhd_set_launch(h, 1, 64)
            L.lbmhd_init(h, *f[r])
            L.lbmhd_step(h, sum(calls))
            assert np.array_equal(L.lbmhd_get_state(h), got[r]), s
        finally:
            L.lbmhd_destroy(h)
