"""Initialisation and read-back of the FP32 forms (csrc/lbmhd_narrow.cuh).

The stored state must be the FP64 equilibria rounded once: FP32 storage equals
the FP64 handle's populations cast to FP32, FP32 deviations equal the high
words of the double-word deviations (which are the FP64 deviations rounded),
FP16 deviations those times the scale in binary16 -- bit for bit, for fields at
rest, with exact zeros, aligned, tiny, large and out of the range that the fast
path takes.  The moments are compared with the same sums in extended
precision: the sums of 24-bit values are exact in FP64 and the quotient is
rounded once or corrected, so 4 ulp (relative) bounds them.
"""
import numpy as np
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


def fields(kind, shape, nf):
    g = np.random.default_rng(11)
    n = (nf - 1) // 2
    rho = np.ones(shape)
    v = [g.normal(0, 0.05, shape) for _ in range(2 * n)]
    if kind == "rest":
        v = [np.zeros(shape) for _ in v]
    elif kind == "zeros":  # single components that vanish
        for k, a in enumerate(v):
            a[..., k::3] = 0.0
    elif kind == "aligned":
        v[n:] = [a.copy() for a in v[:n]]
        rho = 1.0 + g.normal(0, 1e-3, shape)
    elif kind == "tiny":
        v = [a * 10.0 ** g.uniform(-25, 0, shape) for a in v]
        rho = 1.0 + g.normal(0, 1.0, shape) * 10.0 ** g.uniform(-17, -1, shape)
    elif kind == "large":
        v = [a * 10.0 ** g.uniform(0, 3, shape) for a in v]
        rho = 10.0 ** g.uniform(-2, 2, shape)
    elif kind == "extreme":  # leaves the fast path's range in places
        v = [a * 10.0 ** g.choice([-40.0, -5.0, 0.0, 4.0], shape) for a in v]
    return [rho, *v]


KINDS = ["rest", "zeros", "aligned", "tiny", "large", "extreme"]


def states(create, init, raw, destroy, L, dims, f):
    out = {}
    for prec in ("fp64", "fp32", "fp32_dev", "fp16_dev", "ff"):
        if prec == "fp32_dev" and len(dims) == 3:
            continue  # 3D has no such format
        h = create(*dims, L.lbmhd_params_default(precision=prec))
        try:
            init(h, *f)
            out[prec] = raw(h)
        finally:
            destroy(h)
    return out


def check(st):
    same = lambda a, b: np.array_equal(a, b, equal_nan=True)
    with np.errstate(over="ignore"):
        assert same(st["fp32"], st["fp64"].astype(np.float32))
        hi = st["ff"][..., 0]
        if "fp32_dev" in st:
            assert same(st["fp32_dev"], hi)
        assert same(st["fp16_dev"], (hi * np.float32(1024.0)).astype(np.float16))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(1, 1), (37, 23), (300, 200)])
def test_stored_state_is_the_fp64_equilibria_rounded_once(L, kind, shape):
    nx, ny = shape
    check(states(L.lbmhd_create, L.lbmhd_init, L.lbmhd_get_state_raw, L.lbmhd_destroy, L,
                 shape, fields(kind, (ny, nx), 5)))


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("shape", [(1, 1, 1), (40, 31, 27)])
def test_3d_stored_state_is_the_fp64_equilibria_rounded_once(L, kind, shape):
    nx, ny, nz = shape
    check(states(L.lbmhd3_create, L.lbmhd3_init, L.lbmhd3_get_state_raw, L.lbmhd3_destroy, L,
                 shape, fields(kind, (nz, ny, nx), 7)))


def test_a_density_that_is_not_positive_is_still_refused(L):
    f = inputs.orszag_tang(16, 8)
    for prec in ("fp32", "fp32_dev", "fp16_dev"):
        for bad in (0.0, -1.0, np.nan, np.inf):
            h = L.lbmhd_create(16, 8, L.lbmhd_params_default(precision=prec))
            rho = f[0].copy()
            rho[3, 5] = bad
            with pytest.raises(L.LBMHDError):
                L.lbmhd_init(h, rho, *f[1:])
            L.lbmhd_destroy(h)


@pytest.mark.parametrize("prec", ["fp32", "fp32_dev", "fp16_dev"])
@pytest.mark.parametrize("kind", ["zeros", "aligned", "tiny", "large"])
def test_moments_of_the_fp32_forms(L, prec, kind):
    nx, ny = 61, 43
    h = L.lbmhd_create(nx, ny, L.lbmhd_params_default(precision=prec))
    try:
        L.lbmhd_init(h, *fields(kind, (ny, nx), 5))
        raw, m = L.lbmhd_get_state_raw(h), L.lbmhd_moments(h)
    finally:
        L.lbmhd_destroy(h)
    w = np.array([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4)
    # the FP32 form's arithmetic measures deviations from the FP32 weights
    np.seterr(invalid="ignore")
    d = raw.astype(np.longdouble)
    if prec == "fp32":
        d[:9] -= w.astype(np.float32).astype(np.longdouble)[:, None, None]
    if prec == "fp16_dev":
        d /= 1024
    rho = 1 + d[:9].sum(0)
    jx = d[1] - d[3] + d[5] - d[6] + d[8] - d[7]
    jy = d[2] - d[4] + d[5] + d[6] - d[7] - d[8]
    ref = [rho, jx / rho, jy / rho, d[9::2].sum(0), d[10::2].sum(0)]
    mag = [1 + np.abs(d[:9]).sum(0), np.abs(d[:9]).sum(0) / rho, np.abs(d[:9]).sum(0) / rho,
           np.abs(d[9::2]).sum(0), np.abs(d[10::2]).sum(0)]
    for a, b, s in zip(m, ref, mag):
        fine = np.isfinite(b)  # binary16 overflows on the large fields: not finite there either
        assert np.array_equal(fine, np.isfinite(a))
        fine &= np.isfinite(s)
        assert np.max(np.abs(a - b)[fine] / np.maximum(np.abs(s), 1e-300)[fine]) <= 4 * 2.0 ** -52
