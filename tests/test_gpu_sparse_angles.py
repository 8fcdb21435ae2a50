"""Regions of one size with a position angle for each source, small against the
zone height (the sparse count pass in input order): members, counts, best pairs
and joins equal the oracle's and those of the sorted order, the levels of the
result the oracle's, and an angle that is not finite fails the call whatever
the shape."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu
SEP_TOL = 1e-4  # arcsec
DIST_TOL = 1e-9


@pytest.fixture(scope="module")
def xm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm as mod

    return mod


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _host(t):
    import torch

    torch.cuda.synchronize()
    return t.cpu().numpy()


def _catalogues(n, frame):
    """Sources apart from each other, four of B around each."""
    g = synth.rng(1500)
    lon, lat = g.uniform(0.0, 360.0, n), np.degrees(np.arcsin(g.uniform(-0.95, 0.95, n)))
    k = np.repeat(np.arange(n), 4)
    d = g.normal(0.0, 2.0 / 3600.0, (2, k.size))
    b_lat = lat[k] + d[1]
    b_lon = np.mod(lon[k] + d[0] / np.cos(np.radians(b_lat)), 360.0)
    if frame:
        lon, lat = oracle.from_equatorial(lon, lat, oracle.GAL)
    return lon, lat, b_lon, b_lat, g.uniform(-200.0, 400.0, n)


@pytest.mark.parametrize("shape", [1, 2])
@pytest.mark.parametrize("frame", [0, 1])
@pytest.mark.parametrize("prec", [0, 1])
def test_angles_by_source(xm, shape, frame, prec):
    n = 3001
    lon, lat, b_lon, b_lat, pa = _catalogues(n, frame)
    reg = dict(shape=shape, a=4.0, b=1.0, pa_zero_deg=12.5, pa_dir=-1)
    ref = oracle.match(lon, lat, b_lon, b_lat, a_frame=frame, b_frame=0, pa_col=pa, **reg)
    best = oracle.best(ref, n)
    assert ref["a_row"].size > n and ref["border_a"].size == 0 and best["near_tie"].size == 0
    idx = xm.Index(_cuda(b_lon), _cuda(b_lat), zone_height_arcsec=20.0, build_fp64=prec == xm.PREC_FP64)
    name = "k_scan_src" if prec == xm.PREC_FP32 else "k_scan_src_fp64"
    for order in (xm.A_ORDER_INPUT, xm.A_ORDER_SORTED):
        xm.prof_enable(True)
        try:
            # (a fixed angle beside the column is not used)
            res = xm.Result(idx, _cuda(lon), _cuda(lat), frame=frame, precision=prec, a_order=order,
                            pa=float("nan"), pa_col=_cuda(pa), **reg)
            prof = xm.prof_all()
        finally:
            xm.prof_enable(False)
        assert (name in prof) == (order == xm.A_ORDER_INPUT)
        np.testing.assert_array_equal(_host(res.a_row), ref["a_row"])
        np.testing.assert_array_equal(_host(res.b_row), ref["b_row"])
        np.testing.assert_allclose(_host(res.sep), ref["sep"], rtol=0, atol=SEP_TOL)
        np.testing.assert_array_equal(_host(res.best_b), best["best_b"])
        rows, want = res.join("or"), oracle.join(ref, n, b_lon.size, "or")
        np.testing.assert_array_equal(_host(rows.a_row), want["a_row"])
        np.testing.assert_array_equal(_host(rows.b_row), want["b_row"])
        scales = [0.25, 0.5, 0.9]
        con = oracle.concentric(ref, n, scales)
        assert con["border"].size == 0
        lv = res.levels(scales)
        np.testing.assert_allclose(_host(lv.dist), ref["dist"], rtol=0, atol=DIST_TOL)
        np.testing.assert_array_equal(_host(lv.level), con["level"])


@pytest.mark.parametrize("shape", [0, 1, 2])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_bad_angle_fails_the_call(xm, shape, prec, bad):
    lon, lat, b_lon, b_lat, pa = _catalogues(500, 0)
    idx = xm.Index(_cuda(b_lon), _cuda(b_lat), build_fp64=prec == xm.PREC_FP64)
    pa[321] = bad
    for order in (xm.A_ORDER_INPUT, xm.A_ORDER_SORTED):
        with pytest.raises(xm.XMError, match="XM_EINVAL"):
            xm.Result(idx, _cuda(lon), _cuda(lat), shape=shape, a=4.0, b=1.0, pa_col=_cuda(pa),
                      precision=prec, a_order=order)
