"""The index build (a partition into zones, parts of zones and units) on the
catalogues where its cases meet: nothing but empty zones, one split and two,
zones of many sources cut into parts, zones too large for one block, sources
on the seam, at the poles, all on one point, and stored by position. The
matches of sources near the catalogue's own must equal the oracle's, and
sources that match nothing must match nothing."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _sky(g, n):
    return g.uniform(0, 360, n), np.degrees(np.arcsin(g.uniform(-1, 1, n)))


def _catalogue(g, name):
    if name.startswith("sky"):
        n, h = (int(v) for v in name.split("_")[1:])
        return (*_sky(g, n), float(h))
    if name == "stripe":  # a few zones of 30,000 sources each: parts
        return g.uniform(0, 360, 450_000), g.uniform(-0.04, 0.04, 450_000), 20.0
    if name == "seam":  # the same across longitude 0: most parts are empty
        return np.mod(g.uniform(-1, 1, 450_000), 360.0), g.uniform(-0.04, 0.04, 450_000), 20.0
    if name == "one_split":  # zones of thousands of sources, one split
        return g.uniform(10, 40, 60_000), g.uniform(5.0, 5.05, 60_000), 20.0
    if name == "poles":
        lat = 90.0 - np.abs(g.normal(0, 0.05, 430_000))
        return g.uniform(0, 360, 430_000), np.where(g.uniform(0, 1, 430_000) < 0.5, lat, -lat), 12.0
    if name == "by_position":
        lon, lat = _sky(g, 420_000)
        o = np.lexsort((lon, np.floor(lat * 180)))
        return lon[o], lat[o], 20.0
    if name == "point":  # all in one bucket
        return np.full(420_000, 200.25), np.full(420_000, 12.125), 20.0
    raise ValueError(name)


@pytest.mark.parametrize("name", [
    "sky_1_20", "sky_2_20", "sky_1023_20", "sky_65537_36000", "sky_393000_20", "sky_396001_20",
    "sky_430001_1", "sky_430001_36000", "sky_400003_8", "one_split", "stripe", "seam", "poles",
    "by_position", "point"])
def test_index_of_any_distribution(name):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1200 + len(name))
    b_lon, b_lat, h = _catalogue(g, name)
    n = b_lon.size
    pick = g.integers(0, n, 2000) if name != "point" else np.zeros(3, np.int64)
    a_lon = np.concatenate([np.mod(b_lon[pick] + g.normal(0, 2e-4, pick.size), 360.0), _sky(g, 500)[0]])
    a_lat = np.concatenate([np.clip(b_lat[pick] + g.normal(0, 2e-4, pick.size), -90, 90),
                            _sky(g, 500)[1]])
    region = dict(shape=1, a=2.5, b=1.5, pa=30.0)
    ref = oracle.match(a_lon, a_lat, b_lon, b_lat, a_frame=0, b_frame=0, **region)
    assert ref["border_a"].size == 0
    for prec, fp64 in ((xm.PREC_FP32, False), (xm.PREC_FP64, True)):
        idx = xm.Index(_cuda(b_lon), _cuda(b_lat), zone_height_arcsec=h, build_fp64=fp64)
        res = xm.Result(idx, _cuda(a_lon), _cuda(a_lat), precision=prec, **region)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(res.a_row.cpu().numpy(), ref["a_row"])
        np.testing.assert_array_equal(res.b_row.cpu().numpy(), ref["b_row"])
        assert np.max(np.abs(res.sep.cpu().numpy() - ref["sep"]), initial=0.0) <= 1e-4


def test_invalid_positions_fail_the_build():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1300)
    for n in (5_000, 420_000):  # one split, two
        lon, lat = _sky(g, n)
        for col, bad in ((0, np.nan), (0, np.inf), (1, 90.5), (1, np.nan)):
            cols = [lon.copy(), lat.copy()]
            cols[col][n // 3] = bad
            with pytest.raises(xm.XMError, match="XM_EINVAL"):
                xm.Index(_cuda(cols[0]), _cuda(cols[1]))
            idx = xm.Index(_cuda(cols[0]), _cuda(cols[1]), deferred_check=True)
            with pytest.raises(xm.XMError, match="XM_EINVAL"):
                xm.Result(idx, _cuda(lon[:100]), _cuda(lat[:100]), shape=0, a=1.0)
