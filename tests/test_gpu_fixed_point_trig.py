"""Float64 separations at the positions where the fixed-point sines and
cosines change branch: quarter and eighth turns, both poles, the equator, tiny
and largest values. Unit vectors are rounded once (2^-54 a component), so each
of a pair's east and north components is within 6 x 2^-53 of exact and the
separation within 9 x 2^-53 rad = 2.1e-10 arcsec; the reference, from the
differences of the positions in degrees, adds as much again at most."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 5e-10  # arcsec


@pytest.mark.parametrize("lat0", [0.0, 1e-9, -1e-7, 45.0, -45.0, 30.0, 89.999, -89.999, 60.125])
def test_float64_separations_at_branch_points(lat0):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = np.random.Generator(np.random.Philox(key=77))
    base = np.concatenate([np.arange(0, 360, 22.5), [1e-12, 359.9999999999, 44.99999999999, 225.0000000001]])
    a_lon = np.repeat(base, 8)
    a_lat = np.full(a_lon.size, lat0)
    step = g.uniform(-4e-4, 4e-4, (2, a_lon.size))
    b_lon = np.mod(a_lon + step[0], 360.0)
    b_lat = np.clip(a_lat + step[1], -90, 90)
    cu = lambda x: torch.as_tensor(x, device="cuda")  # noqa: E731
    got = []
    for stored in (True, False):
        idx = xm.Index(cu(b_lon), cu(b_lat), build_fp64=stored)
        res = xm.Result(idx, cu(a_lon), cu(a_lat), precision=xm.PREC_FP64, shape=0, a=5.0)
        torch.cuda.synchronize()
        got.append([t.cpu().numpy() for t in (res.a_row, res.b_row, res.sep)])
    for x, y in zip(*got):  # unit vectors stored or computed: the same bits
        np.testing.assert_array_equal(x, y)
    a, b, sep = got[0]
    assert a.size >= a_lon.size  # every planted pair lies within 5 arcsec
    dl = np.radians(np.mod(b_lon[b] - a_lon[a] + 180.0, 360.0) - 180.0)
    db, la, lb = np.radians(b_lat[b] - a_lat[a]), np.radians(a_lat[a]), np.radians(b_lat[b])
    h = np.sin(dl / 2)
    x = np.cos(lb) * np.sin(dl)
    y = np.sin(db) + 2 * np.cos(lb) * np.sin(la) * h * h
    z = np.cos(db) - 2 * np.cos(lb) * np.cos(la) * h * h
    exact = np.degrees(np.arctan2(np.hypot(x, y), z)) * 3600
    assert np.max(np.abs(sep - exact)) <= TOL
