"""Index builds of catalogues with many sources on one spot, in a small field
or in one zone: units of more rows than a block places, units whose rows alone
skip more ids than a tile counts, zones of thousands of parts. Sources matched
on the spot find every row of it, and matches elsewhere equal the oracle's."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu

SPOT = (123.4567, -0.0123)
# name: (sources elsewhere, on the spot, longitudes, latitudes, zone height)
CASES = {
    "one_split_below": (60_000, 16_384, (0, 360), (-90, 90), 20.0),
    "one_split_above": (60_000, 16_385, (0, 360), (-90, 90), 20.0),
    "half": (500_000, 500_000, (0, 360), (-90, 90), 20.0),
    "half_in_its_zone": (200_000, 260_000, (0, 360), (-0.0130, -0.0115), 20.0),
    "most": (20_000, 1_500_000, (0, 360), (-90, 90), 20.0),
    "small_field": (600_000, 20_000, (123.45, 123.466), (-0.02, -0.004), 20.0),
    "wide_zones": (300_000, 500, (0, 360), (-90, 90), 36000.0),
    "wide_zones_two_splits": (2_500_000, 20_000, (0, 360), (-60, 60), 36000.0),
    "many_ids": (800_000, 3_300_000, (0, 360), (-0.0130, -0.0115), 20.0),
}


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("name", list(CASES))
def test_many_sources_on_a_spot(name):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    n, spot, lon_range, lat_range, h = CASES[name]
    g = synth.rng(1700 + len(name))
    lon = g.uniform(*lon_range, n)
    lat = (np.degrees(np.arcsin(g.uniform(-1, 1, n))) if lat_range == (-90, 90)
           else g.uniform(*lat_range, n))
    near = np.hypot((lon - SPOT[0]), lat - SPOT[1]) < 3.0 / 3600.0  # leave the spot alone
    lon[near] += 0.004
    b_lon, b_lat = np.append(lon, np.full(spot, SPOT[0])), np.append(lat, np.full(spot, SPOT[1]))
    order = g.permutation(n + spot)
    b_lon, b_lat = b_lon[order], b_lat[order]
    on_spot = np.nonzero(order >= n)[0]
    idx = xm.Index(_cuda(b_lon), _cuda(b_lat), zone_height_arcsec=h)

    res = xm.Result(idx, _cuda(np.full(2, SPOT[0])), _cuda(np.full(2, SPOT[1])), a=0.5)
    np.testing.assert_array_equal(res.b_row.cpu().numpy(), np.tile(on_spot, 2))
    np.testing.assert_array_equal(res.count.cpu().numpy(), [spot, spot])

    a = 0.3
    pick = g.integers(0, n, 2000)
    a_lon, a_lat = np.mod(lon[pick] + g.normal(0, 2e-5, 2000), 360.0), lat[pick] + g.normal(0, 2e-5, 2000)
    a_lat = np.clip(a_lat, -90, 90)
    keep = order < n  # (the oracle's catalogue: the rest, in its rows' order)
    rows = np.nonzero(keep)[0]
    ref = oracle.match(a_lon, a_lat, b_lon[keep], b_lat[keep], a=a)
    assert ref["border_a"].size == 0
    res = xm.Result(idx, _cuda(a_lon), _cuda(a_lat), a=a)
    np.testing.assert_array_equal(res.a_row.cpu().numpy(), ref["a_row"])
    np.testing.assert_array_equal(res.b_row.cpu().numpy(), rows[ref["b_row"]])
