"""Index builds in zones of about an arcsecond, where the zones add hundreds of
bins to those of the rows, and with more units in a bin than a tile of the
second split counts: half of the sources lie near the north pole, in the last
bins. Matches of sources near the catalogue's own equal the oracle's."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _check(g, b_lon, b_lat, h, region):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    pick = g.integers(0, b_lon.size, 3000)
    a_lon = np.mod(b_lon[pick] + g.normal(0, 2e-4, pick.size), 360.0)
    a_lat = np.clip(b_lat[pick] + g.normal(0, 2e-4, pick.size), -90, 90)
    ref = oracle.match(a_lon, a_lat, b_lon, b_lat, a_frame=0, b_frame=0, **region)
    assert ref["border_a"].size == 0
    idx = xm.Index(_cuda(b_lon), _cuda(b_lat), zone_height_arcsec=h)
    res = xm.Result(idx, _cuda(a_lon), _cuda(a_lat), **region)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(res.a_row.cpu().numpy(), ref["a_row"])
    np.testing.assert_array_equal(res.b_row.cpu().numpy(), ref["b_row"])
    assert np.max(np.abs(res.sep.cpu().numpy() - ref["sep"]), initial=0.0) <= 1e-4


@pytest.mark.parametrize("n,h", [(384_000, 1.0), (390_000, 1.2), (3_000_000, 1.0), (3_000_000, 1.1)])
def test_bins_of_fine_zones(n, h):
    g = synth.rng(1400 + n // 1000)
    lon = g.uniform(0, 360, n)
    lat = np.degrees(np.arcsin(g.uniform(-1, 1, n)))
    pole = 90.0 - 0.5 * np.sqrt(g.uniform(0, 1, n))
    _check(g, lon, np.where(np.arange(n) % 2 == 0, lat, pole), h, dict(shape=1, a=2.5, b=1.5, pa=30.0))


def test_more_units_in_a_bin_than_a_tile_counts():
    g = synth.rng(1450)
    n = 1_400_000  # in one zone, whose parts are 1750 units or more
    lat = (4500.5 * 20.0 + g.uniform(-9.0, 9.0, n)) / 3600.0
    _check(g, g.uniform(0, 360, n), lat, 20.0, dict(shape=0, a=0.8))


def test_two_zones_of_one_counter_word():
    """Millions of sources in two zones whose 16-bit counters share a word:
    every block folds both counters."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1460)
    n = 12_000_000
    lon = g.uniform(0, 360, n)
    lat = 16.0 / 3600.0 * g.uniform(2000.02, 2000.98, n)  # zones 2 k and 2 k + 1 of 8 arcsec
    idx = xm.Index(_cuda(lon), _cuda(lat), zone_height_arcsec=8.0)
    pick = g.integers(0, n, 40)
    a_lon, a_lat = lon[pick], lat[pick] + 0.1 / 3600.0
    res = xm.Result(idx, _cuda(a_lon), _cuda(a_lat), a=1.0)
    near = np.unique(np.concatenate([np.nonzero(np.abs(lon - x) < 0.001)[0] for x in a_lon]))
    ref = oracle.match(a_lon, a_lat, lon[near], lat[near], a=1.0)
    assert ref["border_a"].size == 0 and ref["a_row"].size > 40
    np.testing.assert_array_equal(res.a_row.cpu().numpy(), ref["a_row"])
    np.testing.assert_array_equal(res.b_row.cpu().numpy(), near[ref["b_row"]])
