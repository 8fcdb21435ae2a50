"""Best pairs per B source where two A sources of another frame lie at separations
that differ in their last bits: the pick decides by the float64 separations that
the match reports, ties to the lowest A row."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("frame", [0, 1])
def test_pick_agrees_with_reported_separations(frame):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(2000)
    n = 60_000
    lon = 0.02 * (np.arange(n) % 16_000) + 20.0
    lat = 0.02 * (np.arange(n) // 16_000) + 40.0 + g.uniform(0, 1e-3, n)
    d = 0.5 / 3600.0
    # A on both sides of each B along its parallel
    a_lon = np.concatenate([lon + d, lon - d])
    a_lat = np.concatenate([lat, lat])
    if frame:
        a_lon, a_lat = oracle.from_equatorial(a_lon, a_lat, oracle.GAL)
    order = g.permutation(2 * n)
    idx = xm.Index(_cuda(lon), _cuda(lat), build_fp64=True)
    res = xm.Result(idx, _cuda(a_lon[order]), _cuda(a_lat[order]), frame=frame, precision=xm.PREC_FP64,
                    a=1.0)
    a_row, b_row, sep = (t.cpu().numpy() for t in (res.a_row, res.b_row, res.sep))
    assert a_row.size == 2 * n and np.array_equal(np.sort(b_row), np.repeat(np.arange(n), 2))
    o = np.lexsort((a_row, sep, b_row))
    best = a_row[o][::2]
    gap = np.diff(sep[o].reshape(n, 2), axis=1)[:, 0]
    assert np.sum((gap > 0) & (gap < 2e-11)) > 1000  # arcsec
    rows = res.pick("best_b")
    got_a, got_b = rows.a_row.cpu().numpy(), rows.b_row.cpu().numpy()
    want = np.empty(n, np.int64)
    want[got_b] = got_a
    np.testing.assert_array_equal(want, best)
