"""The join's passes over the A sources (tiles of 1024) and over the bitset of
matched B rows (tiles of 8192), at their edges: every join type over both
selections, with none, some and all of the sources matched, sources of many
members, and as many A sources as take the form of large catalogues (the
unmatched before a tile known from the match). A catalogue of well separated points is matched by copies of its own positions,
so each pair is known without a search and every row must be the expected one;
the separations must be those of the match itself."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu

# name: (A sources, B sources, matched fraction, copies of a B position: on
# average, or, below zero, sources added at the first 20 positions only)
CASES = {
    "one": (1, 1, 1.0, 1),
    "none_matched": (1024, 8192, 0.0, 1),
    "below": (1023, 8191, 0.5, 1),
    "at": (1024, 8192, 1.0, 1),
    "above": (1025, 8193, 0.5, 5),
    "tiles": (40_961, 20_011, 0.3, 3),
    "dense": (3000, 65_537, 0.7, 40),
    "chained": (262_143, 30_031, 0.4, 3),
    "sums": (262_144, 30_031, 0.4, 3),
    "sums_empty": (270_337, 8_192, 0.0, 1),
    "sums_dense": (299_000, 500, 0.9, 5),
    "skewed": (40_000, 3_000, 0.5, -1_000),
    "sums_skewed": (300_000, 21_000, 0.5, -1_000),
    "large": (4_300_001, 300_031, 0.4, 3),
}


@pytest.mark.parametrize("name", list(CASES))
def test_join_rows(name):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    n_a, n_b, frac, copies = CASES[name]
    g = synth.rng(77)
    # points 0.02 degrees apart at the equator's sides, B rows in random order,
    n_pts = max(n_b // copies, 1) if copies > 0 else n_b + copies
    cols = 17_000
    pts = np.arange(n_pts)
    p_lon, p_lat = 0.02 * (pts % cols) + 1.0, 0.02 * (pts // cols) - 10.0
    b_pt = np.concatenate([pts, g.integers(0, n_pts if copies > 0 else 20, n_b - n_pts)])
    g.shuffle(b_pt)
    a_pt = g.integers(0, n_pts, n_a)
    matched = g.uniform(0, 1, n_a) < frac
    a_lon, a_lat = p_lon[a_pt], np.where(matched, p_lat[a_pt], p_lat[a_pt] + 0.01)
    dev = lambda x: torch.as_tensor(np.ascontiguousarray(x), device="cuda")  # noqa: E731
    idx = xm.Index(dev(p_lon[b_pt]), dev(p_lat[b_pt]), zone_height_arcsec=8.0)
    res = xm.Result(idx, dev(a_lon), dev(a_lat), shape=xm.CIRCLE, a=1.0)

    by_pt = np.argsort(b_pt, kind="stable")
    start = np.searchsorted(b_pt[by_pt], np.arange(n_pts + 1))
    num = np.where(matched, (start[1:] - start[:-1])[a_pt], 0)
    ra = np.repeat(np.arange(n_a), num)
    k = np.arange(ra.size) - np.repeat(np.cumsum(num) - num, num)
    rb = by_pt[start[a_pt[ra]] + k]
    host = lambda t: t.cpu().numpy()  # noqa: E731
    np.testing.assert_array_equal(host(res.a_row), ra)
    np.testing.assert_array_equal(host(res.b_row), rb)
    sep = host(res.sep)
    has = num > 0
    bb = host(res.best_b)
    np.testing.assert_array_equal(bb >= 0, has)
    np.testing.assert_array_equal(b_pt[bb[has]], a_pt[has])
    sels = {xm.SEL_ALL: dict(a_row=ra, b_row=rb, sep=sep),
            xm.SEL_BEST: dict(a_row=np.nonzero(has)[0], b_row=bb[has],
                              sep=host(res.best_sep)[has])}
    for code, sel in sels.items():
        for jt in oracle.JOINS:
            rows = res.join(jt, code)
            exp = oracle.join(sel, n_a, n_b, jt)
            msg = f"{jt} selection {code}"
            np.testing.assert_array_equal(host(rows.a_row), exp["a_row"], err_msg=msg)
            np.testing.assert_array_equal(host(rows.b_row), exp["b_row"], err_msg=msg)
            np.testing.assert_array_equal(host(rows.sep), exp["sep"], err_msg=msg)
