"""Joins of a result whose sources have a pair or none but for a few with
hundreds to tens of thousands: the A-side pass lists those (by warps of 32
sources, in chunks of 1024 pairs) for a pass of their own. Counts about the
limits, in the first and last source, alone in a warp and beside each other,
over every join type with pairs; for a positional match, a match of values and
a request of a batch."""

import numpy as np
import pytest

import oracle
from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu

# name: (A sources, {source: members})
CASES = {
    "limit": (4_000, {0: 512, 40: 513, 64: 16, 96: 17, 3_999: 496}),
    "pair": (4_000, {64: 300, 70: 212, 128: 300, 159: 213}),
    "chunks": (20_000, {0: 1024, 33: 1025, 100: 2048, 9_000: 20_000, 19_999: 2049}),
    "warp": (9_000, {320 + k: 700 for k in range(32)}),
    "sums": (270_000, {5: 3_000, 262_150: 40_000, 269_999: 700}),
}


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


def _check_joins(xm, res, n_a, n_b, ra, rb, long_pass=True):
    host = lambda t: t.cpu().numpy()  # noqa: E731
    np.testing.assert_array_equal(host(res.a_row), ra)
    np.testing.assert_array_equal(host(res.b_row), rb)
    sel = dict(a_row=ra, b_row=rb, sep=host(res.sep))
    for jt in ("and", "or", "all1", "all2"):
        xm.prof_enable(True)
        try:
            rows = res.join(jt, xm.SEL_ALL)
            ran = "k_join_long" in xm.prof_all()
        finally:
            xm.prof_enable(False)
        assert ran == long_pass
        exp = oracle.join(sel, n_a, n_b, jt)
        for f in ("a_row", "b_row", "sep"):
            np.testing.assert_array_equal(host(getattr(rows, f)), exp[f], err_msg=f"{jt} {f}")


def _pairs(name):
    """Points of the catalogue: `num` copies of each source's own, in random
    B order; a fifth of the other sources unmatched."""
    n_a, many = CASES[name]
    g = synth.rng(1600 + n_a)
    num = (g.uniform(0, 1, n_a) < 0.8).astype(np.int64)
    for k, m in many.items():
        num[k] = m
    b_pt = np.repeat(np.arange(n_a), num)
    g.shuffle(b_pt)
    rb = np.argsort(b_pt, kind="stable")
    return n_a, num, b_pt, np.repeat(np.arange(n_a), num), rb


@pytest.fixture(scope="module")
def xm():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm as mod

    return mod


@pytest.mark.parametrize("name", list(CASES))
def test_positional(xm, name):
    n_a, num, b_pt, ra, rb = _pairs(name)
    lon, lat = 0.02 * (np.arange(n_a) % 17_000) + 1.0, 0.02 * (np.arange(n_a) // 17_000) - 0.2
    idx = xm.Index(_cuda(lon[b_pt]), _cuda(lat[b_pt]))
    _check_joins(xm, xm.Result(idx, _cuda(lon), _cuda(lat), a=1.0), n_a, b_pt.size, ra, rb)


@pytest.mark.parametrize("name", ["chunks", "sums"])
def test_values(xm, name):
    n_a, num, b_pt, ra, rb = _pairs(name)
    key = synth.rng(5).integers(-2**62, 2**62, n_a)
    _check_joins(xm, xm.ValueResult(_cuda(key), _cuda(key[b_pt])), n_a, b_pt.size, ra, rb)


def test_few_members_need_no_list(xm):
    n_a = 5_000
    num = np.where(np.arange(n_a) % 5 == 0, 16, 0)
    b_pt = np.repeat(np.arange(n_a), num)
    lon = 0.02 * np.arange(n_a) + 1.0
    idx = xm.Index(_cuda(lon[b_pt]), _cuda(np.zeros(b_pt.size)))
    res = xm.Result(idx, _cuda(lon), _cuda(np.zeros(n_a)), a=1.0)
    assert 512 < res.n_pairs <= 4 * n_a
    _check_joins(xm, res, n_a, b_pt.size, np.repeat(np.arange(n_a), num), np.arange(b_pt.size), False)


def test_a_request_of_a_batch(xm):
    n_a, num, b_pt, ra, rb = _pairs("chunks")
    lon, lat = 0.02 * (np.arange(n_a) % 17_000) + 1.0, 0.02 * (np.arange(n_a) // 17_000) - 0.2
    idx = xm.Index(_cuda(lon[b_pt]), _cuda(lat[b_pt]))
    other = dict(lon=_cuda(lon[:999] + 0.01), lat=_cuda(lat[:999]), a=1.0)
    batch = xm.Batch(idx, [other, dict(lon=_cuda(lon), lat=_cuda(lat), a=1.0, join="or",
                                       join_selection=xm.SEL_ALL)])
    xm.prof_enable(True)
    try:
        rows = batch.join(1)
        assert "k_join_long" in xm.prof_all()
    finally:
        xm.prof_enable(False)
    sep = batch.view(1)["sep"].cpu().numpy()
    exp = oracle.join(dict(a_row=ra, b_row=rb, sep=sep), n_a, b_pt.size, "or")
    for f in ("a_row", "b_row", "sep"):
        np.testing.assert_array_equal(getattr(rows, f).cpu().numpy(), exp[f], err_msg=f)
