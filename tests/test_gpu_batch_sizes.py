"""Batches of regions below, at and above the size that the sparse count pass
takes (half a zone, three quarters in float64), in totals about the 32 sources of its chunks and the 256 of
a preparation block: none, all, and some of a chunk too large. Rows, counts and
best pairs equal those of each request matched alone."""

import numpy as np
import pytest

from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu
ZONE_H = 12.0


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("kind", ["large", "edge", "mixed", "some"])
@pytest.mark.parametrize("sizes", [(1,), (31, 1), (33, 222, 1), (256, 257), (5, 1000, 3, 64)])
def test_batch_of_sizes(prec, order, kind, sizes):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1800 + len(sizes))
    lon, lat = g.uniform(20.0, 21.0, 40_000), g.uniform(-0.5, 0.5, 40_000)
    idx = xm.Index(_cuda(lon), _cuda(lat), zone_height_arcsec=ZONE_H, build_fp64=prec == xm.PREC_FP64)
    reqs = []
    for k, n in enumerate(sizes):
        pick = g.integers(0, lon.size, n)
        a = {"large": g.uniform(20.0, 40.0, n), "edge": np.full(n, (0.5 if prec == xm.PREC_FP32 else 0.75) * ZONE_H)
             * (1.0 - 1e-6 + 1e-6 * (np.arange(n) % 3 - 1)),
             "mixed": 0.3 * 200.0 ** g.uniform(0, 1, n),
             "some": np.where(np.arange(n) % 47 == 3, 30.0, 1.5)}[kind]
        reqs.append(dict(lon=_cuda(lon[pick] + g.normal(0, 5e-4, n)), shape=k % 3,
                         lat=_cuda(lat[pick] + g.normal(0, 5e-4, n)), a_col=_cuda(a),
                         b_col=_cuda(a * 0.7), pa_col=_cuda(g.uniform(0, 180, n))))
    batch = xm.Batch(idx, reqs, precision=prec, a_order=order)
    tol = 1e-4 if prec == xm.PREC_FP32 else 1e-9
    for r, q in enumerate(reqs):
        v, q = batch.view(r), dict(q)
        ref = xm.Result(idx, q.pop("lon"), q.pop("lat"), precision=prec, a_order=xm.A_ORDER_SORTED, **q)
        torch.cuda.synchronize()
        for f in ("a_row", "b_row", "count", "best_b"):
            np.testing.assert_array_equal(v[f].cpu().numpy(), getattr(ref, f).cpu().numpy(), err_msg=f)
        for f in ("sep", "best_sep"):
            np.testing.assert_allclose(v[f].cpu().numpy(), getattr(ref, f).cpu().numpy(), rtol=0, atol=tol)


def test_large_batch():
    """As many sources as take several rounds a thread in the preparation."""
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1850)
    lon, lat = g.uniform(0.0, 360.0, 300_000), g.uniform(-60.0, 60.0, 300_000)
    idx = xm.Index(_cuda(lon), _cuda(lat), zone_height_arcsec=ZONE_H)
    reqs = []
    for k, n in enumerate((1_500_001, 2_000_000, 700_077)):
        pick = g.integers(0, lon.size, n)
        q = dict(lon=_cuda(lon[pick]), lat=_cuda(np.clip(lat[pick] + g.normal(0, 5e-4, n), -90, 90)))
        a = 0.5 * 100.0 ** g.uniform(0, 1, n)
        q.update((dict(a=30.0), dict(a_col=_cuda(a)), dict(a=2.0))[k])
        reqs.append(q)
    batch = xm.Batch(idx, reqs)
    for r, q in enumerate(reqs):
        v, q = batch.view(r), dict(q)
        ref = xm.Result(idx, q.pop("lon"), q.pop("lat"), **q)
        for f in ("a_row", "b_row", "count", "best_b"):
            assert torch.equal(v[f], getattr(ref, f)), f
