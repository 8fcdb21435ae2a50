"""Views of a batch of many requests, some without pairs, best pairs or a join:
each equals its request matched alone, and one view asks for a few requests'
arrays, not for all of them."""

import numpy as np
import pytest

from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu


def _cuda(x):
    import torch

    return torch.as_tensor(np.ascontiguousarray(x), device="cuda")


@pytest.mark.parametrize("first", ["all", "best"])
def test_one_view_of_many(monkeypatch, first):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1900)
    lon, lat = g.uniform(20.0, 21.0, 20_000), g.uniform(-0.5, 0.5, 20_000)
    idx = xm.Index(_cuda(lon), _cuda(lat))
    reqs = []
    for k in range(300):
        n = k % 5  # (also requests without a source)
        sel = (xm.SEL_ALL, xm.SEL_BEST, xm.SEL_ALL | xm.SEL_BEST)[(k + (first == "best")) % 3]
        pick = g.integers(0, lon.size, n)
        q = dict(lon=_cuda(lon[pick]), lat=_cuda(lat[pick]), a=10.0, selection=sel)
        if k % 4 == 1:
            q.update(join="all1", join_selection=xm.SEL_ALL if sel & xm.SEL_ALL else xm.SEL_BEST)
        reqs.append(q)
    batch = xm.Batch(idx, reqs)
    calls = []
    real = xm.xm_batch_get
    monkeypatch.setattr(xm, "xm_batch_get", lambda *a: calls.append(a[1]) or real(*a))
    batch.view(150)
    assert len(calls) <= 10
    monkeypatch.undo()
    for r, q in enumerate(reqs):
        v, q = batch.view(r), dict(q)
        join, js = q.pop("join", None), q.pop("join_selection", None)
        sel = q["selection"]
        ref = xm.Result(idx, q.pop("lon"), q.pop("lat"), **q)
        rows = ref.join(join, js) if join else None
        torch.cuda.synchronize()
        want = dict(count=ref.count)
        for f in ("a_row", "b_row", "sep"):
            want[f] = getattr(ref, f) if sel & xm.SEL_ALL else None
            want[f.replace("sep", "row_sep") if f == "sep" else "row_" + f[0]] = getattr(rows, f) if rows else None
        for f in ("best_b", "best_sep"):
            want[f] = getattr(ref, f) if sel & xm.SEL_BEST else None
        for f, t in want.items():
            exp = np.empty(0) if t is None else t.cpu().numpy()
            np.testing.assert_array_equal(v[f].cpu().numpy(), exp, err_msg=f"{r} {f}")
    for bad in (-1, 300):
        with pytest.raises(xm.XMError):
            batch.view(bad)


def test_profiling_a_graph_batch_fails_no_later_call():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(1910)
    lon, lat = _cuda(g.uniform(20.0, 21.0, 5_000)), _cuda(g.uniform(-0.5, 0.5, 5_000))
    idx = xm.Index(lon, lat)
    xm.prof_enable(True)
    try:
        batch = xm.Batch(idx, [dict(lon=lon[:500], lat=lat[:500], a=5.0)], use_graph=True)
        prof = xm.prof_all()
    finally:
        xm.prof_enable(False)
    assert "batch_graph" in prof
    res = xm.Result(xm.Index(lon, lat), lon[:500], lat[:500], a=5.0)  # (the build's first launch failed)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(batch.view(0)["b_row"].cpu().numpy(), res.b_row.cpu().numpy())
