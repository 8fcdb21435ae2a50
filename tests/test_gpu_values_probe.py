"""The Exact Value probe at the edges of what it reads at once: runs of equal
keys from one to far past the words of a bucket it loads together, few and
many A keys around a block's share, keys found first, last and not at all, in
the codes' own order (narrow keys) and under the hash (wide and float64 keys).
Pairs, counts and best rows are those of a sort of B's keys."""

import numpy as np
import pytest

from paper_1611_08494_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_a", [1, 1023, 1025, 5000])
@pytest.mark.parametrize("kind", ["narrow", "wide", "float64", "one_value", "dense_bucket"])
def test_probe_runs(kind, n_a):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1611_08494_gb300 import xm

    g = synth.rng(501)
    if kind == "one_value":
        vals, reps = np.array([7]), np.array([300])
    else:
        vals = np.arange(3000, dtype=np.int64)
        reps = np.concatenate([np.arange(1, 14), np.full(3, 100), [2000]])[g.integers(0, 17, 3000)]
        if kind == "wide":
            vals = vals * 0x9E3779B97F4A7C1 - 2**61
        elif kind == "dense_bucket":  # a few buckets of many different keys
            vals = np.concatenate([vals, 2**31 + vals])
            reps = np.concatenate([np.minimum(reps, 3)] * 2)
    b = np.repeat(vals, reps)
    g.shuffle(b)
    a = np.concatenate([vals, vals + 5000, vals[:1] - 1])[g.integers(0, 2 * vals.size + 1, n_a)]
    if kind == "float64":
        a, b = a * 0.5, b * 0.5
    order = np.argsort(b, kind="stable")
    lo, hi = (np.searchsorted(b[order], a, side=s) for s in ("left", "right"))
    num = hi - lo
    ra = np.repeat(np.arange(n_a), num)
    rb = order[np.repeat(lo - (np.cumsum(num) - num), num) + np.arange(ra.size)]
    res = xm.ValueResult(torch.as_tensor(a, device="cuda"), torch.as_tensor(b, device="cuda"))
    torch.cuda.synchronize()
    np.testing.assert_array_equal(res.count.cpu().numpy(), num)
    np.testing.assert_array_equal(res.a_row.cpu().numpy(), ra)
    np.testing.assert_array_equal(res.b_row.cpu().numpy(), rb)
    first = order[np.minimum(lo, b.size - 1)]
    np.testing.assert_array_equal(res.best_b.cpu().numpy(), np.where(num > 0, first, -1))
