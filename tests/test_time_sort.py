"""The time order of kernel records out of order (GPU): the bucketed sort, its
limits, and the radix sort it leaves crowded times to, against numpy's stable
sort by (start, stream, index)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _times(case, n, rng):
    if case == "spread":
        return rng.integers(0, 1 << 33, n)
    if case == "equal":                       # bins of many equal times, ties by stream and index
        return rng.integers(0, max(n // 200, 1), n) * 1_000_003
    if case == "crowded":                     # almost all in one bucket, one far away
        t = rng.integers(0, 50_000, n)
        t[0] = 1 << 40
        return t
    if case == "long":                        # a span whose key needs more buckets than there may be
        return rng.integers(0, 1 << 52, n)
    assert case == "near"                     # nearly in order
    return np.arange(n) * 900 - rng.integers(0, 4000, n)


@pytest.mark.parametrize("case", ["spread", "equal", "crowded", "long", "near"])
@pytest.mark.parametrize("n", [2, 3073, 8193, 300_007])
def test_time_order(case, n):
    import torch

    import paper_2609_11938_gb300 as opa
    rng = np.random.default_rng(n)
    t = _times(case, n, rng).astype(np.int64) - 5_000_000
    t[:2] = t[:2][::-1].copy() if t[0] < t[1] else t[:2]
    s = rng.choice([0, 3, 255], n).astype(np.uint8)
    order = np.lexsort((np.arange(n), s, t))
    name = rng.integers(0, 50, n).astype(np.int32)
    d = lambda a: torch.from_numpy(a).cuda()
    # as many rows as launches, in launch order: row j belongs to the j-th launch
    tr = opa.DeviceTrace(d(s), d(t), d(np.ones(n, np.int64)), d(name), None, d(s[:0]), d(t[:0]), d(t[:0]), d(s[:0]),
                         d(name[:0]), 0, d(name[order]), torch.zeros((n, 20), device="cuda"))
    with opa.Context(0) as ctx:
        st, idx, kind, summ = ctx.match(tr)
    want = np.empty(n, np.int32)
    want[order] = np.arange(n)
    assert st == opa.OK and summ["fast_path"] == 1
    np.testing.assert_array_equal(idx.cpu().numpy(), want)
