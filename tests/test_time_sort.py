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
    if case in ("most buckets", "too many"):  # 4,096 buckets for few records, and one more
        t = rng.integers(0, 4096 << 24, n)
        t[0], t[-1] = (4096 << 24) - (case == "most buckets"), 0
        return t
    if case == "long":                        # a span whose key needs more buckets than there may be
        return rng.integers(0, 1 << 52, n)
    assert case == "near"                     # nearly in order
    return np.arange(n) * 900 - rng.integers(0, 4000, n)


@pytest.mark.parametrize("case", ["spread", "equal", "crowded", "most buckets", "too many", "long", "near"])
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


def _far_times(case, n, rng):
    """Spans whose (time, stream) key is wider than 64 bits."""
    if case == "wraps":                       # 2^56 and a little: the key of the largest is a small number
        t = rng.integers(0, 1 << 56, n)
        t[-1], t[0] = 0, (1 << 56) + 3
        return t
    if case == "2^60":
        return rng.integers(0, 1 << 60, n)
    t = rng.integers(-(1 << 63), (1 << 63) - 1, n)
    t[-1], t[0] = -(1 << 63), (1 << 63) - 1
    return t


@pytest.mark.parametrize("case", ["wraps", "2^60", "all"])
@pytest.mark.parametrize("n", [2, 3073, 300_007])
def test_time_order_of_far_times(case, n):
    import torch

    import paper_2609_11938_gb300 as opa
    rng = np.random.default_rng(n)
    t = _far_times(case, n, rng).astype(np.int64)
    t[n // 3 + 1:n // 2 + 1] = t[n // 2]      # and ties, by stream and index
    s = rng.choice([0, 3, 255], n).astype(np.uint8)
    order = np.lexsort((np.arange(n), s, t))
    name = rng.integers(0, 50, n).astype(np.int32)
    d = lambda a: torch.from_numpy(a).cuda()
    tr = opa.DeviceTrace(d(s), d(t), d(np.ones(n, np.int64)), d(name), None, d(s[:0]), d(t[:0]), d(t[:0]), d(s[:0]),
                         d(name[:0]), 0, d(name[order]), torch.zeros((n, 20), device="cuda"))
    with opa.Context(0) as ctx:
        st, idx, kind, summ = ctx.match(tr)
    want = np.empty(n, np.int32)
    want[order] = np.arange(n)
    assert st == opa.OK and summ["fast_path"] == 1
    np.testing.assert_array_equal(idx.cpu().numpy(), want)


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("far", [1 << 57, (1 << 58) - 1, (1 << 58) + 12345, 1 << 60, 1 << 62])
def test_far_ranges(far, shuffle):
    """Ranges out of start order with one that begins long before the others,
    at times around what six more bits leave room for, and one that never ends."""
    import dataclasses

    import oracle
    import tracegen
    from gpu_util import assert_parity, gpu_run
    t = tracegen.generate("adversarial", n_kernels=20_000, n_streams=3, max_depth=6, seed=far % 97, shuffle=shuffle)
    first = min(int(t.k_start.min()), int(t.r_start.min()))
    last = max(int(t.k_start.max()), int(t.r_end.max()))
    stream = int(t.r_stream[0])
    i = int(np.nonzero(t.k_stream == stream)[0][-1])
    start = t.k_start.copy()
    start[i] = first - (1 << 54)              # a kernel inside the early range
    add = lambda a, *v: np.concatenate([a, np.array(v, a.dtype)])
    t = dataclasses.replace(t, k_start=start, r_start=add(t.r_start, last + 9, first - far),
                            r_end=add(t.r_end, (1 << 63) - 1, first - 5), r_stream=add(t.r_stream, stream, stream),
                            r_depth=add(t.r_depth, 0, 0), r_op=add(t.r_op, 0, 1))
    o = oracle.run(t, enclose_mode="indexed")
    assert o["range_of_kernel"][i] == t.R - 1
    assert_parity(gpu_run(t), o)
