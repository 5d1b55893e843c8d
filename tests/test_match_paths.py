"""The matching's paths (GPU) where they can go wrong: name runs over tile edges
of the run scan, layer counts on both sides of the counting pass, fast pairings
that fail inside a join.  Against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
import tracegen
from gpu_util import assert_parity, gpu_run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["skip_name", "prefix"])
@pytest.mark.parametrize("k,m,names", [(1, 0, 1), (0, 5, 2), (1, 1, 3), (4095, 1, 1), (4096, 4096, 2), (4097, 4095, 300),
                                       (9000, 7000, 257), (60_000, 66_000, 70_000)])
def test_ordinals_over_tiles(k, m, names, mode):
    rng = np.random.default_rng(k + m + names)
    t = tracegen.small_random(3, shuffle=False)
    counters = rng.uniform(0, 9, (m, 20)).astype(np.float32)
    t = dataclasses.replace(t, k_stream=np.zeros(k, np.uint8), k_start=np.sort(rng.integers(0, 1 << 30, k)),
                            k_dur=rng.integers(0, 100, k), k_name=rng.integers(0, names, k).astype(np.uint32) * 7,
                            ncu_name=rng.integers(0, names, m).astype(np.uint32) * 7, counters=counters)
    assert_parity(gpu_run(t, mode=mode), oracle.run(t, mode=mode))


def _layered(slots, streams, shuffle=False):
    return tracegen.generate("dedup", n_slots=slots, n_streams=streams, n_iters=3, shuffle=shuffle)


@pytest.mark.parametrize("slots,streams", [(3, 1), (127, 2), (255, 1), (128, 2), (100, 3)])
@pytest.mark.parametrize("shuffle", [False, True])
def test_layer_counts(slots, streams, shuffle):
    t = _layered(slots, streams, shuffle)
    assert len(t.class_of_layer) == slots * streams
    assert_parity(gpu_run(t), oracle.run(t))


def _swap_rows(t):
    i = t.M // 2
    j = i + 1 + int(np.nonzero(t.ncu_name[i + 1:] != t.ncu_name[i])[0][0])
    order = np.arange(t.M)
    order[[i, j]] = order[[j, i]]
    stream = None if t.ncu_stream is None else t.ncu_stream[order].copy()
    return dataclasses.replace(t, ncu_name=t.ncu_name[order].copy(), counters=t.counters[order].copy(), ncu_stream=stream)


def _drop_row(t):
    keep = np.arange(t.M) != t.M // 3
    stream = None if t.ncu_stream is None else t.ncu_stream[keep].copy()
    return dataclasses.replace(t, ncu_name=t.ncu_name[keep].copy(), counters=t.counters[keep].copy(), ncu_stream=stream)


@pytest.mark.parametrize("case", ["layers", "layers_many", "streams", "plain", "layers_streams"])
@pytest.mark.parametrize("change", [None, _swap_rows, _drop_row])
@pytest.mark.parametrize("shuffle", [False, True])
def test_join_falls_back(case, change, shuffle):
    """A join goes ahead on the pairing that usually holds and redoes the
    matching when it does not: the three calls' outputs, warning and summary,
    and the oracle's."""
    import paper_2609_11938_gb300 as opa
    dd = case.startswith("layers")
    t = _layered(100, 3, shuffle) if case == "layers_many" else \
        tracegen.generate("dedup" if dd else "gpt2", n_iters=5, shuffle=shuffle)
    if case.endswith("streams"):
        t = tracegen.per_stream_runs(t)
    if change is not None:
        t = change(t)
    o = oracle.run(t, dedup=dd)
    tr = opa.to_device(t)
    with opa.Context(0) as ctx:
        st, out, ops, summ, tot = ctx.join(tr, dedup=dd)
        m_st, idx, kind, msumm = ctx.match(tr, dedup=dd)
    assert st == m_st == o["match_status"] and summ == msumm
    for g in (out["ncu_idx"], idx):
        np.testing.assert_array_equal(g.cpu().numpy(), o["ncu_idx"])
    for g in (out["match_kind"], kind):
        np.testing.assert_array_equal(g.cpu().numpy(), o["match_kind"])
    np.testing.assert_array_equal(out["range_of_kernel"].cpu().numpy(), o["range_of_kernel"])
    for k in oracle.SUMMARY_FIELDS:
        assert summ[k] == o["summary"][k], k
    for k in ("kernel_count", "total_duration_ns", "matched_count"):
        np.testing.assert_array_equal(ops[k].cpu().numpy(), o["ops"][k])
    assert tot["attributed_ns"] == o["totals"]["attributed_ns"]


def test_join_errors_in_order():
    """A bad layer id, bad tables and a range error: the first step's error."""
    import paper_2609_11938_gb300 as opa
    t = tracegen.generate("dedup", n_iters=3)
    bad = t.k_layer.copy()
    bad[7] = len(t.class_of_layer)
    wrong = np.full_like(t.rep_of_class, len(t.class_of_layer))
    end = t.r_end.copy()
    end[5] = t.r_start[5] - 1
    deep = t.r_end.copy()
    i = int(np.nonzero(t.r_depth == 1)[0][0])
    deep[i] = t.r_end.max() + 5
    with opa.Context(0) as ctx:
        for change, want in ((dict(k_layer=bad), opa.E_INVALID_ARG), (dict(rep_of_class=wrong), opa.E_INVALID_ARG),
                             (dict(r_end=deep, rep_of_class=wrong), opa.E_NOT_NESTED),
                             (dict(r_end=end, k_layer=bad), opa.E_INVALID_ARG), (dict(r_end=deep), opa.E_NOT_NESTED)):
            with pytest.raises(opa.OpattrError) as ei:
                ctx.join(opa.to_device(dataclasses.replace(t, **change)))
            assert ei.value.status == want, change.keys()
        st, out, *_ = ctx.join(opa.to_device(t))
        assert st == opa.OK
        np.testing.assert_array_equal(out["ncu_idx"].cpu().numpy(), oracle.run(t)["ncu_idx"])


@pytest.mark.parametrize("call", ["match", "join"])
@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("slots,streams,bad", [(3, 2, 6), (3, 2, 7), (3, 2, 254), (3, 2, 255), (3, 2, 1 << 30), (3, 2, -2),
                                               (254, 1, 254), (255, 1, 255), (255, 1, 256), (300, 1, 301)])
def test_bad_layer_ids(slots, streams, bad, shuffle, call):
    """Layer ids past the table, next to it and far off, on both sides of the
    counting pass: refused, and the context is as good as new."""
    import paper_2609_11938_gb300 as opa
    t = _layered(slots, streams, shuffle)
    ids = t.k_layer.copy()
    ids[[7, t.K // 2, t.K - 1]] = bad
    with opa.Context(0) as ctx:
        for trace in (dataclasses.replace(t, k_layer=ids), t):
            tr = opa.to_device(trace)
            run = (lambda: ctx.match(tr)[:3]) if call == "match" else \
                (lambda: (lambda st, out, *_: (st, out["ncu_idx"], out["match_kind"]))(*ctx.join(tr)))
            if trace is not t:
                with pytest.raises(opa.OpattrError) as ei:
                    run()
                assert ei.value.status == opa.E_INVALID_ARG
                continue
            st, idx, kind = run()
            o = oracle.run(t)
            assert st == o["match_status"]
            np.testing.assert_array_equal(idx.cpu().numpy(), o["ncu_idx"])
            np.testing.assert_array_equal(kind.cpu().numpy(), o["match_kind"])


@pytest.mark.parametrize("case", ["plain", "streams", "layers"])
def test_join_out_of_order_finds_no_key(case):
    """Records out of order whose rows follow the launches: paired through the
    time order, without the largest name that only the sort by names needs."""
    import paper_2609_11938_gb300 as opa
    t = tracegen.generate("dedup" if case == "layers" else "gpt2", n_iters=5, shuffle=True)
    if case == "streams":
        t = tracegen.per_stream_runs(t)
    o = oracle.run(t, dedup=case == "layers")
    tr = opa.to_device(t)
    with opa.Context(0) as ctx:
        ctx.set_timing(True)
        st, out, _, summ, _ = ctx.join(tr, dedup=case == "layers")
        ran = {k for k, (_, n) in ctx.timing_report().items() if n}
    assert st == opa.OK and summ["fast_path"] == 1
    np.testing.assert_array_equal(out["ncu_idx"].cpu().numpy(), o["ncu_idx"])
    assert "bucket_sort" in ran and not ran & {"max_key", "pair_keys"}


@pytest.mark.parametrize("case", ["plain", "names", "streams", "layers"])
def test_first_join_asks_for_scratch_once(case):
    """A context's first join launches what the next ones do: no scratch grows
    between its steps, which would leave the aggregation to zero its counters."""
    import paper_2609_11938_gb300 as opa
    if case == "layers":
        t = tracegen.generate("dedup", n_iters=400)
    else:
        t = tracegen.generate("large", n_kernels=3_000_000 if case == "plain" else 600_000, n_streams=4, seed=4)
        if case == "names":
            t = _drop_row(t)
        elif case == "streams":
            t = tracegen.per_stream_runs(t)
    tr = opa.to_device(t)
    with opa.Context(0) as ctx:
        n = []
        for _ in range(3):
            at = ctx.launch_count()
            ctx.join(tr, dedup=case == "layers")
            n.append(ctx.launch_count() - at)
    assert n[0] == n[1] == n[2], n
