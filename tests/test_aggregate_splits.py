"""Where the aggregation hands an operator over (GPU): one lane, a block of 128
threads, a block of 512, the pieces pass, with the lane's share following the
average length; with and without null counters, against the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
import tracegen
from gpu_util import assert_parity, gpu_run
from test_gpu_parity import _agg_inputs, _check_aggregate, _gpu_aggregate, opa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nan_frac", [0.0, 0.03])
@pytest.mark.parametrize("n_small,k", [(20_000, 80_000),      # short operators: lanes take up to 64 kernels
                                       (200, 30_000),         # long ones: up to 128
                                       (1, 6_000)])           # one more, longer than any other
def test_operator_lengths(opa, n_small, k, nan_frac):  # noqa: F811
    lens = [1, 2, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, 4095, 4096, 4097]
    t, rk, idx = _agg_inputs(31 + n_small, sum(lens) + k, lens, n_small, nan_frac)
    o = oracle.aggregate(t.k_dur, rk, t.r_op, t.counters, idx, t.n_ops)
    _check_aggregate(_gpu_aggregate(opa, t, rk, idx), o)


@pytest.mark.parametrize("n_ops", [1, 4094, 4095, 4096, 32_766, 32_767, 32_768, 77_823, 77_824, 77_825])
@pytest.mark.parametrize("call", ["aggregate", "join", "join_many"])
def test_operator_counts(opa, n_ops, call):  # noqa: F811
    """Where the offsets come from (the count's last block, one block, a chained
    scan) and how many operators a warp takes; with the counters zeroed for the
    call, in a join with those the enclosure's reset left (twice: the arena
    grows in the first), and in one with more operators than records."""
    if call == "aggregate":
        t, rk, idx = _agg_inputs(n_ops, n_ops + 5000, [], n_ops)
        _check_aggregate(_gpu_aggregate(opa, t, rk, idx),
                         oracle.aggregate(t.k_dur, rk, t.r_op, t.counters, idx, t.n_ops))
        return
    t = tracegen.generate("large", n_kernels=int(n_ops * 4.2) if call == "join" else 500, n_streams=2, seed=9)
    t = dataclasses.replace(t, n_ops=max(n_ops, t.n_ops))
    want = gpu_run(t)
    assert_parity(want, oracle.run(t, enclose_mode="indexed"))
    tr = opa.to_device(t)
    with opa.Context(0) as ctx:
        for _ in range(2):
            st, out, ops, summary, totals = ctx.join(tr)
            assert st == want["match_status"] and summary == want["summary"] and totals == want["totals"]
            for k, v in ops.items():
                np.testing.assert_array_equal(v.cpu().numpy(), want["ops"][k])


def test_infinite_counter_in_a_long_operator(opa):  # noqa: F811
    t, rk, idx = _agg_inputs(7, 20_000, [300, 2000], 5000)
    k = int(np.nonzero((t.r_op[np.maximum(rk, 0)] == 1) & (rk >= 0) & (idx >= 0))[0][100])
    t.counters[idx[k], 4] = np.inf
    with pytest.raises(opa.OpattrError) as ei:
        _gpu_aggregate(opa, t, rk, idx)
    assert ei.value.status == opa.E_INVALID_ARG
