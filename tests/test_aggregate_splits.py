"""Where the aggregation hands an operator over (GPU): one lane, a block of 128
threads, a block of 512, the pieces pass, with the lane's share following the
average length; with and without null counters, against the oracle."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import _agg_inputs, _check_aggregate, _gpu_aggregate, opa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nan_frac", [0.0, 0.03])
@pytest.mark.parametrize("n_small,k", [(20_000, 80_000),      # short operators: lanes take up to 64 kernels
                                       (200, 30_000),         # long ones: up to 256
                                       (1, 6_000)])           # one more, longer than any other
def test_operator_lengths(opa, n_small, k, nan_frac):  # noqa: F811
    lens = [1, 2, 63, 64, 65, 127, 128, 129, 255, 256, 257, 1023, 1024, 1025, 4095, 4096, 4097]
    t, rk, idx = _agg_inputs(31 + n_small, sum(lens) + k, lens, n_small, nan_frac)
    o = oracle.aggregate(t.k_dur, rk, t.r_op, t.counters, idx, t.n_ops)
    _check_aggregate(_gpu_aggregate(opa, t, rk, idx), o)


def test_infinite_counter_in_a_long_operator(opa):  # noqa: F811
    t, rk, idx = _agg_inputs(7, 20_000, [300, 2000], 5000)
    k = int(np.nonzero((t.r_op[np.maximum(rk, 0)] == 1) & (rk >= 0) & (idx >= 0))[0][100])
    t.counters[idx[k], 4] = np.inf
    with pytest.raises(opa.OpattrError) as ei:
        _gpu_aggregate(opa, t, rk, idx)
    assert ei.value.status == opa.E_INVALID_ARG
