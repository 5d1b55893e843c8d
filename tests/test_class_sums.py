"""The class roll-up's two paths (GPU): up to 255 classes in one counting pass
with every warp on a share of one class, more of them by a sort; sizes about a
group of kernels and a block's warps, empty classes and classes left out, null
counters.  Against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_close
from test_gpu_parity import _agg_inputs, opa  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nan_frac", [0.0, 0.02])
@pytest.mark.parametrize("k", [1, 31, 33, 2048, 2049, 70_001])
@pytest.mark.parametrize("classes", [1, 2, 64, 254, 255, 256, 1000])
def test_class_counts(opa, k, classes, nan_frac):  # noqa: F811
    import torch
    t, rk, idx = _agg_inputs(k + classes, k, [], max(1, k // 3), nan_frac)
    rng = np.random.default_rng(k)
    # most classes empty or small, one large, some operators in none
    cls = np.minimum(rng.geometric(0.02, t.n_ops) - 1, classes - 1).astype(np.int64)
    cls[rng.random(t.n_ops) < 0.1] = 0xFFFFFFFF
    op = np.where(rk >= 0, t.r_op[np.maximum(rk, 0)].astype(np.int64), 0xFFFFFFFF).astype(np.uint32)
    want = oracle.rollup(t.k_dur, op, t.counters, idx, cls.astype(np.uint32), classes)
    want = want[1] if isinstance(want, tuple) else want
    with opa.Context(0) as ctx:
        _, got = ctx.rollup(opa.to_device(t), torch.from_numpy(rk).cuda(), torch.from_numpy(idx).cuda(),
                            torch.from_numpy(cls.astype(np.uint32).view(np.int32)).cuda(), classes)
    for key in ("kernel_count", "total_duration_ns", "matched_count"):
        np.testing.assert_array_equal(got[key].cpu().numpy(), want[key], err_msg=key)
    assert_close(got["agg"].cpu().numpy(), want["agg"], what="agg")
