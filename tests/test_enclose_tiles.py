"""The enclosure's tiles (GPU) where they can go wrong: parts and tiles of a few
events and one more, more ranges in a tile than one step takes, more streams or
levels than the common layout holds, instants at which many ranges start and
end together cut by a tile's edge, and times that outgrow 32 bits.  Against the
oracle."""
import dataclasses

import numpy as np
import pytest

import oracle
import tracegen
from gpu_util import assert_parity, gpu_run

pytestmark = pytest.mark.gpu


def _check(t):
    assert_parity(gpu_run(t), oracle.run(t, enclose_mode="indexed"))


@pytest.mark.parametrize("n", [1, 395, 396, 397, 800, 16_000, 16_800, 70_001])
def test_tile_edges(n):
    """About 1.29 events per kernel; a tile holds 512 in small traces, and past
    32 parts the carried ranges come from their own pass."""
    _check(tracegen.generate("large", n_kernels=n, n_streams=3, seed=n))


@pytest.mark.parametrize("streams,depth", [(64, 3), (65, 3), (70, 2), (16, 32), (17, 32), (20, 30), (64, 32), (66, 32)])
@pytest.mark.parametrize("shuffle", [False, True])
def test_layouts(streams, depth, shuffle):
    """Streams and levels on both sides of the common layout (64 streams, 512
    levels) and of the wide one (2,048 levels)."""
    _check(tracegen.generate("adversarial", n_kernels=30_000, n_streams=streams, max_depth=depth, seed=streams + depth,
                             shuffle=shuffle))


@pytest.mark.parametrize("shuffle", [False, True])
@pytest.mark.parametrize("streams,depth,n", [(130, 5, 30_000), (255, 4, 30_000), (130, 32, 300), (200, 32, 80_000),
                                             (256, 32, 60_000)])
def test_groups_of_streams(streams, depth, n, shuffle):
    """Past 64 streams, and taken by groups of 16 past 2,048 levels: groups
    without kernels, without ranges and with neither, few events and many."""
    t = tracegen.generate("adversarial", n_kernels=n, n_streams=streams, max_depth=depth, seed=n + depth, shuffle=shuffle)
    _check(t)
    k, r = t.k_stream // 16, t.r_stream // 16
    keep_k, keep_r = ~np.isin(k, (1, 4, 7)), ~np.isin(r, (2, 4))
    t = dataclasses.replace(t, **{f: getattr(t, f)[keep_k].copy() for f in ("k_stream", "k_start", "k_dur", "k_name")},
                            **{f: getattr(t, f)[keep_r].copy() for f in ("r_stream", "r_start", "r_end", "r_depth", "r_op")})
    _check(t)


@pytest.mark.parametrize("seed", range(4))
def test_ties_in_groups_of_streams(seed):
    """Equal starts out of (start, end) order on many streams: sorted, then grouped."""
    t = tracegen.small_random(500 + seed, n_streams=90, n_events=300, t_max=40, max_depth=5, shuffle=bool(seed & 1),
                              n_names=7)
    # with a chain of 32 levels on every stream, long before
    s, d = np.divmod(np.arange(90 * 32), 32)
    add = lambda a, v: np.concatenate([a, v.astype(a.dtype)])
    _check(dataclasses.replace(t, r_stream=add(t.r_stream, s), r_depth=add(t.r_depth, d), r_start=add(t.r_start, d - 500),
                               r_end=add(t.r_end, -400 - d), r_op=add(t.r_op, 0 * s)))


def test_groups_of_many_short_streams():
    """More than 160 streams and 4M events: by groups, though the levels are few."""
    _check(tracegen.generate("adversarial", n_kernels=4_400_000, n_streams=200, max_depth=3, seed=8))


@pytest.mark.parametrize("seed", range(6))
def test_ties_across_tiles(seed):
    """Thousands of events at few instants: ties of starts, ends and kernels
    run over tile and step edges (ranges in array order and permuted)."""
    t = tracegen.small_random(400 + seed, n_streams=1 + seed % 3, n_events=9000, t_max=40, max_depth=5,
                              shuffle=bool(seed & 1), n_names=7)
    _check(t)


def test_ranges_without_kernels():
    """Many more ranges than kernels: tiles of ranges alone, taken in steps."""
    t = tracegen.generate("large", n_kernels=60_000, n_streams=2, seed=3)
    keep = np.arange(t.K) < 40
    n = int(keep.sum())
    t = dataclasses.replace(t, k_stream=t.k_stream[:n].copy(), k_start=t.k_start[:n].copy(), k_dur=t.k_dur[:n].copy(),
                            k_name=t.k_name[:n].copy(), ncu_name=t.ncu_name[:n].copy(), counters=t.counters[:n].copy())
    _check(t)


def _stretch(t, bits):
    t0 = min(int(t.k_start.min()), int(t.r_start.min()))
    return dataclasses.replace(t, k_start=(t.k_start - t0) << bits, r_start=(t.r_start - t0) << bits,
                               r_end=(t.r_end - t0) << bits)


@pytest.mark.parametrize("streams,depth", [(3, 6), (66, 12), (200, 32)])
@pytest.mark.parametrize("bits", [12, 17, 24])
@pytest.mark.parametrize("shuffle", [False, True])
def test_long_traces(streams, depth, bits, shuffle):
    """Times stretched until a part, then a step, then the gap between two
    events is longer than the 32 bits that times in a step have: open ranges
    are made relative to a later event, with ends past 32 bits among them, or
    the trace is taken again with wider times; by each call and by a join."""
    import paper_2609_11938_gb300 as opa
    t = _stretch(tracegen.generate("adversarial", n_kernels=20_000, n_streams=streams, max_depth=depth, seed=bits,
                                   shuffle=shuffle), bits)
    _check(t)
    o = oracle.run(t, enclose_mode="indexed")
    with opa.Context(0) as ctx:
        _, out, ops, _, _ = ctx.join(opa.to_device(t))
    np.testing.assert_array_equal(out["range_of_kernel"].cpu().numpy(), o["range_of_kernel"])
    np.testing.assert_array_equal(out["n_op_enclosing"].cpu().numpy(), o["n_op_enclosing"])
    np.testing.assert_array_equal(ops["kernel_count"].cpu().numpy(), o["ops"]["kernel_count"])


@pytest.mark.parametrize("streams", [2, 80])
@pytest.mark.parametrize("seed", range(4))
def test_ties_far_apart(streams, seed):
    """Few instants, 17 s apart, with many events each: in array order, and out
    of (start, end) order within a level."""
    t = tracegen.small_random(700 + seed, n_streams=streams, n_events=18_000 // streams, t_max=60, max_depth=5,
                              shuffle=bool(seed & 1), n_names=7)
    _check(_stretch(t, 34))
