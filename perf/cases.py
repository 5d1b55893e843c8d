"""What the speed of the framework is measured on: attribution joins as a user
of the library runs them, through ``Context`` (join, the three calls, the
attribution tiers, the class roll-up), from a trace of a few thousand kernel
records to one of fifty million.

A case is a dict of plain values:

  call          what one pass calls
                  join     Context.join: enclosure, matching and aggregation in one call
                  calls    Context.enclose, .match and .aggregate, one after another
                  tiers    Context.enclose, .attribute (correlation and fusion maps),
                           .match, and .aggregate by each kernel's operator
                  rollup   Context.rollup over the results of an earlier join
  kernels       kernel records
  streams       streams they ran on
  depth         deepest nesting of the ranges
  block, ranges kernel records and ranges of one block (a dispatch tree, or a
                layer): the trace is a sequence of blocks drawn from a pool
  bare          share of a block's kernels that lie outside every range
  names         kernel names, drawn Zipf(zipf)
  slots, classes  layered traces: layers of a stream and their structural
                classes (0: operator trees without layers)
  rows          the ncu rows in hand
                  all         one per launch, in launch order
                  stream      one per launch, replayed stream by stream, tagged
                  names       launches of two names in three (a kernel filter)
                  cut         the first 97 % of the launches (a capture cut short)
                  layers      launches of each class's representative layer and
                              outside layers: layer deduplication
  nulls         share of counter values that are null (NaN)
  shuffle       kernel and range records in no order
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2609_11938_gb300 as opa

_DEV = "cuda:0"
NC = 20
SUM = (0, 1, 2, 10, 14, 18)             # counters added up; MAX the largest value; the
MAX = (17, 19)                          # others a mean weighted by duration
STRUCTURAL, NONOP, NONE = 0xFFFFFFFF, 0xFFFFFFFE, 0xFFFFFFFF
ROLLUP_CLASSES = 64

_PLAIN = dict(call="join", kernels=2000, streams=1, depth=4, block=60, ranges=10, bare=0.1, names=40, zipf=1.1,
              slots=0, classes=0, rows="all", nulls=0.0, shuffle=False)


def _case(name, **kw):
    return dict(_PLAIN, name=name, **kw)


def listed():
    return [
        # one step of a small model: what an interactive profiler asks for, over and over
        _case("join_2k"),
        # fifty steps of a 12-layer model on one stream, ncu rows of one layer of the twelve only
        _case("join_dedup_26k", kernels=26_000, depth=6, block=40, ranges=12, bare=0.0, names=120, slots=12,
              classes=1, rows="layers"),
        # the same model on two streams, every launch profiled
        _case("join_52k", kernels=52_000, streams=2, depth=6, block=40, ranges=12, bare=0.0, names=120, slots=12,
              classes=1),
        # a deeper model on four streams, 48 layers in three classes, deduplicated
        _case("join_dedup_416k", kernels=416_000, streams=4, depth=6, block=40, ranges=12, bare=0.0, names=120,
              slots=12, classes=3, rows="layers"),
        # the three calls by themselves (a caller that looks at each result), some counters absent
        _case("calls_1m", call="calls", kernels=1_000_003, streams=8, depth=8, block=60, ranges=16, bare=0.05,
              names=1000, nulls=0.02),
        # ncu rows that a kernel filter left: ordinals by name, the other names unmatched
        _case("join_names_2m", kernels=2_099_999, streams=4, depth=6, block=50, ranges=14, bare=0.05, names=500,
              rows="names"),
        # a multi-stream capture that ncu replayed one stream per run
        _case("join_stream_3m", kernels=3_000_017, streams=16, depth=8, block=61, ranges=16, bare=0.05, names=2000,
              rows="stream"),
        # all attribution tiers: correlation map, ranges, fusion map
        _case("tiers_4m", call="tiers", kernels=4_000_001, streams=8, depth=8, block=63, ranges=16, bare=0.05,
              names=2000),
        # records merged from several exports, in no order
        _case("join_shuffled_6m", kernels=6_000_011, streams=16, depth=8, block=63, ranges=16, bare=0.05, names=5000,
              shuffle=True),
        # the per-class breakdown of a large trace
        _case("rollup_8m", call="rollup", kernels=8_000_009, streams=16, depth=8, block=62, ranges=16, bare=0.05,
              names=5000),
        # a long training capture
        _case("join_20m", kernels=20_000_000, streams=16, depth=8, block=63, ranges=16, bare=0.05, names=5000),
        # the largest: most kernels outside the ranges, ranges nested to the limit
        _case("join_deep_50m", kernels=50_000_000, streams=64, depth=32, block=220, ranges=64, bare=0.8, names=50000,
              zipf=1.5),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    c = dict(_PLAIN)
    c["call"] = rng.choice(["join", "join", "join", "calls", "tiers", "rollup"])
    c["kernels"] = _log_int(rng, 2000, 20_000_000)
    c["streams"] = rng.choice([1, 2, 3, 4, 7, 8, 16, 24])
    c["depth"] = rng.choice([4, 5, 6, 8, 8, 12])
    c["block"] = rng.randint(36, 90)
    c["ranges"] = rng.randint(9, 20)
    c["bare"] = round(rng.choice([0.0, 0.03, 0.05, 0.1, 0.3]), 2)
    c["names"] = _log_int(rng, 40, 10_000)
    if rng.random() < 0.3:
        c["slots"] = rng.choice([4, 12, 24])
        c["classes"] = rng.choice([1, 2, 3])
        c["bare"] = 0.0
    c["rows"] = rng.choice(["all", "all", "stream", "names", "cut", "layers"])
    if c["rows"] == "layers" and not c["slots"]:
        c["rows"] = "all"
    c["nulls"] = rng.choice([0.0, 0.0, 0.02])
    c["shuffle"] = rng.random() < 0.2
    return c


# ---------------------------------------------------------------- inputs
def _blocks(case):
    """Blocks of a stream: enough for the kernels, whole iterations of a layered trace."""
    per = max(1, -(-case["kernels"] // (case["streams"] * case["block"])))
    step = case["slots"] + 1 if case["slots"] else 1
    return -(-per // step) * step


def _zipf(case):
    w = np.arange(1, case["names"] + 1, dtype=np.float64) ** -case["zipf"]
    return w / w.sum()


def _others(case):
    """Ranges of a block, under its root, that are no operators."""
    return int(0.08 * case["ranges"])


def _template(rs, case):
    """One block: `ranges` ranges in a random tree of at most `depth` levels
    under one root, `block` kernels spread over them (a `bare` share before the
    root).  Returns the kernels' and ranges' places in the event sequence."""
    n_r, n_k, depth = case["ranges"], case["block"], case["depth"]
    parent, level = [-1], [0]
    lean = 0.93 if depth > 12 else 0.55                 # how often a range nests in the one just pushed
    for i in range(1, n_r):
        p = i - 1 if rs.rand() < lean else rs.randint(0, i)
        while level[p] + 1 >= depth:
            p = rs.randint(0, i)
        parent.append(p)
        level.append(level[p] + 1)
    n_bare = int(round(case["bare"] * n_k))
    owner = rs.randint(0, n_r, n_k - n_bare)
    kids = [[] for _ in range(n_r)]
    for i in range(1, n_r):
        kids[parent[i]].append(("r", i))
    for i in owner:
        kids[i].insert(rs.randint(0, len(kids[i]) + 1), ("k", 0))
    k_ev, push, pop, n = list(range(n_bare)), [0] * n_r, [0] * n_r, n_bare
    stack = [("r", 0)]
    while stack:
        what, i = stack.pop()
        if what == "k":
            k_ev.append(n)
        elif what == "r":
            push[i] = n
            stack.append(("e", i))
            stack.extend(reversed(kids[i]))
        else:
            pop[i] = n
        n += 1
    kind = np.zeros(n_r, np.int64)                            # operator, namespaced non-op (1), structural (2)
    other = rs.permutation(np.arange(1, n_r))[:_others(case)]
    kind[other] = np.where(rs.rand(len(other)) < 0.4, 2, 1)
    if case["slots"]:
        kind[0] = 2                                           # a layer or step marker
    return np.array(k_ev), np.array(push), np.array(pop), np.array(level), kind


def _trace(case, seed):
    """The arrays of one trace on the GPU, as a dict."""
    rs = np.random.RandomState(seed % (2**32 - 1))
    gen = torch.Generator(device=_DEV)
    gen.manual_seed(seed)
    dev = dict(device=_DEV)
    S, B, n_k, n_r = case["streams"], _blocks(case), case["block"], case["ranges"]
    E = n_k + 2 * n_r
    layered = case["slots"] > 0
    n_t = case["classes"] + 1 if layered else 48
    tpl = [_template(rs, case) for _ in range(n_t)]
    put = lambda j: torch.from_numpy(np.stack([t[j] for t in tpl]).astype(np.int64)).to(_DEV)
    k_ev, push, pop, level, kind = (put(j) for j in range(5))
    slot = None
    if layered:
        slot = torch.arange(B, **dev) % (case["slots"] + 1) - 1            # -1: outside layers
        which = torch.where(slot < 0, 0, 1 + slot % case["classes"]).repeat(S, 1)
    else:
        which = torch.randint(0, n_t, (S, B), generator=gen, **dev)

    # host time before each event (one in ten is none at all), kernel time after each kernel
    host = torch.empty((S, B * E), **dev).exponential_(1 / 500.0, generator=gen)
    host *= torch.rand((S, B * E), generator=gen, **dev) >= 0.1
    t = host.round_().long().cumsum(1)
    del host
    dur = torch.randn((S, B, n_k), generator=gen, **dev).mul_(1.2).exp_().mul_(8000.0).round_().clamp_(min=1).long()
    gap = torch.empty((S, B, n_k), **dev).exponential_(1 / 2000.0, generator=gen).round_().long()
    base = (torch.arange(B, **dev) * E)[None, :, None]
    ke = (k_ev[which] + base).reshape(S, -1)
    busy = torch.zeros((S, B * E + 1), dtype=torch.int64, **dev)
    busy.scatter_(1, ke + 1, (dur + gap).reshape(S, -1))
    t += busy.cumsum_(1)[:, :-1]
    del gap, busy
    t += 1_700_000_000_000_000_000 + torch.randint(0, 100_000, (S, 1), generator=gen, **dev)

    # kernel records in time order, the first `kernels` of them
    K = case["kernels"]
    p = torch.from_numpy(_zipf(case)).to(_DEV).cumsum(0)
    if layered:
        name = torch.searchsorted(p, torch.rand((n_t, n_k), dtype=torch.float64, generator=gen, **dev))[which].reshape(-1)
    else:
        name = torch.searchsorted(p.float(), torch.rand(S * B * n_k, generator=gen, **dev))
    name = name.clamp_(max=case["names"] - 1)
    start = t.gather(1, ke).reshape(-1)
    del ke
    order = torch.argsort(start, stable=True)[:K]
    per = B * n_k
    out = dict(k_stream=(order // per).to(torch.uint8), k_start=start[order], k_dur=dur.reshape(-1)[order],
               k_name=name[order].int(), k_layer=None)
    if layered:
        sid = torch.arange(S, **dev)[:, None]
        layer = torch.where(slot < 0, -1, sid * case["slots"] + slot)[:, :, None].expand(S, B, n_k)
        out["k_layer"] = layer.reshape(-1)[order].int()
    del start, dur, name, order

    # range records in start order; every operator dispatch has an id of its own
    rs_ = t.gather(1, (push[which] + base).reshape(S, -1)).reshape(-1)
    re_ = t.gather(1, (pop[which] + base).reshape(S, -1)).reshape(-1)
    del t
    # ranges of one instant follow the order they were pushed in
    pushed = push[which].argsort(2) + (torch.arange(S * B, **dev) * n_r).reshape(S, B, 1)
    pushed = pushed.reshape(-1)
    order = pushed[torch.argsort(rs_[pushed], stable=True)]
    kd = kind[which].reshape(-1)[order]
    is_op = kd == 0
    op = torch.where(is_op, is_op.long().cumsum(0) - 1, torch.where(kd == 1, NONOP, STRUCTURAL))
    op = torch.where(op >= 2**31, op - 2**32, op).int()                    # u32 ids as the bits of an i32
    out.update(r_stream=(order // (B * n_r)).to(torch.uint8), r_start=rs_[order], r_end=re_[order],
               r_depth=level[which].reshape(-1)[order].to(torch.uint8), r_op=op, n_ops=int(is_op.sum()))
    del order, pushed, kd, is_op, rs_, re_

    # ncu rows: one per replayed launch in launch order, or what the case has of them
    out.update(class_of_layer=None, rep_of_class=None, ncu_stream=None)
    rows = torch.arange(K, **dev)
    if case["rows"] == "layers":
        L = S * case["slots"]
        out["class_of_layer"] = np.arange(L, dtype=np.int32) % case["slots"] % case["classes"]
        out["rep_of_class"] = np.arange(case["classes"], dtype=np.int32)
        lay = out["k_layer"].long()
        rows = rows[(lay < 0) | (lay < case["classes"])]
    elif case["rows"] == "names":
        rows = rows[out["k_name"] % 3 != 2]
    elif case["rows"] == "cut":
        rows = rows[:max(1, int(0.97 * K))]
    elif case["rows"] == "stream":
        rows = torch.argsort(out["k_stream"], stable=True)
        out["ncu_stream"] = out["k_stream"][rows].contiguous()
    out["ncu_name"] = out["k_name"][rows].contiguous()
    M = rows.numel()
    ctr = torch.rand((M, NC), generator=gen, **dev)
    if layered:
        ctr.mul_(math.log(1e6)).exp_().mul_(1e-3)                          # rates over six decades
    else:
        ctr.mul_(100.0)
    if case["nulls"]:
        ctr[torch.rand((M, NC), generator=gen, **dev) < case["nulls"]] = math.nan
    out["counters"] = ctr

    if case["call"] == "tiers":
        # a correlation map of half the launches: (name, launches of that name before, the operator
        # dispatched last before the launch), in no order; a fusion operator for a tenth of the names
        nm = out["k_name"].long()
        inv = _rank_in_groups(nm)
        ops_at = out["r_start"][(out["r_op"] >= 0)]
        opk = (torch.searchsorted(ops_at, out["k_start"], right=True) - 1).clamp_(0, max(out["n_ops"] - 1, 0))
        pick = torch.randperm(K, generator=gen, **dev)[:K // 2]
        fo = torch.randint(0, max(out["n_ops"], 1), (case["names"],), generator=gen, **dev)
        fused = torch.rand(case["names"], generator=gen, **dev) < 0.1
        out.update(corr_name=nm[pick].int(), corr_inv=inv[pick].int(), corr_op=opk[pick].int(),
                   fusion_op=torch.where(fused, fo, -1).int(),
                   fusion_len=torch.randint(1, 5, (case["names"],), generator=gen, **dev).to(torch.uint8))
    if case["shuffle"]:
        pk, pr = torch.randperm(K, generator=gen, **dev), torch.randperm(out["r_start"].numel(), generator=gen, **dev)
        for f in ("k_stream", "k_start", "k_dur", "k_name", "k_layer"):
            if out[f] is not None:
                out[f] = out[f][pk].contiguous()
        for f in ("r_stream", "r_start", "r_end", "r_depth", "r_op"):
            out[f] = out[f][pr].contiguous()
    if case["call"] == "rollup":
        w = np.arange(1, ROLLUP_CLASSES + 1, dtype=np.float64) ** -1.1
        cdf = torch.from_numpy(np.cumsum(w / w.sum())).to(_DEV)
        cls = torch.searchsorted(cdf, torch.rand(out["n_ops"], dtype=torch.float64, generator=gen, **dev))
        cls = cls.clamp_(max=ROLLUP_CLASSES - 1)
        out["class_of_op"] = torch.where(torch.rand(out["n_ops"], generator=gen, **dev) < 0.02, -1, cls).int()
    return out


def _mode(case):
    return "prefix" if case["rows"] == "cut" else "skip_name"


def prepare(case, seed):
    """A trace in device memory and a context, as a program holds them; for a
    roll-up also the ranges and rows that an earlier join gave each kernel."""
    a = _trace(case, seed)
    extra = {k: a.pop(k) for k in ("class_of_op",) if k in a}
    st = dict(trace=opa.DeviceTrace(**a), ctx=opa.Context(0, mismatch=_mode(case)), call=case["call"], **extra)
    if case["call"] == "rollup":
        rok, _ = _enclosing(a)
        st["range_of_kernel"] = rok.int()
        st["ncu_idx"] = _rows_of(a, _mode(case))[0].int()
    return st


def run(state):
    ctx, tr = state["ctx"], state["trace"]
    if state["call"] == "join":
        status, out, ops, summary, totals = ctx.join(tr)
        return dict(status=status, kernels=out, ops=ops, summary=summary, totals=totals)
    if state["call"] == "rollup":
        status, ops = ctx.rollup(tr, state["range_of_kernel"], state["ncu_idx"], state["class_of_op"], ROLLUP_CLASSES)
        return dict(status=status, ops=ops)
    _, rok, nop = ctx.enclose(tr)
    kernels = dict(range_of_kernel=rok, n_op_enclosing=nop)
    op = tiers = None
    if state["call"] == "tiers":
        _, op, tier, fused_with, is_fused, tiers = ctx.attribute(tr, rok, nop)
        kernels.update(op=op, tier=tier, fused_with=fused_with, is_fused=is_fused)
    status, idx, kind, summary = ctx.match(tr)
    kernels.update(ncu_idx=idx, match_kind=kind)
    _, ops, totals = ctx.aggregate(tr, rok, idx, op_of_kernel=op)
    return dict(status=status, kernels=kernels, ops=ops, summary=summary, totals=totals, tiers=tiers)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    K, S = case["kernels"], case["streams"]
    R = S * _blocks(case) * case["ranges"]
    ops = S * _blocks(case) * (case["ranges"] - _others(case) - (1 if case["slots"] else 0))
    M, row = K, 84
    if case["rows"] == "layers":
        M = K * (S + case["classes"]) / (S * (case["slots"] + 1))
    elif case["rows"] == "names":
        M = K * float(_zipf(case)[np.arange(case["names"]) % 3 != 2].sum())
    elif case["rows"] == "cut":
        M = 0.97 * K
    elif case["rows"] == "stream":
        row = 85
    if case["call"] == "rollup":                   # duration, range, row per kernel; operator per range; class per operator
        return {"bytes": int(16 * K + 4 * R + 4 * ops + 80 * M + 184 * ROLLUP_CLASSES), "flops": 0}
    per = 1 + 8 + 8 + 4 + (4 + 1) + (4 + 1)        # stream, start, duration, name; range and count, row and kind
    if case["rows"] == "layers":
        per += 4
    b = per * K + 22 * R + row * M + 184 * ops
    if case["call"] == "tiers":                    # operator, tier, fused operator, fused flag; the two maps
        b += (4 + 1 + 4 + 1) * K + 12 * (K // 2) + 5 * case["names"]
    return {"bytes": int(b), "flops": 0}


def tolerance(case):
    # whole numbers are exact; sums are held in about 48 bits: 0.6e-15 to
    # 3.6e-15 (the roll-up) off the 64-bit results below
    return {"rel": 2e-14, "max": 2e-12}


# ---------------------------------------------------------------- the same in plain torch, 64 bits
def _rank_in_groups(key):
    """Rank of each element among the equal keys before it, in array order."""
    order = torch.argsort(key, stable=True)
    sk = key[order]
    first = torch.searchsorted(sk, sk)
    rank = torch.empty_like(key)
    rank[order] = torch.arange(key.numel(), device=key.device) - first
    return rank


def _u32(x):
    return x.long() & 0xFFFFFFFF


def _enclosing(a):
    """Range of each kernel (-1 none) and operator ranges collected on the way out."""
    ks, kt = a["k_stream"].long(), a["k_start"]
    tmin = min(int(kt.min()), int(a["r_start"].min()))
    order = torch.argsort(a["r_end"], stable=True)
    level = a["r_stream"].long() * 32 + a["r_depth"].long()
    key = (level << 45) | (a["r_start"] - tmin)
    order = order[torch.argsort(key[order], stable=True)]
    key, level, end, op = key[order], level[order], a["r_end"][order], _u32(a["r_op"])[order]
    rok = torch.full_like(kt, -1)
    nop = torch.zeros_like(kt)
    alive = torch.ones_like(kt, dtype=torch.bool)
    for d in range(int(a["r_depth"].max()) + 1):
        p = torch.searchsorted(key, ((ks * 32 + d) << 45) | (kt - tmin), right=True) - 1
        q = p.clamp(min=0)
        alive &= (p >= 0) & (level[q] == ks * 32 + d) & (end[q] >= kt)
        o = op[q]
        cut, hit = alive & (o == STRUCTURAL), alive & (o < NONOP)
        rok = torch.where(cut, -1, torch.where(hit, order[q], rok))
        nop = torch.where(cut, 0, nop + hit)
    return rok, nop


def _time_order(a):
    order = torch.argsort(a["k_stream"], stable=True)
    return order[torch.argsort(a["k_start"][order], stable=True)]


def _rows_of(a, mode):
    """ncu row of each kernel (-1 none) and how it was matched (0 not, 1 by its own row, 2 through its class)."""
    order = _time_order(a)
    name, row_name = _u32(a["k_name"]), _u32(a["ncu_name"])
    dedup = a["class_of_layer"] is not None
    replayed = torch.ones_like(name, dtype=torch.bool)
    if dedup:
        rep = torch.from_numpy(a["rep_of_class"][a["class_of_layer"]]).to(_DEV).long()
        lay = a["k_layer"].long()
        replayed = (lay < 0) | (rep[lay.clamp(min=0)] == lay)
    key, row_key = name, row_name
    if a["ncu_stream"] is not None:
        key, row_key = name << 8 | a["k_stream"].long(), row_name << 8 | a["ncu_stream"].long()
    rk = order[replayed[order]]
    kk = key[rk]
    ordinal = _rank_in_groups(kk)
    by_name = torch.argsort(row_key, stable=True)
    srt = row_key[by_name]
    lo, hi = torch.searchsorted(srt, kk), torch.searchsorted(srt, kk, right=True)
    skk = kk.sort().values
    launches = torch.searchsorted(skk, kk, right=True) - torch.searchsorted(skk, kk)
    ok = ordinal < hi - lo
    if mode == "skip_name":
        ok &= launches == hi - lo
    idx = torch.full_like(name, -1)
    idx[rk] = torch.where(ok, by_name[(lo + ordinal).clamp(max=max(srt.numel() - 1, 0))], -1)
    kind = (idx >= 0).to(torch.uint8)
    if dedup:
        tagged = order[lay[order] >= 0]
        tl = lay[tagged]
        pos = _rank_in_groups(tl)
        by_layer = torch.argsort(tl, stable=True)
        sl = tl[by_layer]
        r = rep[tl]
        rlo, rhi = torch.searchsorted(sl, r), torch.searchsorted(sl, r, right=True)
        src = tagged[by_layer[(rlo + pos).clamp(max=sl.numel() - 1)]]
        got = (r != tl) & (rlo + pos < rhi) & (name[src] == name[tagged]) & (idx[src] >= 0)
        dup = r != tl
        idx[tagged[dup]] = torch.where(got, idx[src], -1)[dup]
        kind[tagged[dup]] = torch.where(got, 2, 0).to(torch.uint8)[dup]
    return idx, kind


def _records(a, op, idx, n):
    """Per-operator records: `op` of each kernel, -1 for none."""
    att = op >= 0
    o, d, j = op[att], a["k_dur"][att], idx[att]
    zero = lambda dt: torch.zeros(n, dtype=dt, device=_DEV)
    out = dict(kernel_count=zero(torch.int64).index_add_(0, o, torch.ones_like(o)),
               total_duration_ns=zero(torch.int64).index_add_(0, o, d))
    m = j >= 0
    o, d, j = o[m], d[m], j[m]
    out["matched_count"] = zero(torch.int64).index_add_(0, o, torch.ones_like(o))
    agg = torch.full((NC, n), math.nan, dtype=torch.float64, device=_DEV)
    for c in range(NC):
        v = a["counters"][:, c][j].double()
        there = ~v.isnan()
        oc, vc, dc = o[there], v[there], d[there].double()
        some = zero(torch.int64).index_add_(0, oc, torch.ones_like(oc)) > 0
        if c in MAX:
            x = zero(torch.float64).fill_(-math.inf).scatter_reduce_(0, oc, vc, "amax")
        elif c in SUM:
            x = zero(torch.float64).index_add_(0, oc, vc)
        else:
            w = zero(torch.float64).index_add_(0, oc, dc)
            some &= w > 0
            x = zero(torch.float64).index_add_(0, oc, vc * dc) / w
        agg[c] = torch.where(some, x, math.nan)
    out["agg"] = agg
    return out


def exact(case, seed):
    a = _trace(case, seed)
    rok, nop = _enclosing(a)
    idx, kind = _rows_of(a, _mode(case))
    r_op = _u32(a["r_op"])
    op = torch.where(rok >= 0, r_op[rok.clamp(min=0)], -1)
    if case["call"] == "rollup":
        cls = torch.where(op >= 0, a["class_of_op"].long()[op.clamp(min=0)], -1)
        return dict(status=None, ops=_records(a, cls, idx, ROLLUP_CLASSES))
    kernels = dict(range_of_kernel=rok.int(), n_op_enclosing=nop.to(torch.uint8), ncu_idx=idx.int(), match_kind=kind)
    if case["call"] == "tiers":
        order = _time_order(a)
        name = _u32(a["k_name"])
        inv = torch.empty_like(name)
        inv[order] = _rank_in_groups(name[order])
        at, pos = (a["corr_name"].long() << 32 | a["corr_inv"].long()).sort()
        want = name << 32 | inv
        q = torch.searchsorted(at, want).clamp(max=max(at.numel() - 1, 0))
        high = at[q] == want if at.numel() else torch.zeros_like(want, dtype=torch.bool)
        fo = a["fusion_op"].long()[name]
        op = torch.where(high, a["corr_op"].long()[pos[q]] if at.numel() else -1, torch.where(op >= 0, op, fo))
        tier = torch.where(high, 1, torch.where(rok >= 0, 2, torch.where(fo >= 0, 3, 0)))
        fused = ((fo >= 0) & (a["fusion_len"].long()[name] > 1)) | ((tier == 2) & (nop > 1))
        kernels.update(op=op.int(), tier=tier.to(torch.uint8), fused_with=fo.int(), is_fused=fused.to(torch.uint8))
    total, att = int(a["k_dur"].sum()), int(a["k_dur"][op >= 0].sum())
    totals = dict(total_ns=total, attributed_ns=att, unattributed_ns=total - att, kernels=case["kernels"],
                  attributed_kernels=int((op >= 0).sum()), matched_kernels=int(((op >= 0) & (idx >= 0)).sum()),
                  attributed_frac=att / total, unattributed_frac=(total - att) / total)
    return dict(status=None, kernels=kernels, ops=_records(a, op, idx, a["n_ops"]), summary=None, totals=totals,
                tiers=None)
