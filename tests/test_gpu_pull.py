"""Pull rounds over the transposed graph (a lane per target, in-edges sorted by
weight): in-degrees around every edge of the layout (no in-edge, one item, the
next item, the longest slice, hubs), extreme weights, partial edges, one and
several value lanes, against the oracle."""
import numpy as np
import pytest

import oracle
from workloads.rmat import EdgeLog

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# in-degrees of the first targets: items end at 16 steps, slices at 512, hubs above
DEGREES = [0, 1, 15, 16, 17, 31, 32, 33, 48, 511, 512, 513, 544, 545, 1700]


def make_log(V, weights, seed, S=70):
    """Targets 1.. with the in-degrees above (cut to what V allows), a chain so
    that most vertices are reachable, and edges that come and go."""
    rng = np.random.default_rng(seed)
    src, dst = [], []
    for i, d in enumerate(DEGREES):
        t = 1 + i
        if t >= V:
            break
        src.append(rng.integers(0, V, size=d))
        dst.append(np.full(d, t))
    src.append(np.arange(0, V - 1))
    dst.append(np.arange(1, V))
    extra = 3 * V
    src.append(rng.integers(0, V, size=extra))
    dst.append(rng.integers(0, V, size=extra))
    src, dst = (np.concatenate(x).astype(np.uint32) for x in (src, dst))
    n = src.shape[0]
    w = np.asarray(weights, np.uint32)[rng.integers(0, len(weights), size=n)]
    t_add = np.where(rng.random(n) < 0.2, rng.integers(0, S, size=n), 0).astype(np.uint32)
    t_del = np.where(rng.random(n) < 0.2, rng.integers(1, S + 1, size=n), S).astype(np.uint32)
    t_del = np.maximum(t_del, t_add + 1)  # live in at least one snapshot
    order = np.argsort(t_add, kind="stable")
    src, dst, w, t_add, t_del = (x[order] for x in (src, dst, w, t_add, t_del))
    add_off = np.searchsorted(t_add, np.arange(S + 1)).astype(np.int64)
    dels = [np.flatnonzero(t_del == s) if s else np.zeros(0, np.int64) for s in range(S)]
    del_off = np.concatenate([[0], np.cumsum([d.shape[0] for d in dels])]).astype(np.int64)
    return EdgeLog(V=V, S=S, src=src, dst=dst, w=w, add_off=add_off, del_off=del_off,
                   del_ids=np.concatenate(dels).astype(np.int64), t_add=t_add, t_del=t_del, meta={})


@pytest.fixture(scope="module")
def svv():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    return svv


WEIGHTS = {"unit": [1], "small": list(range(1, 300)), "extreme": [0, 1, 2, 2**31, 2**32 - 2, 2**32 - 1]}


@pytest.mark.parametrize("V", [2, 33, 1025, 5000])
@pytest.mark.parametrize("kind", list(WEIGHTS))
def test_pull_rounds(svv, V, kind):
    log = make_log(V, WEIGHTS[kind], seed=V)
    windows = [(0, log.S), (5, 40), (64, 6)]
    with svv.Context(0) as ctx:
        ctx.set_tuning("pull_pct", 1)
        ctx.set_tuning("group_pull_pct", 1)
        ctx.set_tuning("group_pull_pct_union", 1)
        ctx.load_log(log)
        want = {}
        for t in range(4):
            for b, L in windows:
                want[t, b, L] = oracle.query(log, t, 0, b, L)
                np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 0, b, L)), want[t, b, L])
        np.testing.assert_array_equal(svv.to_u32(ctx.query(1, 0, 5, 4, plain=True)), want[1, 5, 40][:4])
        # the same in query groups: 2, 4 and 8 value lanes, one type and several
        ctx.set_tuning("batch_mode", 2)
        full = [(t, 0, b, L) for t in range(4) for b, L in windows]
        for mix, specs in [(0, [q for q in full for _ in range(n)]) for n in (1, 2)] + [(1, full), (1, full[::3]), (1, full[2:11:6])]:
            ctx.set_tuning("group_mix", mix)
            outs, status = ctx.query_batch(specs)
            assert status == [0] * len(specs)
            for (t, _, b, L), out in zip(specs, outs):
                np.testing.assert_array_equal(svv.to_u32(out), want[t, b, L])


@pytest.mark.parametrize("kind", list(WEIGHTS))
@pytest.mark.parametrize("V", [33, 1025, 5000])
def test_relaxation_pull_rounds(svv, V, kind):
    """Without pruning every vertex has a row and most rows change at once, so
    the relaxation's rounds pull: rows of 32, 64 and 128 values, slabs, one query
    and pairs (one type and several), every type."""
    log = make_log(V, WEIGHTS[kind], seed=V + 1)
    lens = [17, 32, 33, 64, 65, 70]
    with svv.Context(0) as ctx:
        ctx.set_tuning("prune", 0)
        ctx.set_tuning("batch_mode", 2)
        ctx.set_tuning("group_mix", 1)
        ctx.load_log(log)
        want = {t: oracle.query(log, t, 0, 0, log.S) for t in range(4)}
        for L in lens:
            for t in range(4):
                b = (3 * t) % (log.S - L + 1)
                np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 0, b, L)), want[t][b:b + L])
            for t0, t1 in [(0, 0), (1, 1), (0, 1), (2, 3), (1, 2)]:
                b = (log.S - L) // 2
                outs, status = ctx.query_batch([(t0, 0, 0, L), (t1, 0, b, L)])
                assert status == [0, 0]
                np.testing.assert_array_equal(svv.to_u32(outs[0]), want[t0][:L])
                np.testing.assert_array_equal(svv.to_u32(outs[1]), want[t1][b:b + L])
        ctx.set_tuning("slab_max", 40)
        np.testing.assert_array_equal(svv.to_u32(ctx.query(0, 0, 0, log.S)), want[0])


def test_source_far_from_targets(svv):
    """Most targets unreachable: nothing ends early, every in-edge is looked at."""
    log = make_log(3000, WEIGHTS["small"], seed=9)
    with svv.Context(0) as ctx:
        ctx.set_tuning("pull_pct", 1)
        ctx.load_log(log)
        for t in range(4):
            np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 2990, 3, 50)), oracle.query(log, t, 2990, 3, 50))


@pytest.mark.parametrize("blocks", [1, 0])
def test_rounds_that_queue_mostly_hubs(svv, blocks):
    """Every vertex has 34 work units, so one push round lists far more vertices
    per CTA than its hub list holds (blocks_per_sm = 1), or about as many."""
    rng = np.random.default_rng(5)
    V, d = 24000, 544
    n = V * d
    log = EdgeLog(V=V, S=2, src=np.repeat(np.arange(V, dtype=np.uint32), d),
                  dst=rng.integers(0, V, size=n).astype(np.uint32), w=rng.integers(1, 1000, size=n).astype(np.uint32),
                  add_off=np.array([0, n, n]), del_off=np.array([0, 0, 100]), del_ids=np.arange(100),
                  t_add=np.zeros(n, np.uint32), t_del=np.where(np.arange(n) < 100, 1, 2).astype(np.uint32), meta={})
    with svv.Context(0) as ctx:
        ctx.set_tuning("solve_chunk", 16)
        ctx.set_tuning("pull_pct", 0)
        ctx.set_tuning("group_pull_pct", 0)
        ctx.set_tuning("blocks_per_sm", blocks)
        ctx.load_log(log)
        want = [oracle.query(log, t, 0, 0, 2) for t in (0, 2)]
        for t, w in zip((0, 2), want):
            np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 0, 0, 2)), w)
        ctx.set_tuning("batch_mode", 2)
        outs, _ = ctx.query_batch([(0, 0, 0, 2), (0, 0, 0, 1), (0, 0, 1, 1)])
        np.testing.assert_array_equal(svv.to_u32(outs[0]), want[0])
        np.testing.assert_array_equal(svv.to_u32(outs[2]), want[0][1:])
