"""The edge counts of svv_get_stats in rounds that pull, and by them that such
rounds ran: on graphs whose rounds are known, a push round counts every edge of
its frontier, a pull round those of targets that can still improve."""
import numpy as np
import pytest

import oracle
from test_gpu_pull import WEIGHTS, make_log
from workloads.rmat import EdgeLog

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S = 140


def edge_log(V, S, src, dst, w, t_del):
    n = len(src)
    src, dst, w, t_del = (np.asarray(x).astype(np.uint32) for x in (src, dst, w, t_del))
    dels = [np.flatnonzero(t_del == s) if s else np.zeros(0, np.int64) for s in range(S)]
    return EdgeLog(V=V, S=S, src=src, dst=dst, w=w, add_off=np.concatenate([[0], np.full(S, n)]).astype(np.int64),
                   del_off=np.concatenate([[0], np.cumsum([d.shape[0] for d in dels])]).astype(np.int64),
                   del_ids=np.concatenate(dels).astype(np.int64), t_add=np.zeros(n, np.uint32), t_del=t_del, meta={})


M, D = 2000, 64  # vertices of a layer, in-edges of each vertex of the second one


def layers(seed, wmax):
    """0 -> 1..M by edges gone in the last snapshots, then D in-edges from that
    layer to each of M + 1..2M: nothing but 0 is reached in the intersection of a
    window that ends late, and every other vertex is unstable."""
    rng = np.random.default_rng(seed)
    src = np.concatenate([np.zeros(M, np.int64), rng.integers(1, M + 1, size=M * D)])
    dst = np.concatenate([np.arange(1, M + 1), np.repeat(np.arange(M + 1, 2 * M + 1), D)])
    gone = np.concatenate([rng.integers(S - 10, S, size=M), np.full(M * D, S)])
    return edge_log(2 * M + 1, S, src, dst, rng.integers(1, wmax + 1, size=len(src)), gone)


@pytest.fixture(scope="module")
def svv():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    return svv


def test_pull_rounds_of_a_solve_count_the_edges_they_try(svv):
    """0 -> 1..513 -> 514, both rounds pulled: the first reads every edge once
    (and 31 slots of padding), in the second only the last vertex can still improve."""
    n = 513
    src = np.concatenate([np.zeros(n, np.int64), np.arange(1, n + 1)])
    dst = np.concatenate([np.arange(1, n + 1), np.full(n, n + 1)])
    log = edge_log(n + 2, 4, src, dst, np.ones(2 * n), np.full(2 * n, 4))
    with svv.Context(0) as ctx:
        ctx.set_tuning("pull_pct", 1)
        ctx.load_log(log)
        out = svv.to_u32(ctx.query(0, 0, 0, 4))
        assert (out[:, 1:n + 1] == 1).all() and (out[:, n + 1] == 2).all()
        assert 2 * n <= ctx.stats()["edges_relaxed_cap"] <= 3 * n + 62


@pytest.mark.parametrize("L", [20, 40, 64, 100])  # rows of 32, 64 and 128 values
@pytest.mark.parametrize("prune", [1, 0])
def test_relaxation_pulls_and_counts(svv, L, prune):
    log = layers(1, 1)
    b = S - L
    want = oracle.query(log, 2, 0, b, L)
    counts = {}
    for pull in (0, 1):
        with svv.Context(0) as ctx:
            ctx.set_tuning("pull", pull)
            ctx.set_tuning("prune", prune)
            ctx.load_log(log)
            np.testing.assert_array_equal(svv.to_u32(ctx.query(2, 0, b, L)), want)
            st = ctx.stats()
            assert st["unstable"] == 2 * M + 1 - prune
            counts[pull] = st["edges_relaxed_multi"]
    # pushed: the first layer's M * D out-edges.  Pulled: each vertex of the
    # second layer is done after the first few of its in-edges of every item
    # (16 of them), and every one of them needs at least one.
    assert counts[0] == M * D
    assert M <= counts[1] <= M * D // 2

@pytest.mark.parametrize("mode", [1, 2])
@pytest.mark.parametrize("wmax", [1, 300])
def test_batches_on_a_graph_whose_relaxations_pull(svv, mode, wmax):
    """The same graph in batches: teams of the one-launch kernel (with their own
    scratch, several slabs in one launch) and query groups, every type."""
    log = layers(2, wmax)
    want = {t: oracle.query(log, t, 0, 0, S) for t in range(4)}
    specs = [(t, 0, b, L) for t in range(4) for b, L in [(0, S), (S - 20, 20), (S - 40, 40), (S - 64, 64), (30, 105)]]
    with svv.Context(0) as ctx:
        ctx.set_tuning("batch_mode", mode)
        ctx.set_tuning("batch_teams", 3)
        ctx.load_log(log)
        for _ in range(2):
            outs, status = ctx.query_batch(specs)
            assert status == [0] * len(specs)
            for (t, _, b, L), out in zip(specs, outs):
                np.testing.assert_array_equal(svv.to_u32(out), want[t][b:b + L])
        for pair in ([(2, 0, S - 40, 40), (2, 0, S - 41, 40)], [(0, 0, S - 64, 64), (1, 0, S - 70, 64)]):
            ctx.set_tuning("group_mix", 1)
            outs, status = ctx.query_batch(pair)
            for (t, _, b, L), out in zip(pair, outs):
                np.testing.assert_array_equal(svv.to_u32(out), want[t][b:b + L])


@pytest.mark.parametrize("kind", list(WEIGHTS))
@pytest.mark.parametrize("V", [33, 5000])
def test_one_launch_batches_pull_in_their_solves(svv, V, kind):
    """The in-degrees and weights of test_gpu_pull in the one-launch kernel."""
    log = make_log(V, WEIGHTS[kind], seed=V)
    specs = [(t, s, b, L) for t in range(4) for s, b, L in [(0, 0, log.S), (0, 5, 40), (V - 3, 64, 6), (0, 3, 17)]]
    want = [oracle.query(log, *q) for q in specs]
    with svv.Context(0) as ctx:
        ctx.set_tuning("pull_pct", 1)
        ctx.set_tuning("batch_mode", 1)
        ctx.load_log(log)
        for teams in (1, 8):
            ctx.set_tuning("batch_teams", teams)
            outs, status = ctx.query_batch(specs)
            assert status == [0] * len(specs)
            for q, out, w in zip(specs, outs, want):
                np.testing.assert_array_equal(svv.to_u32(out), w, err_msg=str(q))
