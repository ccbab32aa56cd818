"""A subgraph row's room: the edges present in all window snapshots from its
front, the others from its back, and nothing between them when every edge is kept
(no pruning); and the bytes that partial edges take."""
import numpy as np
import pytest

import oracle
from test_gpu_edge_counts import edge_log

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def svv():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    return svv


def random_log(V, n, S, partial, seed):
    rng = np.random.default_rng(seed)
    src, dst = rng.integers(0, V, size=n), rng.integers(0, V, size=n)
    src[: n // 4] = 0  # a row of many chunks
    return edge_log(V, S, src, dst, rng.integers(1, 100, size=n),
                    np.where(rng.random(n) < partial, rng.integers(1, S, size=n), S))


@pytest.mark.parametrize("V", [1, 40, 700])
@pytest.mark.parametrize("partial", [0.0, 0.5, 1.0])
def test_full_rooms(svv, V, partial):
    S = 80
    log = random_log(V, 12 * V, S, partial, V)
    want = {t: oracle.query(log, t, 0, 0, S) for t in range(4)}
    with svv.Context(0) as ctx:
        ctx.load_log(log)
        for prune in (0, 1):
            ctx.set_tuning("prune", prune)
            for t in range(4):
                for b, L in [(0, 4), (30, 12), (0, 20), (9, 64), (0, 77), (0, S)]:
                    np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 0, b, L)), want[t][b:b + L])
            ctx.set_tuning("batch_mode", 2)
            ctx.set_tuning("group_mix", 1)
            for specs in ([(0, 0, 0, 12), (0, 0, 40, 12)], [(0, 0, 3, 70), (1, 0, 10, 70)], [(2, 0, 1, 20), (3, 0, 50, 20)]):
                outs, status = ctx.query_batch(specs)
                assert status == [0, 0]
                for (t, _, b, L), out in zip(specs, outs):
                    np.testing.assert_array_equal(svv.to_u32(out), want[t][b:b + L])
        ctx.set_tuning("batch_mode", 1)
        specs = [(t, 0, b, L) for t in range(4) for b, L in [(0, 4), (30, 12), (0, 20), (0, S)]]
        outs, status = ctx.query_batch(specs)
        for (t, _, b, L), out in zip(specs, outs):
            np.testing.assert_array_equal(svv.to_u32(out), want[t][b:b + L])


def test_partial_edges_take_no_room_twice(svv):
    """A partial edge is held as such once more (target and weight, source, masks);
    the queries' scratch does not grow with it until a window's masks are needed."""
    V, n, S = 5000, 60_000, 64
    held = []
    for partial in (0.0, 1.0):
        with svv.Context(0) as ctx:
            ctx.set_tuning("pull", 0)
            ctx.load_log(random_log(V, n, S, partial, 1))
            held.append(ctx.device_bytes())
    assert held[1] - held[0] <= n * (8 + 4 + 8) + 3 * 256
