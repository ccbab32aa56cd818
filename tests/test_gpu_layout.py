"""The transposed graph at load, where its construction changes shape: no edge
present in every snapshot, no partial edge, neither; sorts of none to four passes
by weight and none to three by target (the sorted list changes buffers with every
pass); lists shorter and longer than a block of the sort."""
import numpy as np
import pytest

import oracle
from test_gpu_edge_counts import edge_log

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wmax", [0, 1, 255, 256, 70_000, 2**24, 2**32 - 1])
@pytest.mark.parametrize("V", [1, 2, 200, 257, 70_000])
@pytest.mark.parametrize("partial", [0.0, 0.02, 0.6, 1.0])
def test_layout(V, partial, wmax):
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    rng = np.random.default_rng(V + wmax)
    S, n = 5, {1: 3, 2: 5, 200: 1500, 257: 40_000, 70_000: 300_000}[V]
    src, dst = rng.integers(0, V, size=n), rng.integers(0, V, size=n)
    src[:V // 8] = 0
    dst[:n // 50] = V // 2  # an in-degree of its own
    w = rng.integers(0, wmax + 1, size=n)
    t_del = np.where(rng.random(n) < partial, rng.integers(1, S, size=n), S)
    log = edge_log(V, S, src, dst, w, t_del)
    with svv.Context(0) as ctx:
        ctx.set_tuning("pull_pct", 1)
        ctx.set_tuning("isolated_fast", 0)
        for _ in range(2):
            ctx.load_log(log)
            for t in (0, 1, 3):
                np.testing.assert_array_equal(svv.to_u32(ctx.query(t, 0, 0, S)), oracle.query(log, t, 0, 0, S))


def test_graph_without_edges():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    none = np.zeros(0, np.int64)
    log = edge_log(3, 2, none, none, none, none)
    with svv.Context(0) as ctx:
        ctx.set_tuning("isolated_fast", 0)
        ctx.load_log(log)
        assert svv.to_u32(ctx.query(0, 1, 0, 2)).tolist() == [[0xFFFFFFFF, 0, 0xFFFFFFFF]] * 2
