"""A batch beside a live server: both run on the batch teams' scratch and
barriers, so the batch comes after the requests already submitted, and the server
goes on afterwards, also when the batch needs other teams or longer rows."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_batch_beside_a_live_server():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    log = W.scaled_rmat(scale=12, edge_factor=8, n_snapshots=100, rate=0.002, seed=57, add_mode="skewed")
    rng = np.random.default_rng(3)
    served = [(int(rng.integers(0, 4)), int(rng.integers(0, log.V)), int(rng.integers(0, 60)), int(rng.integers(1, 41)))
              for _ in range(24)]
    batch = [(t, int(rng.integers(0, log.V)), 0, L) for t in range(4) for L in (8, 40, 100)]
    want = {q: oracle.query(log, *q) for q in served + batch}
    with svv.Context(0) as ctx:
        ctx.set_tuning("batch_mode", 1)
        ctx.load_log(log)
        svv.svv_serve_start(ctx.h, max_window=40, capacity=32, arena_bytes=32 << 20)
        for teams, specs in ((0, batch[:6]), (3, batch), (3, batch[::3]), (0, batch)):
            ctx.set_tuning("batch_teams", teams)
            tickets = [(svv.svv_submit(ctx.h, *q), q) for q in served]
            assert all(tk is not None for tk, _ in tickets)
            outs, status = ctx.query_batch([q for q in specs])
            assert status == [0] * len(specs)
            for q, out in zip(specs, outs):
                np.testing.assert_array_equal(svv.to_u32(out), want[q])
            for tk, q in tickets:
                assert svv.svv_poll(ctx.h, tk, wait=True) == 0
                addr, _, _ = svv.svv_ticket_info(ctx.h, tk)
                np.testing.assert_array_equal(svv.device_u32(addr, q[3] * log.V).reshape(q[3], log.V), want[q])
                svv.svv_release(ctx.h, tk)
        svv.svv_serve_stop(ctx.h)
