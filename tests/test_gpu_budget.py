"""Batches under a hard budget: a budget that holds some team's scratch is
answered with as many teams as fit, whatever bytes are left over, and a call that
fails gives back what it took."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def svv():
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    return svv


def batch(svv, log, specs, budget):
    ctx = svv.Context(0, hbm_budget_bytes=budget)
    ctx.set_tuning("batch_mode", 1)
    ctx.set_tuning("batch_teams", 8)
    ctx.load_log(log)
    loaded = ctx.device_bytes()
    try:
        outs, status = ctx.query_batch(specs)
    except svv.SvvError as e:
        return ctx, loaded, e.status, None
    assert status == [0] * len(specs)
    return ctx, loaded, ctx.stats()["batch_teams"], [svv.to_u32(o) for o in outs]


def test_teams_fit_what_the_budget_leaves(svv):
    log = W.small_rmat()
    specs = [(t, 0, 0, 8) for t in (0, 1, 2, 3)] * 2
    want = [oracle.query(log, *q) for q in specs]
    ctx, loaded, teams, _ = batch(svv, log, specs, 4 << 30)
    full = ctx.device_bytes()
    ctx.close()
    assert teams == 8
    team = (full - loaded) // 8
    for less in (0, 1, 256, 4096, 20_000, 50_000, 80_000, team - 4096, team + 1, 3 * team + 256, 6 * team + 50_000):
        ctx, _, teams, outs = batch(svv, log, specs, full - less)
        assert ctx.device_bytes() <= full - less
        assert 8 - 1 - -(-less // team) <= teams <= 8 - (less > 0), (less, teams)
        for o, w in zip(outs, want):
            np.testing.assert_array_equal(o, w)
        ctx.close()


def test_refused_batch_keeps_no_bytes(svv):
    """Not even one team fits: refused, again and again, with the same bytes held."""
    log = W.small_rmat()
    specs = [(0, 0, 0, 8)] * 3
    probe, loaded, _, _ = batch(svv, log, specs, 4 << 30)
    probe.close()
    ctx, _, status, _ = batch(svv, log, specs, loaded + (512 << 10))  # a team takes 818 KB
    assert status == 2
    held = ctx.device_bytes()
    for _ in range(3):
        with pytest.raises(svv.SvvError):
            ctx.query_batch(specs)
        assert ctx.device_bytes() == held
    ctx.set_tuning("batch_mode", 2)  # what needs no teams still runs
    np.testing.assert_array_equal(svv.to_u32(ctx.query(0, 0, 0, 8)), oracle.query(log, 0, 0, 0, 8))
    ctx.close()


def test_regrown_pair_rows_are_counted_once(svv):
    """A pair of longer windows replaces the pair arrays: the bytes held are
    those of a context that ran the longer pair only."""
    log = W.scaled_rmat(scale=12, edge_factor=8, n_snapshots=100, rate=0.002, seed=58, add_mode="skewed")
    held = []
    for lengths in ((100,), (8, 30, 100)):
        with svv.Context(0) as ctx:
            ctx.set_tuning("batch_mode", 2)
            ctx.load_log(log)
            for L in lengths:
                outs, status = ctx.query_batch([(0, 0, 0, L), (0, 1, 0, L)])
                assert status == [0, 0]
                np.testing.assert_array_equal(svv.to_u32(outs[0]), oracle.query(log, 0, 0, 0, L))
            held.append(ctx.device_bytes())
    assert held[0] == held[1]
