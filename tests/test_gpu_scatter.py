"""Output rows at every alignment: vertex counts that are no multiple of 4 (rows
start at any word), tiles of 128 vertices and their remainders, output buffers
that start off a 16-byte boundary, every padded row length."""
import numpy as np
import pytest

import oracle
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 3, 127, 128, 129, 131, 254, 1021])
def test_output_alignment(V):
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    S = 130
    log = W.rmat.random_small_log(seed=V, V=V, n_edges=4 * V, S=S, n_add=max(1, V // 16), n_del=max(1, V // 16))
    want = oracle.query(log, 0, 0, 0, S)
    with svv.Context(0) as ctx:
        ctx.load_log(log)
        for b, L in [(0, 1), (2, 3), (1, 8), (5, 9), (0, 31), (7, 33), (0, 64), (3, 77), (0, 128), (0, 130)]:
            for off in (0, 1, 2, 3):
                buf = torch.full((L * V + 8,), -7, dtype=torch.int32, device="cuda:0")
                out = buf[off:off + L * V]
                ctx.query(0, 0, b, L, out=out)
                got = svv.to_u32(buf)
                np.testing.assert_array_equal(got[off:off + L * V].reshape(L, V), want[b:b + L])
                assert (got[:off] == 0xFFFFFFF9).all() and (got[off + L * V:] == 0xFFFFFFF9).all()


@pytest.mark.parametrize("V", [132, 256, 1020, 1024])
def test_output_in_several_wide_tiles(V):
    """Vertex counts that are multiples of 4: several tiles written 16 bytes at a
    time, and a last one that is not full and goes word by word."""
    test_output_alignment(V)
