"""Queries from a source without out-edges: one fill of the output, with fewer
and with more columns than the fill has threads, and rows of every alignment."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,S", [(1, 5000), (2, 3), (3, 1200), (64, 4096), (1000, 311), (1001, 311), (4096, 200),
                                 (311_296, 3), (311_297, 3), (1_245_184, 2), (1_245_188, 2)])
def test_isolated_source(V, S):
    import __graft_entry__ as g
    g.build()
    from paper_2502_10579_gb300 import svv
    source = V - 1
    n = min(V - 1, 8)
    src, dst = np.zeros(n, np.uint32), np.arange(n, dtype=np.uint32)  # every edge leaves vertex 0
    csr = svv.svv_build_versioned_csr(V, S, src, dst, np.ones(n, np.uint32), np.zeros(n, np.uint32), np.full(n, S, np.uint32))
    with svv.Context(0) as ctx:
        ctx.load_csr(V, S, *csr)
        for b, L in {(0, S), (S // 2, 1), (1, S - 1)}:
            for t, at_source, elsewhere in ((0, 0, 0xFFFFFFFF), (1, 0xFFFFFFFF, 0)):
                for off in (0, 1):
                    buf = torch.full((L * V + 8,), -7, dtype=torch.int32, device="cuda:0")
                    ctx.query(t, source, b, L, out=buf[off:off + L * V])
                    got = svv.to_u32(buf)
                    want = np.full((L, V), elsewhere, np.uint32)
                    want[:, source] = at_source
                    np.testing.assert_array_equal(got[off:off + L * V].reshape(L, V), want)
                    assert (got[:off] == 0xFFFFFFF9).all() and (got[off + L * V:] == 0xFFFFFFF9).all()
