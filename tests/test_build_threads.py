"""The versioned-graph builder on several host threads: rows in instance order,
masks and offsets as a plain sort gives them, whatever the ranges (one source
with most edges, sources without any, fewer vertices than threads)."""
import numpy as np
import pytest

from paper_2502_10579_gb300 import svv


@pytest.fixture(scope="module", autouse=True)
def built():
    import __graft_entry__ as g
    g.build()


@pytest.mark.parametrize("n", [0, 1, 65535, 400_000])
@pytest.mark.parametrize("V", [1, 3, 50, 4099])
def test_builder_matches_a_stable_sort(n, V):
    rng = np.random.default_rng(n + V)
    S, W = 70, 2
    src = np.minimum(rng.integers(0, V, n), rng.integers(0, V, n)).astype(np.uint32)
    src[rng.random(n) < 0.4] = V // 2
    dst, w = rng.integers(0, V, n).astype(np.uint32), rng.integers(0, 2**32, n).astype(np.uint32)
    a = rng.integers(0, S + 1, n).astype(np.uint32)
    d = rng.integers(0, S + 1, n).astype(np.uint32)
    rp, col, wt, mask = svv.svv_build_versioned_csr(V, S, src, dst, w, a, d)
    live = np.flatnonzero(a < d)
    order = live[np.argsort(src[live], kind="stable")]
    np.testing.assert_array_equal(rp, np.concatenate([[0], np.cumsum(np.bincount(src[live], minlength=V))]).astype(np.uint64))
    np.testing.assert_array_equal(col, dst[order])
    np.testing.assert_array_equal(wt, w[order])
    bits = (np.arange(64 * W)[None, :] >= a[order][:, None]) & (np.arange(64 * W)[None, :] < d[order][:, None])
    words = np.packbits(bits, axis=1, bitorder="little").view(np.uint64) if len(order) else np.zeros((0, W), np.uint64)
    np.testing.assert_array_equal(mask.reshape(-1, W), words)


def test_builder_refuses_bad_instances_anywhere():
    n = 300_000
    for field, value in (("src", 10), ("dst", 10), ("t_add", 6), ("t_del", 6)):
        for k in (0, n // 2, n - 1):
            x = dict(src=np.zeros(n, np.uint32), dst=np.zeros(n, np.uint32), w=np.ones(n, np.uint32),
                     t_add=np.zeros(n, np.uint32), t_del=np.ones(n, np.uint32))
            x[field][k] = value
            with pytest.raises(svv.SvvError) as e:
                svv.svv_build_versioned_csr(10, 5, **x)
            assert e.value.status == 1
