"""The packed weighted sweep at the edges of its forms: threads per source by
step width, rows around the eight-arc records, buckets that overflow into a
scan, rings of one warp's counters and more, and a graph too large for packed
arcs; distances, counts (by summaries) and BC against the oracle."""
import numpy as np
import pytest

import oracle
from paper_0809_1906_gb300 import graphs as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    from paper_0809_1906_gb300 import native
    native.load()
    return native


def check(nat, g, sources=None, **kw):
    ref = oracle.bc(g, sources) if sources is not None else oracle.bc(g)
    with nat.Graph.from_csr(g) as h:
        h.run(sources, **kw)
        got, code, _ = h.result()
        hs = h.source_hashes(g.n if sources is None else len(sources))
        arcs, _ = h.run_stats()
        h.run(sources, **kw)
        again, _, _ = h.result()
    assert code == nat.BC_OK
    for k in ("hash_sigma", "hash_dist", "dist_sum", "reach"):
        assert np.array_equal(hs[k], ref[k]), k
    tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
    assert np.all(np.abs(got - ref["bc"]) <= tol), float(np.max(np.abs(got - ref["bc"])))
    assert np.array_equal(got, again)


# n / maxw below 72, 150, 4000 and above: 32, 64, 128 and 256 threads
@pytest.mark.parametrize("n,wmax", [(300, 20), (300, 3), (700, 2), (4200, 1)])
@pytest.mark.parametrize("directed", [False, True])
def test_thread_counts(nat, n, wmax, directed):
    if directed:
        g = G.directed_random(n, 4.0 / n, 5100 + n, wmax=wmax)
    else:
        g = G.random_small(n, 4.0 / n, 5100 + n, wmax=max(wmax, 2), connect=n % 200 != 0)
        g = G.Graph(g.n, g.row_ptr, g.col, np.minimum(g.w, wmax).astype(np.int32), "w")
    check(nat, g, None if n < 1000 else G.sample_sources(n, 64, 3))


@pytest.mark.parametrize("deg", [1, 4, 5, 7, 8, 9, 11, 12, 40])
@pytest.mark.parametrize("n,wmax", [(60, 4), (300, 1)])
def test_row_lengths(nat, deg, n, wmax):
    """Circulant graphs: every row has exactly 2 * (deg / 2) arcs, or one more by a matching."""
    at = np.arange(n, dtype=np.int64)
    u = [at for _ in range(deg // 2)]
    v = [(at + k + 1) % n for k in range(deg // 2)]
    if deg % 2:
        u.append(at[: n // 2])
        v.append(at[: n // 2] + n // 2)
    u, v = np.concatenate(u), np.concatenate(v)
    w = 1 + (u * 7 + v * 3 + u * v) % wmax  # the same from either end only by the stored pair
    check(nat, G.csr_from_edges(n, u, v, w, name="circulant"))


@pytest.mark.parametrize("wmax", [2, 31, 32, 33, 200, 4000])
def test_ring_sizes(nat, wmax):
    g = G.random_small(150, 0.04, 5300 + wmax, wmax=wmax, connect=True)
    check(nat, g)


def test_bucket_overflow_scans(nat):
    """A hub whose 900 leaves all fall into one bucket, far past its capacity."""
    n = 1000
    u = np.concatenate([np.zeros(900, np.int64), np.arange(900, 999)])
    v = np.concatenate([np.arange(1, 901), np.arange(901, 1000)])
    w = np.concatenate([np.full(900, 5), 1 + np.arange(99)])
    check(nat, G.csr_from_edges(n, u, v, w, name="hub"))


def test_more_vertices_than_packed_heads(nat):
    """A binary tree of 2^20 + 5 vertices: heads past the packed arcs' 20 bits, plain CSR rows."""
    n = (1 << 20) + 5
    v = np.arange(1, n, dtype=np.int64)
    g = G.csr_from_edges(n, (v - 1) // 2, v, 1 + v % 3, name="tree")
    check(nat, g, np.array([0, 5, n - 1], np.int32))
