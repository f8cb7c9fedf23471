"""The packed weighted sweep on graphs with hubs and on dense ones, on both
sides of the lines between its thread counts (arcs per largest weight, and the
mean degree of 5 up to which one warp takes wider steps), and with buckets that
many vertices share: below their capacity and past it."""
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


def weighted(g, wmax, seed):
    u, v, _ = g.edges()
    return G.csr_from_edges(g.n, u, v, 1 + G.Stream(seed, 8).below(u.size, wmax), name=f"{g.name}_w{wmax}")


@pytest.mark.parametrize("g,wmax,sources", [
    (G.rmat_lcc(10, 16), 200, None),         # 32 threads: a width of some 25
    (G.rmat_lcc(10, 16), 100, None),         # 64, just above 40
    (G.rmat_lcc(10, 16), 40, None),          # 64, near 150
    (G.rmat_lcc(10, 16), 20, None),          # 128
    (G.rmat_lcc(12, 16), 2, 300),            # 128: wide steps, too few vertices for 256
    (G.star_graph(3000), 100, 200),          # 32: a hub of 2999 arcs on one lane
    (G.barabasi_albert(2000, 3, 5), 50, 200),  # 64
    (G.gnp(900, 0.06, 7), 1000, 200),        # 32: mean degree 54, a width of 12
    (G.gnp(900, 0.06, 7), 4000, 200),        # most vertices within a few hundred distances of one another
    (G.er_hamiltonian(1200, 1500, 9), 30, 300),  # mean degree below 5: 32
], ids=lambda x: getattr(x, "name", str(x)))
def test_hubs_and_dense_rows(nat, g, wmax, sources):
    g = weighted(g, wmax, 91)
    src = None if sources is None else G.sample_sources(g.n, sources, 92)
    ref = oracle.bc(g, src)
    with nat.Graph.from_csr(g) as h:
        outs = []
        for _ in range(2):
            h.run(src)
            got, code, _ = h.result()
            assert code == nat.BC_OK
            hs = h.source_hashes(g.n if src is None else len(src))
            for k in ("hash_sigma", "hash_dist", "dist_sum", "reach"):
                assert np.array_equal(hs[k], ref[k]), k
            assert h.run_stats()[0] == int(ref["arcs"].sum())
            outs.append(got)
    tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
    assert np.all(np.abs(outs[0] - ref["bc"]) <= tol), float(np.max(np.abs(outs[0] - ref["bc"])))
    assert np.array_equal(outs[0], outs[1])


@pytest.mark.parametrize("n,p,lo,hi", [(1200, 0.02, 95, 100), (1200, 0.02, 100, 100), (2500, 0.004, 3990, 4000), (700, 0.5, 1, 900)])
def test_crowded_buckets(nat, n, p, lo, hi):
    """Weights in a narrow band: whole frontiers share a few distances, past the
    buckets' capacity (256 entries at the least) or just below it."""
    u, v, _ = G.gnp(n, p, 93).edges()
    g = G.csr_from_edges(n, u, v, lo + G.Stream(94, 8).below(u.size, hi - lo + 1), name="band")
    src = G.sample_sources(n, 150, 95)
    ref = oracle.bc(g, src)
    with nat.Graph.from_csr(g) as h:
        h.run(src)
        got, code, _ = h.result()
        hs = h.source_hashes(len(src))
    assert code == nat.BC_OK
    for k in ("hash_sigma", "hash_dist", "dist_sum", "reach"):
        assert np.array_equal(hs[k], ref[k]), k
    tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * n)
    assert np.all(np.abs(got - ref["bc"]) <= tol), float(np.max(np.abs(got - ref["bc"])))
