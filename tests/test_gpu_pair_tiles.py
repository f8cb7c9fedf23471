"""The pair formula's 64 x 64 tiles and source ranges, and the distance and
count steps' 128-source columns, at the edges of both, against the oracle."""
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


def check(nat, g, flags):
    ref = oracle.bc(g)
    with nat.Graph.from_csr(g) as h:
        h.run(flags=flags)
        got, code, _ = h.result()
        hs = h.source_hashes(g.n)
    assert code == nat.BC_OK
    tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
    assert np.all(np.abs(got - ref["bc"]) <= tol), float(np.max(np.abs(got - ref["bc"])))
    for k in ("hash_sigma", "hash_dist", "dist_sum", "reach"):
        assert np.array_equal(hs[k], ref[k]), k


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 129, 640])
@pytest.mark.parametrize("form", ["unweighted", "weighted", "products"])
def test_tile_edges(nat, n, form):
    wmax = 1 if form == "unweighted" else 6
    g = G.random_small(n, min(1.0, 6.0 / n), 4100 + n, wmax=wmax, connect=n % 2 == 0) if n > 1 else \
        G.csr_from_edges(1, [], [], None if form == "unweighted" else [])
    check(nat, g, nat.BC_DENSE if form == "products" else nat.BC_PAIRS)


def test_products_directed(nat):
    """The steps pull over in-arcs; unreachable pairs stay out."""
    check(nat, G.directed_random(300, 0.012, 4200, wmax=9), nat.BC_DENSE)


@pytest.mark.parametrize("k", [1, 127, 128, 129, 700])
def test_product_source_columns(nat, k):
    """Source counts around the 128-source columns, repeats included."""
    import ctypes
    g = G.random_small(150, 0.05, 4300, wmax=4, connect=False)
    src = (np.arange(k, dtype=np.int32) * 7) % 150
    sig, dist = np.empty((k, 150), np.uint64), np.empty((k, 150), np.int32)
    opt = nat.make_options(0, nat.BC_DENSE)
    with nat.Graph.from_csr(g) as h:
        assert h.lib.bc_forward_rows(h.handle, nat._addr(src), k, nat._addr(sig), nat._addr(dist), ctypes.byref(opt),
                                     nat._stream_ptr(None)) == nat.BC_OK
    for s in np.unique(src):
        o = oracle.source(g, int(s), with_delta=False)
        for i in np.nonzero(src == s)[0]:
            assert np.array_equal(dist[i], o["dist"].astype(np.int32)) and np.array_equal(sig[i], o["sigma"])
