"""The unweighted sweep's forms against each other and the oracle: the whole
run in one launch (up to 8192 vertices) and a launch per level (BC_TIMING, or
more vertices), vertices of few arcs in packs and of more arcs one by one, at
the edges of both. The forms add the same terms per source in the same order,
so BC differs by the FP64 sums over sources alone: 2^-40 relative bounds that
with room for every vertex and batch count here."""
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


HASHES = ("hash_sigma", "hash_dist", "dist_sum", "reach")


def run(nat, h, k, sources=None, batch=0, flags=0):
    h.run(sources, batch=batch, flags=flags)
    bc, code, _ = h.result()
    assert code == nat.BC_OK
    return bc, h.source_hashes(k), h.run_stats()


def check(nat, g, sources=None, batch=0, flags=0):
    ref = oracle.bc(g, sources) if sources is not None else oracle.bc(g)
    k = g.n if sources is None else len(sources)
    with nat.Graph.from_csr(g) as h:
        one, hs, stats = run(nat, h, k, sources, batch, flags)
        again, _, _ = run(nat, h, k, sources, batch, flags)
        per, hp, stats_per = run(nat, h, k, sources, batch, flags | nat.BC_TIMING)
    assert np.array_equal(one, again)
    assert np.all(np.abs(one - per) <= 2.0 ** -40 * np.abs(per))
    for name in HASHES:
        assert np.array_equal(hs[name], ref[name]), name
        assert np.array_equal(hp[name], ref[name]), name
    assert stats == stats_per
    tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
    assert np.all(np.abs(one - ref["bc"]) <= tol), float(np.max(np.abs(one - ref["bc"])))


def circulant(n, deg):
    at = np.arange(n, dtype=np.int64)
    u = [at for _ in range(deg // 2)]
    v = [(at + k + 1) % n for k in range(deg // 2)]
    if deg % 2:
        u.append(at[: n // 2])
        v.append(at[: n // 2] + n // 2)
    return G.csr_from_edges(n, np.concatenate(u), np.concatenate(v), name=f"circulant{n}_{deg}")


@pytest.mark.parametrize("batch", [32, 64, 128, 256])
@pytest.mark.parametrize("deg", [1, 2, 3, 4, 7, 8, 9, 33])
def test_degrees_around_the_light_limit(nat, deg, batch):
    check(nat, circulant(210, deg), batch=batch)


@pytest.mark.parametrize("n,p,batch", [(2, 1.0, 32), (33, 0.2, 32), (257, 0.01, 64), (700, 0.02, 256), (3000, 0.0012, 256)])
def test_random_ragged(nat, n, p, batch):
    """Disconnected members, isolated vertices, a last batch of any size."""
    check(nat, G.random_small(n, p, 6100 + n, connect=n % 2 == 0), batch=batch)


def test_mixed_light_and_heavy(nat):
    check(nat, G.rmat_lcc(10, 8))
    check(nat, G.barabasi_albert(900, 3, 61), np.array([5, 5, 899, 0, 17] * 60, np.int32))


def test_directed_and_options(nat):
    g = G.directed_random(500, 0.008, 6200)
    check(nat, g)
    check(nat, g, flags=nat.BC_KEEP_ORDER, batch=128)
    check(nat, g, flags=nat.BC_FORCE_BOTTOMUP)


def test_counts_past_16_bits(nat):
    """Levels whose counts need more than 16 bits, reached through light
    vertices (a 16 x 16 grid) and heavy ones (layered bicliques)."""
    check(nat, G.grid_graph(16))
    check(nat, G.layered_biclique(7, 12))


def test_deeper_than_the_level_capacity(nat):
    """The capacity grows and the launch starts over; accumulation is untouched by the first try."""
    g = G.path_graph(400)
    check(nat, g, batch=32)
    with nat.Graph.from_csr(g) as h:
        a, _, _ = run(nat, h, 5, np.arange(5, dtype=np.int32))
    with nat.Graph.from_csr(g) as h:
        h.run(np.arange(2, dtype=np.int32))
        h.run(np.arange(2, 5, dtype=np.int32), flags=nat.BC_ACCUMULATE)
        b, _, _ = h.result()
    assert np.all(np.abs(a - b) <= 2.0 ** -40 * np.abs(a))


def test_all_sources_after_a_subset(nat):
    """The staged list of every vertex is not mistaken for another one."""
    g = G.er_hamiltonian(400, 1200, 62)
    with nat.Graph.from_csr(g) as h:
        first, hs, _ = run(nat, h, g.n)
        run(nat, h, 40, np.arange(40, dtype=np.int32))
        h.forward_rows(np.arange(3, dtype=np.int32))
        second, ht, _ = run(nat, h, g.n)
        third, _, _ = run(nat, h, g.n, flags=nat.BC_KEEP_ORDER)
        fourth, hu, _ = run(nat, h, g.n)
    assert np.array_equal(first, second) and np.array_equal(first, fourth)
    for name in HASHES:
        assert np.array_equal(hs[name], ht[name]) and np.array_equal(hs[name], hu[name]), name
    assert np.allclose(first, third, rtol=1e-5, atol=1e-6 * g.n)


def test_per_level_form_on_a_large_mesh(nat):
    """More than 8192 vertices: lanes of launches per level, mostly light vertices."""
    g = G.grid_longrange(96, 0.05)
    g = G.Graph(g.n, g.row_ptr, g.col, None, "mesh96")
    check(nat, g, G.sample_sources(g.n, 700, 63))


@pytest.mark.parametrize("batch", [32, 64, 128, 256])
def test_many_graphs_around_the_pack_limit(nat, batch):
    """The many-graph kernel's packs: degrees at their limit of 16 arcs, mixed
    degrees, counts past 16 bits, an edgeless graph; BC and summaries per graph."""
    gs = [circulant(90 + deg, deg) for deg in (1, 2, 8, 15, 16, 17, 34)]
    gs += [G.barabasi_albert(300, 3, 64), G.grid_graph(16), G.csr_from_edges(40, [], []), G.star_graph(80),
           G.random_small(257, 0.03, 6300, connect=False)]
    hs = [nat.Graph.from_csr(g) for g in gs]
    with nat.ManyPlan(hs, batch=batch) as plan:
        for _ in range(2):
            plan.run()
            assert plan.result()[0] == nat.BC_OK
        for g, h in zip(gs, hs):
            ref = oracle.bc(g)
            got, _, _ = h.result()
            tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
            assert np.all(np.abs(got - ref["bc"]) <= tol), g.name
            sums = h.source_hashes(g.n)
            for name in HASHES:
                assert np.array_equal(sums[name], ref[name]), (g.name, name)
    for h in hs:
        h.close()
