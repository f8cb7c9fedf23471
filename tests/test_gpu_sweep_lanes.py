"""The launch-per-level form of the unweighted sweep on several concurrent
lanes, on graphs that the one-launch form does not take (its rule counts the
items per warp, one_launch in bc_api.cu) and on small ones kept off it by a
device wait bound: light vertices in full packs, capacity growth under way on
other lanes, directed sinks beside full rows. Which form ran is told by the
number of launches."""
import numpy as np
import pytest

import oracle
from paper_0809_1906_gb300 import graphs as G

pytestmark = pytest.mark.gpu

HASHES = ("hash_sigma", "hash_dist", "dist_sum", "reach")
KEEP_OFF = 10_000_000  # device_wait_us that no wait comes near


@pytest.fixture(scope="module")
def nat():
    from paper_0809_1906_gb300 import native
    native.load()
    return native


def check(nat, g, src, batch, levels, **kw):
    """levels: a lower bound on the launches of one batch; 0 for the one-launch
    form. Where counts pass 2^64 (the oracle says), BC is not a number to compare."""
    ref = oracle.bc(g, src) if src is not None else oracle.bc(g)
    k = g.n if src is None else len(src)
    wraps = bool(ref["flags"] & 1)
    outs = []
    with nat.Graph.from_csr(g) as h:
        for _ in range(2):  # the second run starts with the capacity that the first one reached
            h.run(src, batch=batch, **kw)
            got, code, st = h.result()
            assert code == (nat.BC_WARN_SIGMA_OVERFLOW if wraps else nat.BC_OK) and st == int(wraps)
            hs = h.source_hashes(k)
            for name in HASHES:
                assert np.array_equal(hs[name], ref[name]), name
            assert h.run_stats()[0] == int(ref["arcs"].sum())
            tol = np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)
            assert wraps or np.all(np.abs(got - ref["bc"]) <= tol), float(np.max(np.abs(got - ref["bc"])))
            assert (h.launch_count() > levels * (k // batch)) if levels else (h.launch_count() <= 4)
            outs.append(got)
    assert np.array_equal(outs[0], outs[1], equal_nan=wraps)


@pytest.mark.parametrize("batch,sources", [(32, 250), (64, 640), (256, 1900)])
def test_large_grid_on_many_lanes(nat, batch, sources):
    """16,384 vertices of two to four arcs, 150 levels and more from any source
    (the capacity starts at 32), the last batch ragged."""
    g = G.grid_graph(128)
    check(nat, g, G.sample_sources(g.n, sources, 63), batch, 150)


@pytest.mark.parametrize("batch,sources", [(32, 250), (256, 1900)])
@pytest.mark.parametrize("kind", ["comb", "mesh"])
def test_large_light_graphs_on_many_lanes(nat, kind, batch, sources):
    """The same size without counts past 2^64: a comb (a path of 128 vertices,
    each with a path of 127 hung on, up to 380 levels) and a mesh with long edges."""
    if kind == "comb":
        at = np.arange(16384)
        tooth = at[at % 128 != 0]
        spine = at[(at % 128 == 0) & (at > 0)]
        g = G.csr_from_edges(16384, np.concatenate([tooth - 1, spine - 128]), np.concatenate([tooth, spine]), name=kind)
    else:
        g = G.grid_longrange(128, 0.05)
        g = G.Graph(g.n, g.row_ptr, g.col, None, kind)
    check(nat, g, G.sample_sources(g.n, sources, 63), batch, 120 if kind == "comb" else 15)


@pytest.mark.parametrize("g,src,levels", [
    (G.path_graph(300), None, 150),
    (G.random_small(700, 0.004, 64, connect=False), None, 2),
    (G.grid_longrange(30, 0.05), np.array([5, 5, 899, 0, 17] * 60, np.int32), 5),
    (G.barabasi_albert(900, 3, 61), None, 2),
], ids=["path", "random", "mesh", "attachment"])
def test_small_graphs_kept_off_one_launch(nat, g, src, levels):
    g = G.Graph(g.n, g.row_ptr, g.col, None, g.name)
    check(nat, g, src, 32, levels, device_wait_us=KEEP_OFF)


def eights_and_sinks(eights, sinks, seed):
    """Vertices of exactly eight arcs out, to any vertex, and vertices of none."""
    n = eights + sinks
    rng = np.random.default_rng(seed)
    u, v = [], []
    for x in range(eights):
        heads = rng.choice(n - 1, 8, replace=False)
        u.append(np.full(8, x))
        v.append(heads + (heads >= x))
    return G.csr_from_arcs(n, np.concatenate(u), np.concatenate(v), name="eights+sinks")


@pytest.mark.parametrize("eights,sinks", [(3001, 2999), (5996, 4), (204, 5796)])
@pytest.mark.parametrize("keep_off", [0, KEEP_OFF])
def test_sinks_behind_full_packs(nat, eights, sinks, keep_off):
    """Packs filled by four vertices of eight arcs with vertices of no arcs
    behind them in the same group (a warp's share is 13 or more here)."""
    g = eights_and_sinks(eights, sinks, 65)
    check(nat, g, np.arange(0, g.n, 12, dtype=np.int32), 32, 2 if keep_off else 0, device_wait_us=keep_off)


@pytest.mark.parametrize("scale,sources,keep,lanes", [(13, 257, False, True), (13, 300, False, False),
                                                      (13, 2304, False, True), (12, 2304, False, False),
                                                      (13, 2600, True, True), (12, 900, True, False)])
def test_uneven_and_spread_batches_take_the_lanes(nat, scale, sources, keep, lanes):
    """Which form runs when one batch holds all but a sliver of the sources, the
    groups' last round is nearly empty, or the caller's order is kept, on both
    sides of the line; either form gives the oracle's values."""
    g = G.rmat_lcc(scale, 16)
    check(nat, g, G.sample_sources(g.n, sources, 66), 256, 2 if lanes else 0, flags=nat.BC_KEEP_ORDER if keep else 0)
