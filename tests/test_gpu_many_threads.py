"""The many-graph kernel's CTA sizes: sets of thousands of tiny graphs, of some
hundred vertices each, and just below the counts from which those sizes are
used; BC and summaries of every graph against the oracle."""
import numpy as np
import pytest

import oracle
from paper_0809_1906_gb300 import graphs as G

pytestmark = pytest.mark.gpu

HASHES = ("hash_sigma", "hash_dist", "dist_sum", "reach")


@pytest.fixture(scope="module")
def nat():
    from paper_0809_1906_gb300 import native
    native.load()
    return native


def members(count, lo, hi):
    """`count` handles over a few dozen distinct graphs of lo to hi vertices, stars and an edgeless one among them."""
    gs = G.many_graphs(24, lo, hi, seed=67) + [G.star_graph(hi), G.csr_from_edges(lo, [], []), G.path_graph(min(hi, 60))]
    return [gs[i % len(gs)] for i in range(count)]


# 8 and 4 CTAs per SM of 152 are 1216 and 608 batches
@pytest.mark.parametrize("count,lo,hi,batch", [
    (1300, 10, 64, 32), (1300, 10, 64, 256), (1215, 10, 32, 64), (1300, 10, 65, 128),
    (320, 70, 256, 32), (700, 70, 200, 64), (320, 70, 257, 32)])
def test_sets_of_small_graphs(nat, count, lo, hi, batch):
    gs = members(count, lo, hi)
    refs = {id(g): oracle.bc(g) for g in gs}
    hs = [nat.Graph.from_csr(g, trust_input=True) for g in gs]
    try:
        with nat.ManyPlan(hs, batch=batch) as plan:
            plan.run()
            assert plan.result()[0] == nat.BC_OK
            for g, h in zip(gs, hs):
                ref = refs[id(g)]
                got, _, _ = h.result()
                assert np.all(np.abs(got - ref["bc"]) <= np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n)), g.name
                sums = h.source_hashes(g.n)
                for name in HASHES:
                    assert np.array_equal(sums[name], ref[name]), (g.name, name)
    finally:
        for h in hs:
            h.close()
