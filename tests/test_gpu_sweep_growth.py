"""The level capacity that grows in the middle of a run: batches that ended
before keep their results, whichever form runs them."""
import time

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


def random_and_path(n, m, tail, seed):
    """G(n, m) and a path of `tail` vertices beside it."""
    u, v, _ = G.er_hamiltonian(n, m, seed).edges()
    at = n + np.arange(tail - 1)
    return G.csr_from_edges(n + tail, np.concatenate([u, at]), np.concatenate([v, at + 1]), name="random+path")


@pytest.mark.parametrize("batch,first_deep", [(32, False), (64, True), (256, False)])
def test_batches_before_and_after_the_growth(nat, batch, first_deep):
    """Shallow batches, deep ones of 40, 90 and 300 levels among them, counted
    and added once each: summaries, arcs and BC against the oracle."""
    g = random_and_path(900, 2700, 301, 91)
    deep = np.array([900, 900 + 210, 900 + 260, 1200], np.int32)
    src = np.arange(900, dtype=np.int32)
    at = 0 if first_deep else 500
    src = np.concatenate([src[:at], deep, src[at:]])
    ref = oracle.bc(g, src)
    with nat.Graph.from_csr(g) as h:
        outs = []
        for flags in (nat.BC_KEEP_ORDER, nat.BC_KEEP_ORDER, 0):
            h.run(src, batch=batch, flags=flags)
            got, code, st = h.result()
            assert code == nat.BC_OK and st == 0
            hs = h.source_hashes(len(src))
            for name in HASHES:
                assert np.array_equal(hs[name], ref[name]), name
            assert h.run_stats()[0] == int(ref["arcs"].sum())
            assert np.all(np.abs(got - ref["bc"]) <= np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n))
            outs.append(got)
    assert np.array_equal(outs[0], outs[1])  # grown on the way or grown before: the same sums


def test_growth_does_not_repeat_finished_batches(nat):
    """One deep source among 90,000 shallow ones, five doublings of the capacity:
    the first run of a handle costs the aborted tries of the deep batch and the
    growth itself (10 ms allowed) beyond a run at full capacity, not the other
    batches five times more."""
    import torch
    g = random_and_path(2500, 7500, 1000, 92)
    src = np.concatenate([np.tile(np.arange(2500, dtype=np.int32), 36), [2500]]).astype(np.int32)

    def timed(h):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        h.run(src, batch=32)
        h.result()
        return time.perf_counter() - t0

    firsts, steady = [], []
    for _ in range(3):  # the first handle also fills the pools of lanes and device blocks
        with nat.Graph.from_csr(g) as h:
            firsts.append(timed(h))
            steady += [timed(h), timed(h)]
    assert min(firsts) < 2.0 * min(steady) + 0.010, (firsts, steady)
