"""Handles used by several kinds of calls in turn: what one call leaves in a
handle must not be taken for another's, nor a plan write where a handle's
results no longer are."""
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


def close(got, ref, n):
    return np.all(np.abs(got - ref) <= np.maximum(1e-5 * np.abs(ref), 1e-6 * n))


def test_plan_follows_its_handles_summaries(nat):
    """A run of one handle with three sources per vertex (repeats are allowed)
    needs longer summaries and moves them; the plan's next run writes to where
    they are now."""
    gs = [G.er_hamiltonian(120, 300, 71), G.barabasi_albert(90, 3, 72), G.csr_from_edges(30, [], [])]
    refs = [oracle.bc(g) for g in gs]
    hs = [nat.Graph.from_csr(g) for g in gs]
    with nat.ManyPlan(hs, batch=64) as plan:
        for rep in range(3):
            plan.run()
            assert plan.result()[0] == nat.BC_OK
            for g, h, ref in zip(gs, hs, refs):
                got, _, _ = h.result()
                assert close(got, ref["bc"], g.n), (rep, g.name)
                sums = h.source_hashes(g.n)
                for name in HASHES:
                    assert np.array_equal(sums[name], ref[name]), (rep, g.name, name)
            g, h = gs[rep], hs[rep]
            src = np.tile(np.arange(g.n, dtype=np.int32), 3)
            h.run(src)
            sums = h.source_hashes(len(src))
            for name in HASHES:
                assert np.array_equal(sums[name], np.tile(refs[rep][name], 3)), (rep, name)
    for h in hs:
        h.close()


def test_result_survives_rows_after_a_failed_run(nat):
    """A run that fails before it cleared the handle's BC leaves nothing to be
    cleared later: rows asked of the handle after a plan has given it its result
    leave that result alone."""
    import torch
    g = G.er_hamiltonian(400, 1600, 73)
    ref = oracle.bc(g)
    with nat.Graph.from_csr(g) as h:
        stream = torch.cuda.Stream()
        h.run(flags=nat.BC_KEEP_ORDER, stream=stream)  # state and sources in place: the next run only waits
        h.result()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)  # some 50 ms: the run's own work starts after it
        with pytest.raises(nat.BcError) as e:
            h.run(flags=nat.BC_KEEP_ORDER, wait_limit_ms=1, stream=stream)
        assert e.value.code == nat.BC_ERR_TIMEOUT
        torch.cuda.synchronize()
        with nat.ManyPlan([h], batch=64) as plan:
            plan.run()
            assert plan.result()[0] == nat.BC_OK
            h.forward_rows(np.arange(3, dtype=np.int32), batch=64)
            got, _, _ = h.result()
            assert close(got, ref["bc"], g.n)


@pytest.mark.parametrize("first,second", [((32, 8), (32, 0)), ((256, 4), (64, 16)), ((64, 0), (32, 8))])
def test_next_run_waits_for_the_last_ones_plan_and_state(nat, first, second):
    """Runs one after another on a stream of its own, none of them waited for:
    the next one, with other work items and another width, replaces plans and
    counters only after the backward pass before it (a long path hung on a hub of
    split items) has read them."""
    import torch
    at = np.arange(1200)
    spokes = 1200 + np.arange(900)
    g = G.csr_from_edges(2100, np.concatenate([at[:-1], np.zeros(900, np.int64)]), np.concatenate([at[1:], spokes]),
                         name="path+hub")
    src = np.concatenate([np.arange(0, 1200, 50), spokes[:8]]).astype(np.int32)
    ref = oracle.bc(g, src)["bc"]
    stream = torch.cuda.Stream()
    with nat.Graph.from_csr(g) as h:
        for batch, chunk in (first, second):  # the level capacity and both plans' room are there afterwards
            h.run(src, batch=batch, chunk=chunk, stream=stream)
            h.result()
        for rep in range(3):
            h.run(src, batch=first[0], chunk=first[1], stream=stream)
            h.run(src, batch=second[0], chunk=second[1], stream=stream, flags=nat.BC_ACCUMULATE)
            h.run(src, batch=first[0], chunk=first[1], stream=stream, flags=nat.BC_ACCUMULATE)
            got, code, st = h.result()
            assert code == nat.BC_OK and st == 0
            assert close(got, 3.0 * ref, 3 * g.n), rep
