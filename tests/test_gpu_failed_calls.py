"""What a call leaves behind when it fails, and what the next one then gives:
waits that run out, on the host and on the device, by limits that the caller
sets. Nothing here faults or hangs the GPU; every wait is bounded."""
import ctypes
import time

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


def close(got, ref, n):
    return np.all(np.abs(got - ref) <= np.maximum(1e-5 * np.abs(ref), 1e-6 * n))


def test_rows_left_unwritten_after_a_failed_call(nat):
    """Rows go straight into the caller's device memory, from several internal
    streams. A call whose host wait runs out (1 ms, with the stream held for some
    20) must have ended on all of them when it returns: the caller may free or
    refill the buffers. The first batch's sources are isolated, so the caller's own
    stream is done early; the second one's second level takes longer (24
    hubs, each joined to every one of 400,000 vertices)."""
    import torch
    leaves, hubs, alone = 400_000, 24, 256
    n = leaves + hubs + alone
    g = G.csr_from_edges(n, np.tile(np.arange(leaves), hubs), np.repeat(leaves + np.arange(hubs), leaves), name="hubs")
    src = np.concatenate([leaves + hubs + np.arange(alone), np.arange(256)]).astype(np.int32)
    sig = torch.zeros((512, n), dtype=torch.int64, device="cuda")
    dist = torch.zeros((512, n), dtype=torch.int32, device="cuda")

    def rows(h, wait_ms):
        opt = nat.make_options(256, 0, 0, wait_ms)
        return h.lib.bc_forward_rows(h.handle, nat._addr(src), len(src), nat._addr(sig), nat._addr(dist),
                                     ctypes.byref(opt), nat._stream_ptr(stream))

    stream = torch.cuda.Stream()
    left = []
    with nat.Graph.from_csr(g, trust_input=True) as h:
        assert rows(h, 0) == nat.BC_OK  # plans and state are in place: the next calls only launch
        for _ in range(3):  # the least of three: a held-up host thread is no failure
            torch.cuda.synchronize()
            with torch.cuda.stream(stream):
                torch.cuda._sleep(40_000_000)
            code = rows(h, 1)
            t0 = time.perf_counter()
            torch.cuda.synchronize()
            left.append(time.perf_counter() - t0)
            assert code == nat.BC_ERR_TIMEOUT
        sig.zero_(), dist.zero_()
        torch.cuda.synchronize()
        assert rows(h, 0) == nat.BC_OK
    # an idle device answers in some 30 us; the level in flight left 680 us
    assert min(left) < 2.5e-4, left
    for i in (0, 255, 256, 511):
        o = oracle.source(g, int(src[i]), with_delta=False)
        assert np.array_equal(sig[i].cpu().numpy().view(np.uint64), o["sigma"])
        assert np.array_equal(dist[i].cpu().numpy(), o["dist"].astype(np.int32))


@pytest.mark.parametrize("g", [G.er_hamiltonian(400, 1600, 81), G.star_graph(700)], ids=lambda g: g.name)
def test_barrier_expiry_spoils_no_sum(nat, g):
    """A barrier of the one-launch form whose last arrival never comes gives up
    after 2 ms: bc_result reports the timeout, the sums of the runs before stay
    as they were (halving included), and the next runs on the handle, in either
    form, are right. The star's hub is split into items that meet at counters."""
    ref = oracle.bc(g)["bc"]
    with nat.Graph.from_csr(g) as h:
        h.run()
        first, code, _ = h.result()
        assert code == nat.BC_OK and close(first, ref, g.n)
        h.run(flags=nat.BC_ACCUMULATE | nat.BC_HALVE | nat.BC_TEST_BARRIER_EXPIRY, device_wait_us=2000)
        with pytest.raises(nat.BcError) as e:
            h.result()
        assert e.value.code == nat.BC_ERR_TIMEOUT
        for flags in (0, nat.BC_TIMING):
            h.run(flags=nat.BC_ACCUMULATE | nat.BC_TEST_BARRIER_EXPIRY, device_wait_us=2000)
            h.run(flags=nat.BC_ACCUMULATE | flags)
            got, code, st = h.result()
            assert code == nat.BC_OK and st == 0
            first = first + ref
            assert close(got, first, 3 * g.n)


def test_wait_limit_is_per_batch(nat):
    """1250 batches in one launch take several times the host's wait limit, each
    of them a fraction of it: the run is not cut short."""
    import torch
    g = G.er_hamiltonian(2000, 8000, 82)
    src = np.tile(np.arange(g.n, dtype=np.int32), 20)
    ref = 20.0 * oracle.bc(g)["bc"]
    with nat.Graph.from_csr(g) as h:
        h.run(src, batch=32)
        h.result()
        t0 = time.perf_counter()
        h.run(src, batch=32)
        h.result()
        whole = 1e3 * (time.perf_counter() - t0)
        assert whole > 15.0, whole  # else the limit below says nothing
        h.run(src, batch=32, wait_limit_ms=4)
        got, code, _ = h.result()
    assert code == nat.BC_OK and close(got, ref, 20 * g.n)


def test_run_returns_before_the_backward_pass_ends(nat):
    """bc_run waits for the forward passes alone: on a path of 1500 levels the
    backward pass, as long again, is still under way when it returns."""
    import torch
    g = G.path_graph(1500)
    src = np.arange(32, dtype=np.int32)
    with nat.Graph.from_csr(g) as h:
        h.run(src, batch=32)
        h.result()
        running = []
        for _ in range(3):  # one of three: the host thread may be held up between the two
            h.run(src, batch=32)
            time.sleep(3e-4)
            running.append(not torch.cuda.current_stream().query())
            got, code, _ = h.result()
            assert code == nat.BC_OK and close(got, oracle.bc(g, src)["bc"], g.n)
    assert any(running)


def test_out_of_memory_leaves_the_handle_usable(nat):
    """A path of three million vertices needs more level capacity than the GPU
    holds: the run reports that it is out of memory, and so does the next one
    (it must not take the half-grown state for a whole one); sources of a small
    component beside it then run on the same handle."""
    n, k = 3_000_000, 5
    at = np.arange(n - 1)
    g = G.csr_from_edges(n + k, np.concatenate([at, n + np.arange(k - 1)]), np.concatenate([at + 1, n + 1 + np.arange(k - 1)]),
                         name="paths")
    src = n + np.arange(k, dtype=np.int32)
    ref = oracle.bc(G.path_graph(k))["bc"]
    with nat.Graph.from_csr(g, trust_input=True) as h:
        for _ in range(2):
            with pytest.raises(nat.BcError) as e:
                h.run(np.array([0], np.int32))
            assert e.value.code == nat.BC_ERR_OOM
        h.run(src)
        got, code, st = h.result()
        assert code == nat.BC_OK and st == 0
    assert np.all(got[:n] == 0.0) and close(got[n:], ref, k)
    nat.release_cached_memory()
