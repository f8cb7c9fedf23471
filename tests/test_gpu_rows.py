"""Forward rows written straight into device buffers (bc_forward_rows): the
32 x 32 tiles at ragged vertex and source counts, one output alone, and a
buffer that the kernels cannot write (misaligned), all against the oracle."""
import numpy as np
import pytest

import oracle
from paper_0809_1906_gb300 import graphs as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0809_1906_gb300 import native
    native.load()
    return native


def rows(nat, h, src, n, batch, want_sigma=True, want_dist=True, shift=0):
    import ctypes

    import torch
    k = len(src)
    sig = torch.full((k * n + 1,), -7, dtype=torch.int64, device="cuda")
    dist = torch.full((k * n + 2,), -7, dtype=torch.int32, device="cuda")
    opt = nat.make_options(batch)
    code = h.lib.bc_forward_rows(h.handle, nat._addr(src), k, sig.data_ptr() + shift if want_sigma else None,
                                 dist.data_ptr() + shift if want_dist else None, ctypes.byref(opt),
                                 torch.cuda.current_stream().cuda_stream)
    assert code == nat.BC_OK
    s = sig.cpu().numpy().view(np.uint8)[shift:shift + 8 * k * n].view(np.uint64)
    d = dist.cpu().numpy().view(np.uint8)[shift:shift + 4 * k * n].copy().view(np.int32)
    return s.reshape(k, n), d.reshape(k, n)


@pytest.mark.parametrize("n,k,batch", [(1, 1, 32), (31, 31, 32), (33, 33, 64), (301, 200, 256), (1000, 257, 256)])
def test_device_rows(nat, n, k, batch):
    g = G.random_small(n, min(1.0, 3.0 / n), 3100 + n, connect=n % 2 == 0) if n > 1 else G.csr_from_edges(1, [], [])
    src = G.sample_sources(n, k, 5)
    with nat.Graph.from_csr(g) as h:
        hs, hd, _ = h.forward_rows(src, batch=batch)  # host buffers
        s, d = rows(nat, h, src, n, batch)
        assert np.array_equal(s, hs) and np.array_equal(d, hd)
        s, _ = rows(nat, h, src, n, batch, want_dist=False)
        assert np.array_equal(s, hs)
        _, d = rows(nat, h, src, n, batch, want_sigma=False)
        assert np.array_equal(d, hd)
    ref = oracle.bc(g, src)
    ids = np.arange(1, n + 1, dtype=np.uint64)
    assert np.array_equal((hs * ids).sum(1, dtype=np.uint64), ref["hash_sigma"])
    assert np.array_equal(np.where(hd >= 0, (hd + 1).astype(np.uint64) * ids, 0).sum(1, dtype=np.uint64),
                          ref["hash_dist"])


def test_misaligned_device_rows(nat):
    """4-byte aligned uint64 rows (and 4 bytes into the int32 buffer) still arrive whole."""
    g = G.er_hamiltonian(200, 600, 3)
    src = G.sample_sources(200, 40, 6)
    with nat.Graph.from_csr(g) as h:
        hs, hd, _ = h.forward_rows(src, batch=64)
        s, d = rows(nat, h, src, 200, 64, shift=4)
    assert np.array_equal(s, hs) and np.array_equal(d, hd)


def test_deep_rows(nat):
    """Distances that need many bit planes (a path of 700 vertices)."""
    g = G.path_graph(700)
    src = np.array([0, 350, 699], np.int32)
    with nat.Graph.from_csr(g) as h:
        s, d = rows(nat, h, src, 700, 32)
    assert np.array_equal(d, np.abs(np.arange(700)[None, :] - src[:, None]))
    assert np.all(s == 1)
