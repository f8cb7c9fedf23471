"""Runs on a stream that has a part of the GPU's SMs (a green context of the
CUDA driver): the one-launch form needs its blocks resident together and is
left for the launches per level."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_0809_1906_gb300 import graphs as G

pytestmark = pytest.mark.gpu

CU_DEV_RESOURCE_TYPE_SM = 1
CU_GREEN_CTX_DEFAULT_STREAM = 1
CU_STREAM_NON_BLOCKING = 1


@pytest.fixture(scope="module")
def nat():
    from paper_0809_1906_gb300 import native
    native.load()
    return native


@pytest.fixture()
def part_stream(nat):
    """A stream with 16 SMs or a little more, or a skip where the driver has no such contexts."""
    import torch
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    if not hasattr(cu, "cuGreenCtxStreamCreate"):
        pytest.skip("no green contexts")
    dev = ctypes.c_int(0)
    every, part = ctypes.create_string_buffer(1024), ctypes.create_string_buffer(1024)
    groups, desc, ctx, stream = ctypes.c_uint(1), ctypes.c_void_p(), ctypes.c_void_p(), ctypes.c_void_p()
    if cu.cuDeviceGetDevResource(dev, every, CU_DEV_RESOURCE_TYPE_SM) != 0 \
            or cu.cuDevSmResourceSplitByCount(part, ctypes.byref(groups), every, None, 0, 16) != 0 \
            or cu.cuDevResourceGenerateDesc(ctypes.byref(desc), part, 1) != 0 \
            or cu.cuGreenCtxCreate(ctypes.byref(ctx), desc, dev, CU_GREEN_CTX_DEFAULT_STREAM) != 0:
        pytest.skip("the driver gives no green context here")
    assert cu.cuGreenCtxStreamCreate(ctypes.byref(stream), ctx, CU_STREAM_NON_BLOCKING, 0) == 0
    yield stream.value
    torch.cuda.synchronize()
    cu.cuStreamDestroy_v2(stream)
    cu.cuGreenCtxDestroy(ctx)


def test_small_run_on_a_part_of_the_device(nat, part_stream):
    g = G.er_hamiltonian(400, 1600, 95)
    ref = oracle.bc(g)
    with nat.Graph.from_csr(g) as h:
        for stream, one in ((part_stream, False), (None, True)):
            h.run(stream=stream)
            got, code, st = h.result()
            assert code == nat.BC_OK and st == 0
            assert np.all(np.abs(got - ref["bc"]) <= np.maximum(1e-5 * np.abs(ref["bc"]), 1e-6 * g.n))
            assert np.array_equal(h.source_hashes(g.n)["hash_sigma"], ref["hash_sigma"])
            assert (h.launch_count() <= 4) == one
