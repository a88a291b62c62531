"""corr_dump's copy of the long integration: stored by the dump kernel only where it lies in
the handle's device's own memory; other memory that a copy reaches (another device's; here
page-locked host memory, to need one device only) is written by a copy, as it always was."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import _lib, api

pytestmark = pytest.mark.gpu
KERNEL, MEMCPY = 0, 1  # CUgraphNodeType


def _recorded(stream, fn):
    """Kinds of graph nodes that fn leaves when it is recorded (nothing runs)."""
    cu = ctypes.CDLL("libcuda.so.1")
    s, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert cu.cuStreamBeginCapture_v2(s, 1) == 0
    try:
        fn()
    finally:
        assert cu.cuStreamEndCapture(s, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kinds = []
    for node in nodes:
        t = ctypes.c_int()
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(t)) == 0
        kinds.append(t.value)
    assert cu.cuGraphDestroy(graph) == 0
    return sorted(kinds)


@pytest.mark.parametrize("deferred", [False, True])
def test_only_memory_of_the_device_is_stored_to(cuda_ok, deferred):
    n_in, K, n_chan = 40, 64, 3
    X = synth.chan_int8(n_chan, n_in, K, seed=7)
    v = oracle.cmac(X)
    V = v[..., 0] + 1j * v[..., 1]
    x = torch.from_numpy(X).cuda()
    host = torch.zeros(V.shape, dtype=torch.complex128, pin_memory=True)
    dev = torch.zeros(V.shape, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    c = api.Correlator(n_in, 1, n_chan, K, precision="int8")

    def dump(out):
        _lib.check(_lib.load().corr_dump(c.h, out.data_ptr(), stream.cuda_stream), "corr_dump")

    with torch.cuda.stream(stream):
        for n, out in enumerate((host, dev), 1):
            c.xengine(x)
            if deferred:
                c.dump(copy=False)
            dump(out)
            stream.synchronize()
            assert np.array_equal(out.cpu().numpy(), n * V)
        c.xengine(x)
        assert _recorded(stream, lambda: dump(dev)) == [KERNEL]
        c.xengine(x)
        assert _recorded(stream, lambda: dump(host)) == [KERNEL, MEMCPY]
    c.close()
