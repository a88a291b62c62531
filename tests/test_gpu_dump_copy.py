"""corr_dump with a copy: the same sums in the copy and in the long integration, from the
current integration, from a deferred one, from neither, over sizes around the kernel's
rounds, and into a buffer that is only 8-byte aligned."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import _lib, api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("precision", ["int8", "fp32", "fp16"])
@pytest.mark.parametrize("n_in,n_chan", [(1, 1), (40, 3), (90, 7), (150, 120)])
@pytest.mark.parametrize("offset", [0, 1])
def test_dump_copies_the_long_integration(cuda_ok, precision, n_in, n_chan, offset):
    K = 16
    if precision == "int8":
        X = synth.chan_int8(n_chan, n_in, K, seed=n_in)
    else:
        X = synth.chan_sources(n_chan, n_in, K, n_src=1, seed=n_in)
    x = torch.from_numpy(X).to(DEV)
    c = api.Correlator(n_in, 1, n_chan, K, precision=precision)
    c.xengine(x)
    acc = c.accum().cpu().numpy()
    V = (acc[..., 0] + 1j * acc[..., 1]) if precision == "int8" else acc.astype(np.complex128)
    n = n_chan * c.n_base
    buf = torch.full((2 * n + 3,), -7.0, dtype=torch.float64, device=DEV)

    def dump():
        p = ctypes.c_void_p(buf.data_ptr() + 8 * offset)
        _lib.check(_lib.load().corr_dump(c.h, p, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)), "corr_dump")
        b = buf.cpu().numpy()
        assert np.all(b[:offset] == -7.0) and np.all(b[offset + 2 * n:] == -7.0)
        return b[offset:offset + 2 * n].view(np.complex128).reshape(n_chan, -1)

    assert np.array_equal(dump(), V)
    assert np.array_equal(dump(), V)          # nothing new
    c.xengine(x)
    c.dump(copy=False)                        # deferred on the tensor-core INT8 X-engine
    assert np.array_equal(dump(), V + V)
    c.xengine(x)
    c.dump(copy=False)
    c.xengine(x)
    assert np.array_equal(dump(), (V + V) + V + V)
    if precision == "int8":
        want = oracle.cmac(X)
        assert np.array_equal(V, want[..., 0] + 1j * want[..., 1])
    c.close()
