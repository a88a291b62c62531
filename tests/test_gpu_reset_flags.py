"""corr_reset clears only what is not known to be clear: every order of resets, dumps,
restores and X-engine calls leaves the sums that cleared memory would give (exact
integers), also where the calls are replayed from a CUDA graph."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _complex(V):
    return V[..., 0] + 1j * V[..., 1]


@pytest.mark.parametrize("kw", [dict(precision="int8"), dict(precision="int8", fused_dump=True),
                                dict(precision="int8", xengine="cudacore")])
def test_reset_after_every_use(cuda_ok, kw):
    n_in, K, n_chan = 40, 64, 2
    X = synth.chan_int8(n_chan, n_in, K, seed=3)
    V = _complex(oracle.cmac(X))
    x = torch.from_numpy(X).to(DEV)
    c = api.Correlator(n_in, 1, n_chan, K, **kw)
    vis = lambda: c.dump().cpu().numpy()  # noqa: E731
    c.reset()
    c.reset()
    assert not vis().any()
    c.xengine(x)
    c.dump(copy=False)          # deferred, added or fused
    c.reset()                   # a pending dump is dropped, a finished one cleared
    assert not vis().any()
    c.xengine(x)
    assert np.array_equal(vis(), V)
    c.xengine(x)
    c.dump(copy=False)
    c.xengine(x)                # carries the deferred dump of the call before
    c.reset()
    assert not vis().any()
    c.xengine(x)
    c.dump(copy=False)
    c.flush()
    c.reset()
    c.xengine(x)
    assert np.array_equal(vis(), V)
    c.reset()
    c.restore_vis(torch.from_numpy(3 * V).to(DEV))
    c.xengine(x)
    assert np.array_equal(vis(), 4 * V)
    c.reset()
    assert not vis().any()
    c.close()


def test_reset_with_replayed_calls(cuda_ok):
    """A graph's replays add to the long integration behind the handle's back: a reset
    after them still clears it."""
    n_in, K, n_chan = 24, 32, 2
    X = synth.chan_sources(n_chan, n_in, K, n_src=1, seed=5)
    x = torch.from_numpy(X).to(DEV)
    c = api.Correlator(n_in, 1, n_chan, K, precision="fp32")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        c.xengine(x)
        c.dump(copy=False)
        c.reset()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            c.xengine(x)
            c.dump(copy=False)
        c.reset()
        g.replay()
        g.replay()
        twice = c.dump().clone()
        c.reset()
        none = c.dump().clone()
        g.replay()
        once = c.dump().clone()
    torch.cuda.synchronize()
    assert not none.cpu().numpy().any()
    assert np.array_equal(twice.cpu().numpy(), 2 * once.cpu().numpy()) and once.abs().max() > 0
    c.close()
