"""Deferred dumps of every size around the line between fixed shares for each CTA's idle
warps and chunks claimed by all of the launch: the long integration holds the exact sums."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu


# 2048 visibilities per CTA is the line: 63 and 64 inputs have 2016 and 2080 per channel
@pytest.mark.parametrize("precision", ["int8", "fp16_hilo"])
@pytest.mark.parametrize("n_in,n_chan", [(1, 1), (3, 1), (22, 1), (23, 1), (63, 1), (64, 1), (63, 16), (64, 16), (90, 3),
                                         (20, 160), (150, 2)])
def test_sums_after_deferred_dumps(cuda_ok, precision, n_in, n_chan):
    K = 40
    X = [synth.chan_int8(n_chan, n_in, K, seed=s + n_in) for s in (1, 2, 3)]
    V = sum(oracle.cmac(x).astype(np.float64) for x in X)
    c = api.Correlator(n_in, 1, n_chan, K, precision=precision, xengine="tcgen05")
    for x in X:
        t = torch.from_numpy(x).cuda()
        c.xengine(t if precision == "int8" else torch.view_as_complex(t.float()))
        c.dump(copy=False)
    assert np.array_equal(c.dump().cpu().numpy(), V[..., 0] + 1j * V[..., 1])
    c.check_status()
    c.close()
