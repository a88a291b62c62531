"""Few-input X-engines (blocks of 4 x 4 inputs, K ranges per warp): INT8 exact against the
oracle over every load width (K a multiple of 8, even, odd), block count and K-range split,
stored and added, -128 included, AUTO and CUDA-core handles; more inputs than blocks of one
round; the planar handle (tensor cores) agrees."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("xengine", ["auto", "cudacore"])
@pytest.mark.parametrize("n_in,K,n_chan", [
    (1, 1, 2), (1, 5000, 1), (2, 8, 3), (3, 7, 2), (4, 1024, 2), (5, 2050, 1), (8, 1999, 1), (16, 96, 5), (17, 2048, 1),
    (20, 258, 2), (25, 33, 1), (29, 640, 2), (32, 4096, 1), (32, 31, 3), (33, 64, 2)])
def test_int8_few_inputs_exact(cuda_ok, xengine, n_in, K, n_chan):
    X = synth.chan_int8(n_chan, n_in, K, seed=n_in * K, sigma=60.0, lo=-128)
    X[0, -1] = -128
    V = oracle.cmac(X)
    c = api.Correlator(n_in, 1, n_chan, K, precision="int8", xengine=xengine)
    x = torch.from_numpy(X).to(DEV)
    c.xengine(x)
    assert np.array_equal(c.accum().cpu().numpy().astype(np.int64), V)
    c.xengine(x)
    assert np.array_equal(c.accum().cpu().numpy().astype(np.int64), 2 * V)
    c.dump(copy=False)
    c.xengine(x)
    vis = c.dump().cpu().numpy()
    assert np.array_equal(vis, 3 * (V[..., 0] + 1j * V[..., 1]))
    c.check_status()
    c.close()


@pytest.mark.parametrize("n_in,K,n_chan", [(23, 600, 2), (27, 1031, 1), (31, 64, 3), (32, 2048, 1)])
def test_fp32_up_to_32_inputs(cuda_ok, n_in, K, n_chan):
    X = synth.chan_sources(n_chan, n_in, K, n_src=2, seed=n_in)
    ref = oracle.cmac(X)
    c = api.Correlator(n_in, 1, n_chan, K)
    c.xengine(torch.from_numpy(X).to(DEV))
    V = c.accum().cpu().numpy()
    i, j = oracle.tri_pairs(n_in)
    aut = np.abs(ref[..., oracle.packed_index(np.arange(n_in), np.arange(n_in))])
    assert np.max(np.abs(V - ref) / np.sqrt(aut[..., i] * aut[..., j])) <= 1e-5
    c.close()
