"""AUTO's choice of the INT8 X-engine for few inputs in the complex int8 layout: on the CUDA
cores (no conversion pass) where that measured faster, else on the tensor cores; the exact
sums on both sides of every line."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,K,cudacore", [
    (32, 4000, True), (33, 8, False), (28, 4002, True), (29, 1000, True), (29, 1002, False), (32, 4, True),
    (32, 1004, False), (16, 4001, True), (17, 1499, True), (17, 1501, False), (20, 1499, True), (20, 1501, False),
    (21, 499, True), (21, 501, False), (24, 499, True), (24, 1001, False), (25, 33, False)])
def test_route_and_sums(cuda_ok, n_in, K, cudacore):
    X = synth.chan_int8(2, n_in, K, seed=K + n_in, lo=-128)
    c = api.Correlator(n_in, 1, 2, K, precision="int8")
    c.set_stage_timing(True)
    c.xengine(torch.from_numpy(X).cuda())
    assert np.array_equal(c.accum().cpu().numpy().astype(np.int64), oracle.cmac(X))
    assert c.stage_times()["prep"][1] == (0 if cudacore else 1)
    c.close()
