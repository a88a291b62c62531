"""Operand passes at every alignment of their rows: the conversion of complex int8 rows of
any length for the tensor-core X-engine, and the adjoint's scale exponents for gradients
that start between two 16-byte boundaries, wherever the largest entry lies."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


# row lengths of every residue modulo 8, short, and past one chunk of 8 spectra per lane
@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 10, 12, 14, 20, 30, 33, 100, 250, 1006])
@pytest.mark.parametrize("n_in,xengine", [(21, "tcgen05"), (40, "auto")])
def test_int8_rows_on_the_tensor_cores(cuda_ok, K, n_in, xengine):
    n_chan = 3
    X = synth.chan_int8(n_chan, n_in, K, seed=K, lo=-128)
    c = api.Correlator(n_in, 1, n_chan, K, precision="int8", xengine=xengine)
    c.set_stage_timing(True)
    c.xengine(torch.from_numpy(X).to(DEV))
    assert np.array_equal(c.accum().cpu().numpy().astype(np.int64), oracle.cmac(X))
    assert c.stage_times()["prep"][1] == 1  # by way of the conversion
    c.close()


@pytest.mark.parametrize("n_in", [8, 40])
@pytest.mark.parametrize("where", [0, 1, 2, -2, -1])
def test_adjoint_of_unaligned_gradients(cuda_ok, n_in, where):
    K, n_chan = 16, 3
    B = n_in * (n_in + 1) // 2
    rng = np.random.default_rng(n_in)

    def cplx(*shape):
        return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)

    x, g, G = cplx(n_chan, n_in, K), cplx(n_in), cplx(n_chan, B)
    G[:, where] *= 3000          # sets the channel's scale: missed, FP16 would overflow
    c = api.Correlator(n_in, 1, n_chan, K, precision="fp16_hilo")
    xd, gd = torch.from_numpy(x).to(DEV), torch.from_numpy(g).to(DEV)
    buf = torch.zeros(n_chan * B + 2, dtype=torch.complex64, device=DEV)
    got = []
    for off in (0, 1):           # the buffer is 16-byte aligned, entries take 8 bytes
        part = buf[off:off + n_chan * B].view(n_chan, B)
        part.copy_(torch.from_numpy(G))
        assert part.data_ptr() % 16 == 8 * off
        got.append([t.cpu().numpy() for t in c.backward(part, xd, gd)])
    assert all(np.array_equal(a, b) for a, b in zip(*got)) and np.isfinite(got[0][0]).all()
    c.close()
