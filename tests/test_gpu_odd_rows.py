"""Corner turn and operand conversion where rows start off every alignment: numbers of
spectra of all residues, short last blocks, both layouts. The F-engine's codes equal those
of the same frames in an aligned record (one spectrum's codes do not depend on K), and the
int8 X-engine is exact."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("N", [16, 64, 256, 1024, 2048, 4096])
@pytest.mark.parametrize("fengine", ["auto", "cudacore"])
def test_codes_do_not_depend_on_row_alignment(cuda_ok, N, fengine):
    n_ant, n_pol, Kmax = 3, 1, 64 if N <= 1024 else 32
    v = synth.volt_int8(n_ant, n_pol, N, Kmax, seed=N)
    scale = torch.full((N,), 1.0 / np.sqrt(N), device=DEV)
    c = api.Correlator(n_ant, n_pol, N, Kmax, precision="int8", fengine=fengine)
    want = c.fengine(torch.from_numpy(v).to(DEV), scale).cpu().numpy()
    c.close()
    for K in (1, 2, 3, 7, 8, 9, 15, 16, 17, 18, 24, 31):
        part = torch.from_numpy(np.ascontiguousarray(v[:, :K * N])).to(DEV)
        c = api.Correlator(n_ant, n_pol, N, K, precision="int8", fengine=fengine)
        guard = torch.full((N * n_ant * K * 2 + 64,), 99, dtype=torch.int8, device=DEV)
        out = guard[:N * n_ant * K * 2].view(N, n_ant, K, 2)
        c.fengine(part, scale, out=out)
        assert np.array_equal(out.cpu().numpy(), want[:, :, :K]), K
        assert bool((guard[N * n_ant * K * 2:] == 99).all())
        c.close()
        if K % 8 == 0:
            c = api.Correlator(n_ant, n_pol, N, K, precision="int8", planar=True, fengine=fengine)
            planes = c.fengine(part, scale).cpu().numpy()
            assert np.array_equal(np.transpose(planes, (0, 2, 3, 1)).astype(np.int8), want[:, :, :K]), K
            c.close()


@pytest.mark.parametrize("K", [1, 2, 3, 4, 5, 6, 7, 8, 12, 20, 30, 33, 100])
def test_int8_conversion_of_any_row_length(cuda_ok, K):
    n_in, n_chan = 21, 3
    X = synth.chan_int8(n_chan, n_in, K, seed=K, lo=-128)
    c = api.Correlator(n_in, 1, n_chan, K, precision="int8")
    c.xengine(torch.from_numpy(X).to(DEV))
    assert np.array_equal(c.accum().cpu().numpy().astype(np.int64), oracle.cmac(X))
    c.close()
