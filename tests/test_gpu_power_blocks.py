"""The per-channel power pass where a CTA goes over several blocks of spectra: enough
inputs and spectra for that at each length, ragged last blocks, int8 and FP32 voltages,
with and without delays, against a 64-bit DFT."""
import numpy as np
import pytest
import torch

from paper_1305_5639_gb300.api import Correlator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["int8", "fp32"])
@pytest.mark.parametrize("N,K", [(16, 7001), (64, 2503), (128, 2051), (256, 1302), (512, 1301),
                                 (1024, 1237), (2048, 651), (4096, 619), (1024, 3)])
def test_power_blocks(cuda_ok, N, K, prec):
    n_in = 128
    g = torch.Generator(device="cuda").manual_seed(N + K)
    v = torch.randint(-60, 61, (n_in, K * N, 2), dtype=torch.int8, device="cuda", generator=g)
    c = Correlator(n_in // 2, 2, N, K, precision=prec)
    volt = v if prec == "int8" else v.float()
    p = c.fengine_power(volt).double()
    ref = torch.zeros(N, dtype=torch.float64, device="cuda")
    for i in range(n_in):
        x = torch.view_as_complex(v[i].double()).view(K, N)
        ref += torch.fft.fft(x, dim=1).abs().square().sum(0)
    ref /= 2 * n_in * K
    # |X|^2 of an FP32 transform (log2 N stages, two roundings each, both factors of the
    # square), at most 12 FP32 additions, one rounding of the result
    tol = (4 * np.log2(N) + 12 + 1) * 2.0**-24
    assert float(((p - ref).abs() / ref).max()) < tol
    # with delays: the record advanced by the integer part, zero outside; the phase of the
    # fraction leaves the powers alone (two more factors of two roundings each)
    c.set_delays(np.full(n_in, 3.25, np.float32))
    q = c.fengine_power(volt).double()
    w = torch.zeros_like(v)
    w[:, :-3] = v[:, 3:]
    c.set_delays(None)
    r = c.fengine_power(w if prec == "int8" else w.float()).double()
    assert float(((q - r).abs() / r).max()) < 2 * tol + 12 * 2.0**-24
    c.close()
