"""The filter bank fused into the int8 F-engine against the two-pass form (FIR pass, then
FFT), which float voltages take: the same int8 samples given as floats go through the same
FMAs in the same order, so the codes equal the re-packed FP32 spectra exactly (the product
with the scale is exact in FP64, rounded half to even)."""
import numpy as np
import pytest
import torch

import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("N,K,P,delays,planar", [
    (64, 70, 4, False, False), (64, 33, 7, True, False), (128, 40, 8, True, True), (256, 72, 2, True, True),
    (256, 31, 5, False, False), (512, 35, 3, True, False), (512, 64, 8, False, True), (1024, 16, 4, False, True),
    (1024, 19, 4, True, False), (1024, 40, 8, True, True), (1024, 1, 1, False, False), (2048, 17, 4, True, False),
    (2048, 24, 6, False, True), (4096, 9, 4, True, False), (4096, 8, 8, True, True), (64, 9, 9, True, False)])
def test_fused_filter_bank_equals_two_pass(cuda_ok, N, K, P, delays, planar):
    n_ant, n_pol = 3, 2
    n_in = n_ant * n_pol
    v = synth.volt_int8(n_ant, n_pol, N, K, seed=N + K + P)
    r = np.random.default_rng(N * P + K)
    h = r.standard_normal((P, N)).astype(np.float32)
    # whole and fractional, multiples of four and not, before and past the record
    d = np.array([0.0, 4.0, -7.25, 2.5 * N + 1.3, -1.2 * N, K * N + 3.0], np.float32) if delays else None
    scale = (16.0 / (16.0 * np.sqrt(N * P)) * r.uniform(0.5, 2.0, N)).astype(np.float32)
    a = api.Correlator(n_ant, n_pol, N, K, precision="int8", planar=planar)
    b = api.Correlator(n_ant, n_pol, N, K, precision="fp32")
    for c in (a, b):
        c.set_pfb(h)
        c.set_delays(d)
    codes = a.fengine(torch.from_numpy(v).to(DEV), torch.from_numpy(scale).to(DEV)).cpu().numpy()
    if planar:
        codes = np.transpose(codes, (0, 2, 3, 1))
    vf = torch.view_as_complex(torch.from_numpy(v).to(DEV).float())
    S = b.fengine(vf).cpu().numpy()
    S = np.stack([S.real, S.imag], axis=-1).astype(np.float64) * scale.astype(np.float64)[:, None, None, None]
    assert np.array_equal(codes.astype(np.float64), np.clip(np.rint(S), -127, 127) + 0.0)
    a.close()
    b.close()


def test_power_pass_makes_its_frames_during_a_capture(cuda_ok):
    """The fused filter bank needs no frame buffer; the power pass makes it when first
    called, in a stream capture too, and its replays give the powers of the eager call."""
    N, K, n_in = 256, 24, 4
    v = torch.from_numpy(synth.volt_int8(n_in, 1, N, K, seed=8)).to(DEV)
    h = np.random.default_rng(2).standard_normal((4, N)).astype(np.float32)
    c = api.Correlator(n_in, 1, N, K, precision="int8")
    c.set_pfb(h)
    out = torch.zeros(N, device=DEV)
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(s), torch.cuda.graph(g, stream=s):
        c.fengine_power(v, out=out)
    out.zero_()
    g.replay()
    torch.cuda.synchronize()
    d = api.Correlator(n_in, 1, N, K, precision="int8")
    d.set_pfb(h)
    want = d.fengine_power(v)
    assert torch.allclose(out, want, rtol=1e-5) and bool((out > 0).all())
    c.close()
    d.close()
