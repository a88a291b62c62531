"""The power pass with a window that the F-engine filters by itself, against the two-pass
form (FIR pass, then FFT) that the same samples take as floats: the frames and transforms are
the same, only the order of the sums differs."""
import numpy as np
import pytest
import torch

from paper_1305_5639_gb300.api import Correlator

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,n_in,P", [
    (64, 1, 3, 4), (64, 2501, 130, 4), (64, 700, 16, 8), (128, 33, 5, 3), (128, 2050, 130, 8), (256, 17, 4, 5),
    (256, 1300, 200, 4), (512, 47, 3, 8), (512, 1301, 100, 4), (1024, 1, 2, 1), (1024, 1237, 70, 4), (1024, 40, 6, 7),
    (2048, 65, 5, 4), (2048, 203, 20, 8), (4096, 9, 2, 4), (4096, 61, 16, 8)])
@pytest.mark.parametrize("delays", [False, True])
def test_power_of_filtered_frames(cuda_ok, N, K, n_in, P, delays):
    g = torch.Generator(device="cuda").manual_seed(N + K)
    v = torch.randint(-60, 61, (n_in, K * N, 2), dtype=torch.int8, device="cuda", generator=g)
    h = np.random.default_rng(K).standard_normal((P, N)).astype(np.float32)
    d = np.random.default_rng(N).uniform(-9, 9, n_in).astype(np.float32) if delays else None
    # every input's weight in the sum differs, so that none can take another's place
    v = (v.float() * torch.linspace(0.2, 2.0, n_in, device="cuda")[:, None, None]).to(torch.int8)
    p = []
    for prec, volt in (("int8", v), ("fp32", v.float())):
        c = Correlator(n_in, 1, N, K, precision=prec)
        c.set_pfb(h)
        c.set_delays(d)
        p.append(c.fengine_power(volt).double())
        c.close()
    # the same frames and transforms; FP32 sums of at most 16 spectra (8 + 1 additions), the
    # result rounded, in each
    assert float(((p[0] - p[1]).abs() / p[1]).max()) < 2 * (9 + 1) * 2.0**-24


def test_power_pass_allocates_nothing(cuda_ok):
    N, K, n_in = 256, 4096, 64   # 512 MB of frames
    h = np.ones((4, N), np.float32)
    v = torch.ones((n_in, K * N, 2), dtype=torch.int8, device="cuda")
    out = torch.empty(N, device="cuda")
    free = []
    for _ in range(2):           # the first round loads the kernels
        c = Correlator(n_in, 1, N, K, precision="int8")
        c.set_pfb(h)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        c.fengine_power(v, out=out)
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
        c.close()
    assert free[2] == free[3]
