"""The sums of the per-channel power pass: at most 16 spectra of an input join in FP32, the
rest in FP64. Frames with one sample at the start have the same exact spectrum in every
channel, so that the sums alone round."""
import numpy as np
import pytest
import torch

from paper_1305_5639_gb300.api import Correlator

pytestmark = pytest.mark.gpu
LENGTHS = [16, 64, 128, 256, 512, 1024, 2048, 4096]


def _power(N, n_in, amp, delays=False):
    """Sum of the powers of n_in inputs: the amplitudes amp at the start of input 0's frames,
    1 at the start of the others'."""
    K = len(amp)
    v = torch.zeros((n_in, K, N), dtype=torch.complex64, device="cuda")
    v[:, :, 0] = 1
    v[0, :, 0] = torch.tensor(amp, dtype=torch.complex64)
    c = Correlator(n_in, 1, N, K, precision="fp32")
    if delays:
        c.set_delays(np.zeros(n_in, np.float32))
    p = c.fengine_power(v.view(n_in, -1)).cpu().numpy().astype(np.float64)
    c.close()
    return p * (2 * n_in * K)


# one input, and enough of them that a CTA goes over several blocks of spectra
@pytest.mark.parametrize("N,n_in", [(N, 1) for N in LENGTHS] + [(N, 512 if N <= 1024 else 128) for N in LENGTHS])
@pytest.mark.parametrize("delays", [False, True])
def test_large_power_hides_sixteen_spectra_at_most(cuda_ok, N, n_in, delays):
    # powers 2^30 and 82 among n = 512 n_in - 2 ones: 2^30 + n + 2 + 80. FP32 steps at 2^30
    # are 128, so the ones that meet the large power in FP32 are lost, up to 15 of them; that
    # leaves more than half a step above 2^30 + n + 2, which the result rounds up to the next
    # step (16 lost: a tie, down)
    amp = np.ones(512, np.complex64)
    amp[0], amp[-1] = 2.0**15, 9 + 1j
    assert np.array_equal(_power(N, n_in, amp, delays), np.full(N, 2.0**30 + 512 * n_in + 128))


@pytest.mark.parametrize("N", LENGTHS)
def test_infinite_power_stays_infinite(cuda_ok, N):
    amp = np.ones(100, np.complex64)
    amp[37] = 1e25
    assert np.all(np.isposinf(_power(N, 1, amp)))
