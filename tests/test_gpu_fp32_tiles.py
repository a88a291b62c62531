"""FP32 X-engine and adjoint at the edges of their register tiles (32, 48 and 64 inputs,
the few-input kernel's 4 x 4 blocks, even and odd spectra), against the FP64 oracle, with
the FP32 parity bars (1e-5 of the autocorrelations; gradients 1e-4 relative L2)."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _err(V, ref, n_in):
    i, j = oracle.tri_pairs(n_in)
    aut = np.abs(ref[..., oracle.packed_index(np.arange(n_in), np.arange(n_in))])
    return float(np.max(np.abs(V - ref) / np.sqrt(aut[..., i] * aut[..., j])))


@pytest.mark.parametrize("n_in,K,n_chan", [
    (1, 1, 3), (4, 300, 2), (5, 513, 1), (17, 700, 2), (21, 64, 3), (22, 1026, 1),  # few inputs, K ranges
    (23, 7, 2), (32, 16, 5), (33, 17, 1), (47, 33, 2), (48, 2, 1), (49, 31, 2), (64, 15, 1), (65, 48, 2),
    (96, 20, 400), (97, 21, 1), (144, 18, 2), (250, 40, 3), (257, 19, 1)])
def test_xengine_fp32_tiles(cuda_ok, n_in, K, n_chan):
    X = synth.chan_sources(n_chan, n_in, K, n_src=2, seed=n_in + K)
    g = synth.gains(n_in, seed=K)
    ref = oracle.apply_gains(oracle.cmac(X), g, n_in)
    c = api.Correlator(n_in, 1, n_chan, K)
    Xt, gt = torch.from_numpy(X).to(DEV), torch.from_numpy(g).to(DEV)
    c.xengine(Xt, gt)
    once = c.accum().cpu().numpy()
    assert _err(once, ref, n_in) <= 1e-5
    c.xengine(Xt, gt)  # added to the first
    assert np.array_equal(c.accum().cpu().numpy(), once + once)
    c.close()


@pytest.mark.parametrize("n_in,K,n_chan,with_gains", [
    (1, 1, 2, True), (16, 2, 1, False), (31, 63, 2, True), (32, 64, 1, True), (33, 65, 1, True), (48, 130, 2, False),
    (49, 127, 1, True), (64, 66, 2, True), (96, 5, 3, True), (130, 100, 2, True), (161, 33, 1, False)])
def test_backward_fp32_tiles(cuda_ok, n_in, K, n_chan, with_gains):
    X = synth.chan_sources(n_chan, n_in, K, n_src=2, seed=n_in)
    g = synth.gains(n_in, seed=1) if with_gains else np.ones(n_in, np.complex64)
    r = np.random.default_rng(n_in * K)
    B = n_in * (n_in + 1) // 2
    G = (r.standard_normal((n_chan, B)) + 1j * r.standard_normal((n_chan, B))).astype(np.complex64)
    # Y = G^ diag(g) X with G^ the Hermitian completion; dX = diag(conj g) Y, dg_m = sum conj(X) Y
    i, j = oracle.tri_pairs(n_in)
    L = np.zeros((n_chan, n_in, n_in), np.complex128)
    L[:, i, j] = G
    Y = (L + np.conj(np.transpose(L, (0, 2, 1)))) @ (g[:, None].astype(np.complex128) * X)
    dX_ref, dg_ref = np.conj(g)[:, None] * Y, np.sum(np.conj(X.astype(np.complex128)) * Y, axis=(0, 2))
    c = api.Correlator(n_in, 1, n_chan, K)
    dX, dg = c.backward(torch.from_numpy(G).to(DEV), torch.from_numpy(X).to(DEV),
                        torch.from_numpy(g).to(DEV) if with_gains else None)
    assert np.linalg.norm(dX.cpu().numpy() - dX_ref) <= 1e-4 * np.linalg.norm(dX_ref)
    assert np.linalg.norm(dg.cpu().numpy() - dg_ref) <= 1e-4 * np.linalg.norm(dg_ref)
    only, none = c.backward(torch.from_numpy(G).to(DEV), torch.from_numpy(X).to(DEV),
                            torch.from_numpy(g).to(DEV) if with_gains else None, want_gains=False)
    assert none is None and torch.equal(only, dX)
    c.close()
