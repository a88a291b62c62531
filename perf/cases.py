"""The work a user of the correlator has it do, as measurable cases.

A case is a dict of plain values; ``kind`` names the part of the public interface:

  fx       a whole integration: F-engine, X-engine, the integration's visibilities
           copied out, dump into the FP64 long integration
  host     the same from host buffers in one call (copies pipelined with the engines)
  fengine  channelisation alone (plain FFT, delay compensation, polyphase filter bank)
  xengine  correlation alone, with its dump (all precisions, with and without gains)
  cal      gain calibration: the gained X-engine and its adjoint through autograd
  batch    many uneven sub-arrays correlated by one planned launch

Buffers that a program keeps from one integration to the next (channelised data,
visibilities, the handle) are made in ``prepare``; ``run`` is what it calls per
integration.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1305_5639_gb300.api import Batch, Correlator
from paper_1305_5639_gb300.autograd import CorrFn


def listed():
    return [
        # The smallest deployment that is still an array: eight dual-polarisation antennas
        # and 64 channels, short integrations; the call is launches and latency.
        dict(name="fx_int8_16in", kind="fx", n_ant=8, n_pol=2, n_chan=64, n_spectra=96, prec="int8", planar=False,
             copy_vis=True),
        # Float voltages on a small array, the FP32 workload of the benchmark.
        dict(name="fx_fp32_16in", kind="fx", n_ant=16, n_pol=1, n_chan=256, n_spectra=1024, prec="fp32",
             planar=False, copy_vis=False),
        # The benchmark's INT8 workload: 256 antennas x 2 pol, the integration's INT32
        # visibilities copied out, its FP64 dump left to the next integration's launch.
        dict(name="fx_int8_512in", kind="fx", n_ant=256, n_pol=2, n_chan=1024, n_spectra=4096, prec="int8",
             planar=True, copy_vis=False),
        # Voltages that arrive in host memory, visibilities wanted there.
        dict(name="host_int8_128in", kind="host", n_ant=64, n_pol=2, n_chan=1024, n_spectra=1024, prec="int8",
             planar=True),
        # Channelisation with per-antenna delay compensation, as a tracking array has it.
        dict(name="fengine_delay_1024", kind="fengine", n_ant=64, n_pol=2, n_chan=1024, n_spectra=4096, prec="int8",
             planar=True, delays=True, taps=0),
        # The four-tap polyphase filter bank in front of the FFT.
        dict(name="fengine_pfb_1024", kind="fengine", n_ant=64, n_pol=2, n_chan=1024, n_spectra=2048, prec="int8",
             planar=True, delays=False, taps=4),
        # A spectral-line mode: the longest FFT, byte layout, an odd number of spectra.
        dict(name="fengine_4096_odd", kind="fengine", n_ant=31, n_pol=2, n_chan=4096, n_spectra=403, prec="int8",
             planar=False, delays=False, taps=0),
        # Byte data from another channeliser, sizes that are no multiple of a tile.
        dict(name="xengine_int8_250in", kind="xengine", n_in=250, n_chan=128, n_spectra=1500, prec="int8",
             planar=False, gains=False),
        # A large array at 16 bits with per-input gains: a few channels of 2048 inputs.
        dict(name="xengine_fp16_2048in", kind="xengine", n_in=2048, n_chan=16, n_spectra=2048, prec="fp16",
             planar=False, gains=True),
        # A calibration step of 512 inputs on the tensor cores.
        dict(name="cal_hilo_512in", kind="cal", n_in=512, n_chan=256, n_spectra=1024, prec="fp16_hilo"),
        # A calibration step at full FP32, odd sizes.
        dict(name="cal_fp32_130in", kind="cal", n_in=130, n_chan=64, n_spectra=500, prec="fp32"),
        # Sub-arrays of 32 to 2048 antennas, one window of channels each.
        dict(name="batch_32sub", kind="batch", n_sub=32, n_chan=16, shapes=0),
    ]


def _log(rng: random.Random, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(["fx", "fx", "fx", "host", "fengine", "fengine", "fengine", "xengine", "xengine", "cal",
                           "cal", "batch"])
        if kind in ("fx", "host", "fengine"):
            prec = "int8" if kind != "fx" else rng.choice(["int8", "int8", "fp32"])
            planar = prec == "int8" and (kind == "host" or rng.random() < 0.6)
            c = dict(kind=kind, n_ant=_log(rng, 4, 256), n_pol=rng.choice([1, 2]),
                     n_chan=rng.choice([64, 256, 512, 1024, 1024, 2048, 4096]), n_spectra=_log(rng, 48, 4096),
                     prec=prec, planar=planar)
            if kind == "host":
                c["n_spectra"] = max(64, c["n_spectra"] // 2)
            if planar:
                c["n_spectra"] = max(8, c["n_spectra"] // 8 * 8)
            if kind == "fx":
                c["copy_vis"] = prec == "int8" and rng.random() < 0.5
            if kind == "fengine":
                c["delays"] = rng.random() < 0.4
                c["taps"] = rng.choice([0, 0, 0, 4, 8])
        elif kind == "xengine":
            prec = rng.choice(["int8", "int8", "fp16", "fp16_hilo", "fp32"])
            planar = prec == "int8" and rng.random() < 0.5
            K = _log(rng, 64, 4096)
            c = dict(kind=kind, n_in=_log(rng, 8, 2048), n_chan=_log(rng, 1, 256),
                     n_spectra=max(8, K // 8 * 8) if planar else K, prec=prec, planar=planar,
                     gains=prec != "int8" and rng.random() < 0.5)
        elif kind == "cal":
            prec = rng.choice(["fp16_hilo", "fp32"])
            c = dict(kind=kind, n_in=_log(rng, 16, 512), n_chan=_log(rng, 4, 256), n_spectra=_log(rng, 64, 1024),
                     prec=prec)
            if prec == "fp16_hilo":  # the tensor-core adjoint wants multiples of 8
                c["n_in"], c["n_spectra"] = c["n_in"] // 8 * 8, c["n_spectra"] // 8 * 8
        else:
            c = dict(kind=kind, n_sub=_log(rng, 2, 32), n_chan=rng.choice([4, 8, 16]), shapes=rng.randrange(1, 10**6))
        w = work(c)
        limit = 2.0e9 if kind == "host" else 8.0e9
        flops = 2.0e12 if c.get("prec") == "fp32" else 3.0e13 if kind == "cal" else 9.0e13
        if w["bytes"] <= limit and w["flops"] <= flops:
            return c


# ------------------------------------------------------------------------- inputs
def _n_in(case):
    return case["n_in"] if "n_in" in case else case["n_ant"] * case["n_pol"]


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 7919 + 17)


def _voltages(case, seed):
    """[n_in, n_spectra * n_chan] complex: receiver noise plus a common source that each
    antenna hears a few samples later; 8-bit samples (sigma 16) or complex64."""
    g = _gen(seed)
    n_ant, n_pol, T = case["n_ant"], case["n_pol"], case["n_spectra"] * case["n_chan"]
    i8 = case["prec"] == "int8"
    sigma, amp = (16.0, 1.6) if i8 else (1.0, 0.1)
    d = np.random.default_rng(seed).integers(0, 16, n_ant)
    src = torch.randn((T + 16, 2), generator=g, device="cuda") * amp
    out = torch.empty((n_ant * n_pol, T, 2), dtype=torch.int8 if i8 else torch.float32, device="cuda")
    z = torch.empty((T, 2), device="cuda")
    for i in range(n_ant * n_pol):
        z.normal_(0.0, sigma, generator=g)
        o = 16 - int(d[i // n_pol])
        z += src[o:o + T]
        out[i] = z.round_().clamp_(-127, 127) if i8 else z
    return out if i8 else torch.view_as_complex(out)


def _scale(case, seed):
    """Per-channel re-packing scale: a band pass equalised to an RMS of about 16."""
    r = np.random.default_rng(seed + 1)
    s = (16.0 / 16.1) / math.sqrt(case["n_chan"]) * r.uniform(0.8, 1.25, case["n_chan"])
    return torch.from_numpy(s.astype(np.float32)).cuda()


def _delays(case, seed):
    return np.random.default_rng(seed + 2).uniform(-20.0, 20.0, _n_in(case)).astype(np.float32)


def _window(case, seed):
    """A Hann-windowed sinc over taps x channels, its gain varied a little by seed."""
    P, N = case["taps"], case["n_chan"]
    x = (np.arange(P * N) + 0.5) / N - P / 2
    w = np.sinc(x) * np.sin(np.pi * (np.arange(P * N) + 0.5) / (P * N)) ** 2
    return (w * np.random.default_rng(seed + 3).uniform(0.9, 1.1)).reshape(P, N).astype(np.float32)


def _channelised(n_chan, n_in, K, prec, planar, g):
    """Channelised data as the X-engine takes it: codes of RMS 16, or noise plus a
    source common to all inputs."""
    if prec == "int8":
        shape = (2, n_in, K) if planar else (n_in, K, 2)
        out = torch.empty((n_chan, *shape), dtype=torch.float16 if planar else torch.int8, device="cuda")
        for c in range(n_chan):
            out[c] = (torch.randn(shape, generator=g, device="cuda") * 16).round_().clamp_(-127, 127)
        return out
    out = torch.empty((n_chan, n_in, K, 2), device="cuda")
    for c in range(n_chan):
        out[c].normal_(0.0, 1.0, generator=g)
        out[c] += 0.3 * torch.randn((1, K, 2), generator=g, device="cuda")
    return torch.view_as_complex(out)


def _gains(n_in, seed):
    r = np.random.default_rng(seed + 4)
    v = r.uniform(0.8, 1.2, n_in) * np.exp(1j * r.uniform(-np.pi, np.pi, n_in))
    return torch.from_numpy(v.astype(np.complex64)).cuda()


def _grad_vis(n_chan, n_in, g):
    """dL/dV of a least-squares loss over visibilities normalised by the integration."""
    B = n_in * (n_in + 1) // 2
    return torch.view_as_complex(torch.randn((n_chan, B, 2), generator=g, device="cuda") * 1e-6)


def _subs(case):
    """(inputs, spectra) of each sub-array: antennas log-uniform from 32 to 2048, spectra
    uniform from 512 to 4096 in steps of 64."""
    r = random.Random(case["shapes"])
    return [(_log(r, 32, 2048), 64 * r.randint(8, 64)) for _ in range(case["n_sub"])]


def prepare(case, seed):
    kind, s = case["kind"], dict(kind=case["kind"], case=case)
    if kind == "batch":
        g = _gen(seed)
        s["batch"] = Batch([_channelised(case["n_chan"], m, K, "int8", True, g) for m, K in _subs(case)])
        s["batch"].tune()
        return s
    n_in, N, K, prec = _n_in(case), case["n_chan"], case["n_spectra"], case["prec"]
    if kind in ("xengine", "cal"):
        c = Correlator(n_in, 1, N, K, precision=prec, planar=case.get("planar", False))
        g = _gen(seed)
        s |= dict(c=c, x=_channelised(N, n_in, K, prec, case.get("planar", False), g))
        if kind == "cal":
            s |= dict(x=s["x"].requires_grad_(), g=_gains(n_in, seed).requires_grad_(), grad=_grad_vis(N, n_in, g))
        else:
            s |= dict(g=_gains(n_in, seed) if case["gains"] else None, acc=c.accum_buffer())
        return s
    c = Correlator(case["n_ant"], case["n_pol"], N, K, precision=prec, planar=case["planar"])
    if case.get("delays"):
        c.set_delays(_delays(case, seed))
    if case.get("taps"):
        c.set_pfb(_window(case, seed))
    s |= dict(c=c, volt=_voltages(case, seed), scale=_scale(case, seed) if prec == "int8" else None)
    if kind == "host":
        s["volt"] = s["volt"].cpu().pin_memory()
        s["acc"] = torch.empty((N, c.n_base, 2), dtype=torch.int32).pin_memory()
        return s
    s["chan"] = c.chan_buffer()
    if kind == "fx":
        s["acc"] = c.accum_buffer()
        if case["copy_vis"]:
            s["vis"] = torch.empty((N, c.n_base), dtype=torch.complex128, device="cuda")
    return s


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].run()
        return state["batch"].vis
    c = state["c"]
    if kind == "host":
        c.fx_host_accum(state["volt"], state["scale"], state["acc"])
        return state["acc"]
    if kind == "fengine":
        return c.fengine(state["volt"], state["scale"], out=state["chan"])
    if kind == "cal":
        v = CorrFn.apply(state["x"], state["g"], c)
        gx, gg = torch.autograd.grad(v, (state["x"], state["g"]), grad_outputs=state["grad"])
        return v.detach(), gx, gg
    if kind == "xengine":
        c.xengine(state["x"], state["g"])
        c.accum(out=state["acc"])
        c.dump(copy=False)
        return state["acc"]
    c.fengine(state["volt"], state["scale"], out=state["chan"])
    c.xengine(state["chan"])
    c.accum(out=state["acc"])
    if "vis" in state:
        return state["chan"], state["acc"], c.dump(out=state["vis"])
    c.dump(copy=False)
    return state["chan"], state["acc"]


# ------------------------------------------------------------------------- work
def work(case):
    kind, nbytes, flops = case["kind"], 0, 0
    if kind == "batch":
        for m, K in _subs(case):
            B = m * (m + 1) // 2
            nbytes += case["n_chan"] * (4 * m * K + 8 * B)
            flops += 8 * case["n_chan"] * B * K
        return dict(bytes=nbytes, flops=flops)
    n_in, N, K, prec = _n_in(case), case["n_chan"], case["n_spectra"], case["prec"]
    B = n_in * (n_in + 1) // 2
    sample = 2 if prec == "int8" else 8                           # raw voltage
    chan = 4 if case.get("planar") else sample                    # channelised sample
    fft = n_in * K * N * 5 * math.log2(N)
    x_flops = 8 * N * B * K
    if kind == "fengine":
        flops = fft + n_in * K * N * (4 * case["taps"] + (6 if case["delays"] else 0))
        return dict(bytes=n_in * K * N * (sample + chan), flops=flops)
    if kind == "host":  # device memory: the voltages and visibilities that cross the link
        return dict(bytes=n_in * K * N * sample + 8 * N * B, flops=fft + x_flops)
    if kind == "cal":
        # X and dL/dV in, V and dL/dX out; forward and the dense product of the adjoint
        return dict(bytes=N * (16 * n_in * K + 16 * B), flops=x_flops + 8 * N * n_in * n_in * K)
    if kind == "xengine":
        return dict(bytes=N * (chan * n_in * K + (8 + 32) * B), flops=x_flops)
    # voltages in, channelised data out and in, visibilities out, long integration updated
    vis = 8 + 32 + (16 if case["copy_vis"] else 0)
    return dict(bytes=n_in * K * N * (sample + 2 * chan) + vis * N * B, flops=fft + x_flops)


# ------------------------------------------------------------------------- 64 bits
def _pairs(n_in):
    i, j = np.tril_indices(n_in)
    return torch.from_numpy(i).cuda(), torch.from_numpy(j).cuda()


def _visibilities(x):
    """Packed lower triangle of X X^H for complex128 [n_chan, n_in, K]."""
    i, j = _pairs(x.shape[1])
    return torch.stack([(a @ a.mH)[i, j] for a in x])


def _spectra(case, s):
    """Complex128 [inputs of a block, n_spectra, n_chan] in blocks of inputs."""
    n_in, N, K = _n_in(case), case["n_chan"], case["n_spectra"]
    T = N * K
    P = case.get("taps", 0)
    k = torch.arange(N, device="cuda", dtype=torch.float64)
    step = max(1, (1 << 26) // T)
    for i0 in range(0, n_in, step):
        v = s["volt"][i0:i0 + step]
        v = torch.complex(v[..., 0].double(), v[..., 1].double()) if v.dtype == torch.int8 else v.to(torch.complex128)
        frac = None
        if case.get("delays"):
            tau = s["delays"][i0:i0 + step].astype(np.float64)
            whole = np.where(tau >= 0, np.floor(tau + 0.5), -np.floor(-tau + 0.5)).astype(np.int64)
            frac = torch.from_numpy(tau - whole).cuda()
            moved = torch.zeros_like(v)
            for i, d in enumerate(whole):
                a, b = max(0, -int(d)), T - max(0, int(d))
                if b > a:
                    moved[i, a:b] = v[i, a + int(d):b + int(d)]
            v = moved
        v = v.reshape(v.shape[0], K, N)
        if P:
            y = torch.zeros_like(v)
            for p in range(min(P, K)):
                y[:, :K - p] += s["window"][p] * v[:, p:]
            v = y
        v = torch.fft.fft(v, dim=-1)
        if frac is not None:
            v = v * torch.exp(2j * math.pi * k * frac[:, None] / N)[:, None, :]
        yield i0, v


def _codes(case, s):
    """The re-packed channelised data in FP64, in the layout of the case."""
    n_in, N, K = _n_in(case), case["n_chan"], case["n_spectra"]
    out = torch.empty((N, 2, n_in, K) if case["planar"] else (N, n_in, K, 2), dtype=torch.float64, device="cuda")
    sc = s["scale"].double()
    for i0, S in _spectra(case, s):
        S = torch.view_as_real(S * sc).round_().clamp_(-127, 127)  # [i, a, k, 2]
        i1 = i0 + S.shape[0]
        if case["planar"]:
            out[:, :, i0:i1] = S.permute(2, 3, 0, 1)
        else:
            out[:, i0:i1] = S.permute(2, 0, 1, 3)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "host"):
        return None  # whole numbers
    n_in, N, K, prec = _n_in(case), case["n_chan"], case["n_spectra"], case["prec"]
    if kind in ("fx", "fengine"):
        s = dict(volt=_voltages(case, seed), scale=_scale(case, seed))
        if case.get("delays"):
            s["delays"] = _delays(case, seed)
        if case.get("taps"):
            s["window"] = torch.from_numpy(_window(case, seed)).cuda().double()
        if prec == "int8":
            codes = _codes(case, s)
            if kind == "fengine":
                return codes
            return [codes, None, None] if case["copy_vis"] else [codes, None]  # visibilities: whole numbers
        x = torch.empty((N, n_in, K), dtype=torch.complex128, device="cuda")
        for i0, S in _spectra(case, s):
            x[:, i0:i0 + S.shape[0]] = S.permute(2, 0, 1)
        if kind == "fengine":
            return x
        return x, _visibilities(x)
    if prec == "int8":
        return None
    g = _gen(seed)
    x = _channelised(N, n_in, K, prec, False, g)
    gain = _gains(n_in, seed).to(torch.complex128)
    if kind == "xengine":
        if 8.0 * n_in * n_in * K * N > 8e12:
            return None
        i, j = _pairs(n_in)
        v = _visibilities(x.to(torch.complex128))
        return v * (gain[i] * gain[j].conj()) if case["gains"] else v
    grad = _grad_vis(N, n_in, g)
    i, j = _pairs(n_in)
    V = torch.empty((N, n_in * (n_in + 1) // 2), dtype=torch.complex128, device="cuda")
    gx = torch.empty((N, n_in, K), dtype=torch.complex128, device="cuda")
    gg = torch.zeros(n_in, dtype=torch.complex128, device="cuda")
    for f in range(N):
        a = x[f].to(torch.complex128)
        V[f] = (a @ a.mH)[i, j] * (gain[i] * gain[j].conj())
        L = torch.zeros((n_in, n_in), dtype=torch.complex128, device="cuda")
        L[i, j] = grad[f].to(torch.complex128)
        y = (L + L.mH) @ (gain[:, None] * a)
        gx[f] = gain.conj()[:, None] * y
        gg += (a.conj() * y).sum(1)
    return V, gx, gg
