"""Calls recorded into a CUDA graph after eager calls on the same handle: the recording
runs nothing, so eager calls made before the first replay see the accumulator and the long
integration as the eager calls left them, and each replay adds what it recorded, once.
Integer-valued inputs: every precision gives the oracle's exact sums."""
import numpy as np
import pytest
import torch

import oracle
import synth
from paper_1305_5639_gb300 import api

pytestmark = pytest.mark.gpu
DEV = "cuda"
N_CHAN, K = 3, 64

KINDS = [dict(precision="fp32", n_in=20), dict(precision="fp32", n_in=70), dict(precision="int8", n_in=16),
         dict(precision="int8", n_in=70), dict(precision="int8", n_in=70, xengine="cudacore"),
         dict(precision="int8", n_in=70, planar=True), dict(precision="fp16", n_in=70),
         dict(precision="fp16_hilo", n_in=70)]


def _id(kw):
    return "-".join(str(v) for v in kw.values())


class Case:
    def __init__(self, n_in, **kw):
        self.c = api.Correlator(n_in, 1, N_CHAN, K, **kw)
        self.int8, self.planar = kw["precision"] == "int8", kw.get("planar", False)
        codes = [synth.chan_int8(N_CHAN, n_in, K, seed=s) for s in (1, 2)]
        self.x = [self.input(X) for X in codes]
        self.V = [self.complex(oracle.cmac(X)) for X in codes]
        torch.cuda.synchronize()

    @staticmethod
    def complex(v):
        return v[..., 0] + 1j * v[..., 1]

    def input(self, X):
        t = torch.from_numpy(X).to(DEV)
        if self.planar:
            return t.permute(0, 3, 1, 2).contiguous().to(torch.float16)
        return t if self.int8 else torch.view_as_complex(t.float())

    def accum(self):
        a = self.c.accum().cpu().numpy()
        return self.complex(a.astype(np.float64)) if self.int8 else a.astype(np.complex128)

    def record(self, fn, mode="global"):
        """fn recorded on the current stream, without waiting for what is queued there."""
        g = torch.cuda.CUDAGraph()
        g.capture_begin(capture_error_mode=mode)
        try:
            fn()
        finally:
            g.capture_end()
        return g


@pytest.fixture(params=KINDS, ids=_id)
def case(request, cuda_ok):
    k = Case(**request.param)
    with torch.cuda.stream(torch.cuda.Stream()):
        yield k
        torch.cuda.synchronize()
    k.c.close()


@pytest.mark.parametrize("mode", ["global", "thread_local"])
@pytest.mark.parametrize("clear", ["reset", "dump", "restore_vis"])
def test_recorded_xengine_then_eager_one(case, clear, mode):
    c = case.c
    c.xengine(case.x[0])
    c.accum()
    busy = torch.ones((4096, 4096), device=DEV)
    for _ in range(40):                      # the eager calls below wait in the queue
        busy = busy @ busy * 1e-4
    c.xengine(case.x[0])
    if clear == "dump":
        c.dump(out=torch.empty((N_CHAN, c.n_base), dtype=torch.complex128, device=DEV))
    else:
        getattr(c, clear)()
    g = case.record(lambda: c.xengine(case.x[1]), mode)
    assert not case.accum().any()            # nothing has run since the accumulator was cleared
    c.xengine(case.x[0])
    assert np.array_equal(case.accum(), case.V[0])
    del g


def test_recorded_accum_reads_what_is_there(case):
    c = case.c
    c.xengine(case.x[0])
    out = c.accum()
    g = case.record(lambda: c.accum(out=out))
    c.reset()
    g.replay()
    assert not out.abs().cpu().numpy().any()


def test_replays_add_only_what_they_recorded(case):
    """A deferred dump that waits when the recording begins is added once, not per replay."""
    c = case.c
    vis = torch.empty((N_CHAN, c.n_base), dtype=torch.complex128, device=DEV)
    c.xengine(case.x[0])
    c.dump(copy=False)

    def step():
        c.xengine(case.x[1])
        c.dump(out=vis)

    g = case.record(step)
    g.replay()
    assert np.array_equal(vis.cpu().numpy(), case.V[0] + case.V[1])
    g.replay()
    assert np.array_equal(vis.cpu().numpy(), case.V[0] + 2 * case.V[1])


def test_warm_up_reset_record_replay(case):
    c = case.c
    vis = torch.empty((N_CHAN, c.n_base), dtype=torch.complex128, device=DEV)

    def step():
        c.xengine(case.x[1])
        c.dump(out=vis)

    step()
    c.reset()
    g = case.record(step)
    for n in (1, 2):
        g.replay()
        assert np.array_equal(vis.cpu().numpy(), n * case.V[1])
    c.reset()
    g.replay()
    assert np.array_equal(vis.cpu().numpy(), case.V[1])
    c.xengine(case.x[0])
    assert np.array_equal(c.dump().cpu().numpy(), case.V[0] + case.V[1])
