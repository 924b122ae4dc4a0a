"""A call whose launches are turned down reports it, and the next one starts from there.

The stream is put into a capture and the capture invalidated by a synchronisation, which the
runtime answers with an error: every launch on the stream is then refused on the host, and
nothing reaches the GPU.  A step call in that state must fail and must not count: once the
capture has ended, the run gives the bits of one that never failed (its noise above all,
which the failed call had been about to make).
"""
import ctypes

import numpy as np
import pytest

from helpers import gpu_ctx
from paper_1905_02521_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qtb():
    import torch
    assert torch.cuda.is_available()
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb as q
    return q


class RefusingStream:
    """Between entry and exit every launch on `stream` is refused by the runtime."""

    def __init__(self, stream):
        self.cu = ctypes.CDLL("libcuda.so.1")
        self.st = ctypes.c_void_p(stream)

    def __enter__(self):
        assert self.cu.cuStreamBeginCapture_v2(self.st, 2) == 0
        assert self.cu.cuStreamSynchronize(self.st) != 0

    def __exit__(self, *exc):
        g = ctypes.c_void_p()
        assert self.cu.cuStreamEndCapture(self.st, ctypes.byref(g)) != 0
        return False


def _run(qtb, kind, precision, generator, before, n, fail):
    import torch
    if kind == "pair":
        s, pot = W.mgo_system(2, 300.0)
        kw = {}
    else:
        s, pot = W.oscillators(33, 120.0, 4e-3, x0=0.4, spread=0.1, seed=5)[0], W.well_potential()
        kw = dict(potential=qtb.POT_DOUBLEWELL, ext={"V0": 0.1, "a": 0.5})
    N = len(s["types"])
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = gpu_ctx(qtb, [s], pot, 0.5, precision=precision, seed=3, obs_stride=16, **kw)
        try:
            qtb.qtb_set_filter(ctx, 0, qtb.NOISE_QTB, 513, 0.3)
            if generator:
                qtb.qtb_set_generator(ctx, qtb.GEN_FOURIER, 2)
            qtb.qtb_step_n(ctx, before)
            qtb.qtb_sync(ctx)
            if fail:
                with RefusingStream(stream.cuda_stream):
                    with pytest.raises(qtb.QtbError):
                        qtb.qtb_step_n(ctx, n)
                assert qtb.qtb_get_step(ctx) == before
            qtb.qtb_step_n(ctx, n)
            return qtb.qtb_get_state(ctx, 0, 1, N) + (qtb.qtb_get_series(ctx, 0, 100),)
        finally:
            qtb.qtb_destroy(ctx)


@pytest.mark.parametrize("generator", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["pair", "wells"])
@pytest.mark.parametrize("before,n", [(0, 100), (0, 300), (256, 256), (250, 300)])
def test_refused_step_does_not_count(qtb, kind, precision, generator, before, n):
    ok, retried = (_run(qtb, kind, precision, generator, before, n, f) for f in (False, True))
    assert all(np.array_equal(a, b) for a, b in zip(ok, retried))
