"""Contexts side by side: what one sets up must not limit the kernels of another.

The dynamic shared memory a kernel may be launched with is a property of the function on
the device, not of a context.  A context whose kernels need much of it (long FP32 filter,
dense cell lists, long Fourier segments) is made, then one that needs little, then the first
is stepped, by part of a block and through whole blocks.  It must run, and give the bits it
gives alone.
"""
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


def _wells(qtb, precision, setup):
    s = W.oscillators(33, 120.0, 4e-3, x0=0.4, spread=0.1, seed=5)[0]
    ctx = gpu_ctx(qtb, [s], W.well_potential(), 0.5, precision=precision, filter_prec=1, seed=3,
                  potential=qtb.POT_DOUBLEWELL, ext={"V0": 0.1, "a": 0.5}, obs_stride=64)
    setup(ctx)
    return ctx, 33


def _crystal(qtb, precision, r_cut):
    s, pot = W.mgo_system(4, 1500.0)
    ctx = gpu_ctx(qtb, [s], dict(pot, r_cut=r_cut), 1.0, precision=precision, seed=3, obs_stride=64)
    return ctx, len(s["types"])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("what", ["filter", "segments", "lists"])
def test_second_context_changes_nothing(qtb, what, precision):
    if what == "filter":
        big = lambda: _wells(qtb, precision, lambda c: qtb.qtb_set_filter(c, 0, qtb.NOISE_QTB, 2049, 0.3))
        small = lambda: _wells(qtb, precision, lambda c: None)
    elif what == "segments":
        big = lambda: _wells(qtb, precision, lambda c: (qtb.qtb_set_generator(c, qtb.GEN_FOURIER, 8),
                                                        qtb.qtb_set_filter(c, 0, qtb.NOISE_QTB, 513, 0.3)))
        small = lambda: _wells(qtb, precision, lambda c: qtb.qtb_set_generator(c, qtb.GEN_FOURIER, 1))
    else:
        big, small = lambda: _crystal(qtb, precision, 8.0), lambda: _crystal(qtb, precision, 2.6)
    out = []
    for beside in (False, True):
        ctx, N = big()
        other = small()[0] if beside else None
        try:
            for n in (100, 156, 512):
                qtb.qtb_step_n(ctx, n)
            out.append(qtb.qtb_get_state(ctx, 0, 1, N))
        finally:
            qtb.qtb_destroy(ctx)
            if other:
                qtb.qtb_destroy(other)
    assert all(np.array_equal(a, b) for a, b in zip(*out))
