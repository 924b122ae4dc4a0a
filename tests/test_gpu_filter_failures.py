"""A filter or generator set-up that runs out of device memory leaves a usable context.

Every allocation that the call makes is made to fail in turn (the allocator the library is
given returns null), once or from there on.  A call that fails must leave the run as it would
have been without it, or, where not even the former set-up could be restored, a context that
refuses to step; a call that succeeds all the same must give its noise to rounding.  Afterwards,
with memory to be had again, the call goes through and gives the bits of a fresh context.
A filter too long for the shared memory is refused and changes nothing either.
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


class Memory:
    """The library's allocator with a switch: allocation number `at` fails (all from there on
    with `rest`)."""

    def __init__(self, qtb, monkeypatch):
        alloc, free = qtb._torch_allocator()
        self.n, self.at, self.rest = 0, None, False

        def get(nbytes, user):
            self.n += 1
            if self.at is not None and (self.n == self.at or (self.rest and self.n > self.at)):
                return None
            return alloc(nbytes, user)

        self.cb = (qtb.ALLOC_FN(get), free)
        monkeypatch.setattr(qtb, "_torch_allocator", lambda: self.cb)

    def fail(self, at, rest=False):
        self.n, self.at, self.rest = 0, at, rest


CALLS = {
    "longer filter": lambda q, c: q.qtb_set_filter(c, 0, q.NOISE_QTB, 1025, 0.3),
    "solved filter": lambda q, c: q.qtb_set_filter(c, 1, q.NOISE_QTB_PIMD, 513, 0.6),
    "segments": lambda q, c: q.qtb_set_generator(c, q.GEN_FOURIER, 4),
}


def _ctx(q, precision, filter_prec):
    sys = [W.oscillators(33, 120.0, 4e-3, x0=0.4, spread=0.1, seed=5)[0],
           W.oscillators(21, 90.0, 4e-3, n_beads=3, x0=0.4, spread=0.1, seed=6)[0]]
    ctx = gpu_ctx(q, sys, W.well_potential(), 0.5, precision=precision, filter_prec=filter_prec, seed=3,
                  potential=q.POT_HARMONIC, ext={"omega": 0.02}, obs_stride=64)
    q.qtb_set_filter(ctx, 0, q.NOISE_QTB, 129, 0.3)
    q.qtb_step_n(ctx, 300)
    return ctx


def _go(q, ctx):
    q.qtb_step_n(ctx, 400)
    return q.qtb_get_state(ctx, 0, 1, 33) + q.qtb_get_state(ctx, 1, 3, 21)


def _run(q, precision, filter_prec, call=None):
    ctx = _ctx(q, precision, filter_prec)
    try:
        if call:
            call(q, ctx)
        return _go(q, ctx)
    finally:
        q.qtb_destroy(ctx)


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("precision,filter_prec", [(0, 0), (1, 1), (1, 2)])
@pytest.mark.parametrize("name", list(CALLS))
def test_failed_allocations(qtb, monkeypatch, name, precision, filter_prec):
    mem = Memory(qtb, monkeypatch)
    call = CALLS[name]
    old, new = _run(qtb, precision, filter_prec), _run(qtb, precision, filter_prec, call)
    tol = 1e-9 if precision == 0 else 1e-4   # (a success may have taken another form of the same filter)
    ctx = _ctx(qtb, precision, filter_prec)
    mem.fail(None)
    call(qtb, ctx)
    count = mem.n
    qtb.qtb_destroy(ctx)
    assert count > 0
    for at in range(1, count + 1):
        for rest in (False, True):
            ctx = _ctx(qtb, precision, filter_prec)
            try:
                mem.fail(at, rest)
                try:
                    call(qtb, ctx)
                    failed = False
                except qtb.QtbError:
                    failed = True
                mem.fail(None)
                refused = False
                try:
                    got = _go(qtb, ctx)
                except qtb.QtbError:
                    refused = True
                if refused:
                    assert failed and qtb.qtb_get_step(ctx) == 300
                    call(qtb, ctx)
                    assert _same(_go(qtb, ctx), new)
                elif failed:
                    assert _same(got, old)
                else:
                    assert all(np.allclose(x, y, rtol=tol, atol=tol * np.abs(y).max()) for x, y in zip(got, new))
            finally:
                mem.fail(None)
                qtb.qtb_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
def test_filter_too_long_changes_nothing(qtb, precision):
    old = _run(qtb, precision, 1)
    ctx = _ctx(qtb, precision, 1)
    try:
        with pytest.raises(qtb.QtbError):
            qtb.qtb_set_filter(ctx, 0, qtb.NOISE_QTB, 30001, 0.3)
        assert _same(_go(qtb, ctx), old)
    finally:
        qtb.qtb_destroy(ctx)


@pytest.mark.parametrize("atoms,taps", [((80000, 80000), (2049, 2049)), ((165000, 5), (2049, 81))])
def test_spectra_limit_is_the_contexts(qtb, monkeypatch, atoms, taps):
    # two systems within the 16 GiB that a ring of spectra may take but not together, and a
    # short one beside one that passes it alone: no allocation is larger than the limit
    mem = Memory(qtb, monkeypatch)
    sizes = []
    get, free = mem.cb
    cb = (qtb.ALLOC_FN(lambda nbytes, user: (sizes.append(nbytes), get(nbytes, user))[1]), free)
    monkeypatch.setattr(qtb, "_torch_allocator", lambda: cb)
    sys = [W.oscillators(n, 120.0, 4e-3, x0=0.4, spread=0.1, seed=k)[0] for k, n in enumerate(atoms)]
    ctx = gpu_ctx(qtb, sys, W.well_potential(), 0.5, precision=0, potential=qtb.POT_HARMONIC, ext={"omega": 0.02},
                  obs_stride=256, max_records=4)
    try:
        for k, n in enumerate(taps):
            qtb.qtb_set_filter(ctx, k, qtb.NOISE_QTB, n, 0.3)
        dofs = 3 * sum(atoms)
        assert 2 * 8 * 9 * 256 * dofs > 16 << 30
        assert 8 * 9 * 256 * dofs <= max(sizes) <= 16 << 30
    finally:
        qtb.qtb_destroy(ctx)
