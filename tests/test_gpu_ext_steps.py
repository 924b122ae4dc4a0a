"""External potentials, many steps per launch: a run cut into uneven calls gives the same
trajectory bit for bit as one call (block graphs, partial blocks), and the same records
(sums in FP64: 1e-12 relative; FP32 form 1e-6, its own rounding of bead sums differs
nowhere but in the last place of a float-float sum), for the bead counts that are carried
through a launch and one that is not (16), alone in a ragged unit and batched; harmonic
FP64 rings follow the oracle."""
import numpy as np
import pytest

from helpers import gpu_ctx, oracle_sim, rel_inf
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


def _systems(Ps):
    return [W.oscillators(33 - k, 120.0, 4e-3, n_beads=P, x0=0.4, spread=0.1, seed=5 + k)[0] for k, P in enumerate(Ps)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("stride", [1, 7, 300])
@pytest.mark.parametrize("Ps", [(1,), (8,), (3, 1, 16, 6)])
def test_cuts_change_nothing(qtb, precision, stride, Ps):
    pot = W.well_potential()
    out = []
    for cuts in ([600], [256, 1, 255, 88], [100, 300, 200]):
        ctx = gpu_ctx(qtb, _systems(Ps), pot, 0.5, precision=precision, filter_prec=1, seed=3,
                      potential=qtb.POT_DOUBLEWELL, ext={"V0": 0.1, "a": 0.5}, obs_stride=stride, max_records=1000)
        try:
            for n in cuts:
                qtb.qtb_step_n(ctx, n)
            out.append([qtb.qtb_get_state(ctx, k, P, 33 - k) + (qtb.qtb_get_forces(ctx, k, P, 33 - k),)
                        for k, P in enumerate(Ps)] + [[qtb.qtb_get_series(ctx, k, 1000) for k in range(len(Ps))]])
            assert len(out[-1][-1][0]) == 600 // stride
            assert np.array_equal(qtb.qtb_observables(ctx, 0), out[-1][-1][0][-1])
        finally:
            qtb.qtb_destroy(ctx)
    for o in out[1:]:
        for a, b in zip(o[:-1], out[0][:-1]):
            assert all(np.array_equal(x, y) for x, y in zip(a, b))
        for a, b in zip(o[-1], out[0][-1]):
            assert np.allclose(a, b, rtol=1e-12 if precision == 0 else 1e-6, atol=1e-12)


@pytest.mark.parametrize("P", [1, 2, 5, 8])
def test_records_match_oracle(qtb, oracle, P):
    s, pot = W.oscillators(35, 150.0, 2e-3, n_beads=P, x0=0.3, spread=0.1)
    ctx = gpu_ctx(qtb, [s], pot, 0.5, precision=0, seed=8, potential=qtb.POT_HARMONIC, ext={"omega": 0.05}, obs_stride=5)
    try:
        sim = oracle_sim(oracle, s, pot, 0.5, seed=8, potential=qtb.POT_HARMONIC, ext={"omega": 0.05})
        qtb.qtb_step_n(ctx, 40)
        rec = np.asarray(sim.step(40, record=True)).reshape(-1, 23)[4::5]
        ser = qtb.qtb_get_series(ctx, 0, 100)
        x, v = qtb.qtb_get_state(ctx, 0, P, 35)
        xo, vo, _, _ = sim.state()
        assert rel_inf(x, xo) < 1e-11 and rel_inf(v, vo) < 1e-11
        # (slot 20, the cell volume, is the oracle's own business without a box; off-diagonal
        # virials of a separable potential are not formed)
        for q in (0, 1, 2, 3, 4, 5, 9, 13, 14, 15, 16, 17, 18, 19):
            assert np.allclose(ser[:, q], rec[:, q], rtol=1e-10, atol=1e-10), q
    finally:
        qtb.qtb_destroy(ctx)
