"""Steps that are not recorded: every lane count and every variant of the pair-force kernel.

A step that may be recorded always takes 16 lanes (a captured block whose stride does not
divide its 256 steps: all of them), so these runs record none, or one in 256.
* The forces of the last of a few steps against the oracle at the positions reached, with 8,
  16, 32 lanes and the count by size (128 for the smallest, 32 or 16 for the others), over
  list lengths, damping (none, the workloads', beyond the polynomial form) and cells (minimum
  image or image bits).  Tolerances: tests/tolerances.py, derived for these forces.
* The lane count changes no bit of a trajectory with list rebuilds where the minimum image
  holds, with the exponential form, for ring polymers, and in a batch of unlike systems.
"""
import numpy as np
import pytest

from helpers import gpu_ctx, rel_inf, rel_l2
from paper_1905_02521_gb300 import workloads as W
from tolerances import F32_INF, F32_L2, F64_TOL

pytestmark = pytest.mark.gpu

NEVER = 1 << 20


@pytest.fixture(scope="module")
def qtb():
    import torch
    assert torch.cuda.is_available()
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb as q
    return q


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncell,P,r_cut,alpha,strain", [
    (2, 1, 2.6, 0.2, 1.0), (2, 1, 8.0, 0.2, 1.0), (2, 3, 5.0, 0.2, 1.0), (3, 1, 8.0, 0.0, 1.0), (3, 1, 8.0, 0.35, 1.0),
    (3, 2, 8.0, 0.2, 1.03), (5, 1, 8.0, 0.35, 1.0), (5, 1, 8.0, 0.2, 1.03), (5, 2, 8.0, 0.2, 1.0)])
def test_forces_of_unrecorded_steps(qtb, oracle, precision, ncell, P, r_cut, alpha, strain):
    s, pot = W.mgo_system(ncell, 300.0, sigma=0.06, seed=50 + ncell, n_beads=P)
    f = np.array([strain, 1.0, 1.0 / strain])
    s = dict(s, pos=s["pos"] * f, box=s["box"] * f)
    pot = dict(pot, r_cut=r_cut, dsf_alpha=alpha)
    N = len(s["types"])
    for lanes in (8, 16, 32, 0):
        ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=precision, list_lanes=lanes, obs_stride=NEVER, max_records=1)
        try:
            qtb.qtb_step_n(ctx, 5)
            x, _ = qtb.qtb_get_state(ctx, 0, P, N)
            fg = qtb.qtb_get_forces(ctx, 0, P, N)
        finally:
            qtb.qtb_destroy(ctx)
        fo = np.stack([oracle.pair_forces(x[b], s["types"], s["box"], pot)[0] for b in range(P)]) / P
        if precision == 0:
            assert rel_inf(fg, fo) < F64_TOL, lanes
        else:
            assert rel_l2(fg, fo) < F32_L2 and rel_inf(fg, fo) < F32_INF, (lanes, rel_l2(fg, fo), rel_inf(fg, fo))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncells,P,alpha,scope", [((5,), 1, 0.2, 0), ((5,), 1, 0.35, 0), ((3,), 1, 0.35, 0),
                                                 ((5,), 2, 0.2, 0), ((5, 6), 1, 0.2, 0), ((2, 5, 3), 1, 0.2, 1)])
def test_lane_count_changes_no_bit(qtb, precision, ncells, P, alpha, scope):
    systems = []
    for k, n in enumerate(ncells):
        s, pot = W.mgo_system(n, 1500.0, n_beads=P, seed=70 + k)
        keep = np.setdiff1d(np.arange(s["pos"].shape[1]), np.arange(3 + k) * 7)
        systems.append(dict(s, pos=s["pos"][:, keep], vel=s["vel"][:, keep], types=s["types"][keep]))
    pot = dict(pot, dsf_alpha=alpha)
    out = []
    for lanes in (16, 0, 8, 32):
        ctx = gpu_ctx(qtb, systems, pot, 2.0, precision=precision, seed=5, list_lanes=lanes, obs_stride=256,
                      max_records=4, skin=0.3, rebuild_scope=scope)
        try:
            qtb.qtb_step_n(ctx, 300)
            out.append([a for k, s in enumerate(systems) for a in qtb.qtb_get_state(ctx, k, P, len(s["types"]))])
            assert qtb.qtb_list_rebuilds(ctx) > 3
        finally:
            qtb.qtb_destroy(ctx)
    for o in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(o, out[0]))


@pytest.mark.parametrize("K", [39, 40, 41])
def test_fp64_noise_around_the_fast_convolution(qtb, oracle, K):
    # the half length from which on the FP64 filter is a fast convolution, and either side
    from oracle import spectra as S
    s, pot = W.oscillators(43, 300.0, 1e-3)
    ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=0, seed=99, potential=qtb.POT_HARMONIC, ext={"omega": 0.02},
                  obs_stride=512, max_records=1)
    try:
        qtb.qtb_set_filter(ctx, 0, qtb.NOISE_QTB, 2 * K + 1, 0.3)
        qtb.qtb_step_n(ctx, 256)
        eta, blk = qtb.qtb_get_noise(ctx, 0, 129)
        ref = oracle.colored_block(99, 0, 129, 256, 256, S.taps(2 * K + 1, 1.0, 300.0, 0.3))
        assert blk == 1 and rel_inf(eta, ref.T) < 1e-12
    finally:
        qtb.qtb_destroy(ctx)
