"""The pair-force step kernel at the edges of its list blocks, lane counts and variants.

* the lane count (8, 16, 32, or the default by size: 128 here) changes no bit of a
  trajectory, with list rebuilds in it, in both forms, for one bead and ring polymers;
* forces, energy and virial against the oracle with lists shorter than one 64-entry
  block, around one and of several, with the damping at zero, at the workloads' value
  and beyond the range of the polynomial Coulomb term (alpha r_cut = 2.8: the
  exponential form takes over), in cubic and orthorhombic cells (minimum image or
  image bits).  Tolerances: tests/tolerances.py, derived for these forces.
"""
import numpy as np
import pytest

from helpers import gpu_ctx, rel_inf, rel_l2
from paper_1905_02521_gb300 import workloads as W
from tolerances import F32_INF, F32_L2, F64_TOL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qtb():
    import torch
    assert torch.cuda.is_available()
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb as q
    return q


def _ragged(ncell, P, T, drop):
    s, pot = W.mgo_system(ncell, T, n_beads=P)
    keep = np.setdiff1d(np.arange(s["pos"].shape[1]), np.arange(drop) * 7)
    return dict(s, pos=s["pos"][:, keep], vel=s["vel"][:, keep], types=s["types"][keep]), pot


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncell,P,drop", [(2, 1, 3), (3, 1, 5), (2, 3, 1)])
def test_lane_count_changes_no_bit(qtb, precision, ncell, P, drop):
    s, pot = _ragged(ncell, P, 1500.0, drop)
    out = []
    for lanes in (16, 0, 8, 32):
        ctx = gpu_ctx(qtb, [s], pot, 2.0, precision=precision, seed=5, list_lanes=lanes, obs_stride=50, skin=0.3)
        try:
            qtb.qtb_step_n(ctx, 300)
            out.append(qtb.qtb_get_state(ctx, 0, P, len(s["types"])) + (qtb.qtb_get_series(ctx, 0, 6),))
            assert qtb.qtb_list_rebuilds(ctx) > 3
        finally:
            qtb.qtb_destroy(ctx)
    for o in out[1:]:
        for a, b in zip(o, out[0]):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncell,r_cut,alpha,strain", [
    (2, 2.6, 0.2, 1.0), (2, 5.0, 0.2, 1.0), (3, 8.0, 0.0, 1.0), (3, 8.0, 0.35, 1.0), (5, 8.0, 0.35, 1.0),
    (5, 8.0, 0.2, 1.03), (3, 8.0, 0.2, 1.03), (5, 8.0, 0.2, 1.0)])
def test_forces_over_list_lengths_and_variants(qtb, oracle, precision, ncell, r_cut, alpha, strain):
    s, pot = W.mgo_system(ncell, 300.0, sigma=0.06, seed=50 + ncell)
    f = np.array([strain, 1.0, 1.0 / strain])
    s = dict(s, pos=s["pos"] * f, box=s["box"] * f)
    pot = dict(pot, r_cut=r_cut, dsf_alpha=alpha)
    ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=precision)
    try:
        N = len(s["types"])
        x, _ = qtb.qtb_get_state(ctx, 0, 1, N)
        fo, eo, vo = oracle.pair_forces(x[0], s["types"], s["box"], pot)
        fg = qtb.qtb_get_forces(ctx, 0, 1, N)[0]
        obs = qtb.qtb_observables(ctx, 0)
        if precision == 0:
            assert rel_inf(fg, fo) < F64_TOL
            tol = F64_TOL
        else:
            assert rel_l2(fg, fo) < F32_L2 and rel_inf(fg, fo) < F32_INF, (rel_l2(fg, fo), rel_inf(fg, fo))
            tol = F32_L2
        assert obs[2] == pytest.approx(eo, rel=10 * tol, abs=10 * tol)
        assert np.allclose(obs[5:14].reshape(3, 3), vo, rtol=10 * tol, atol=10 * tol * np.abs(vo).max())
        # the plain step variant (not recorded) starts from the same forces
        qtb.qtb_step_n(ctx, 0)
        assert np.array_equal(qtb.qtb_get_forces(ctx, 0, 1, N)[0], fg)
    finally:
        qtb.qtb_destroy(ctx)
