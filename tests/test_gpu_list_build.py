"""Neighbour-list build: rows too full to park their shell entries, cells shared by CTAs.

* A sparse box with one dense cluster: the list capacity follows the mean density, so the
  rows of the cluster's middle are nearly full and are listed by the second scan, while
  those of its corners are not.  Forces, energy and virial against the oracle.
* A thick skin: more than 128 parked entries a row, moved in several batches.
Tolerances: tests/tolerances.py, derived for these forces.
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


def _cluster(edge, side, spacing):
    pot = W.mgo_potential()
    g = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 3)
    pos = 3.0 + spacing * g + np.random.default_rng(11).normal(0.0, 0.05, g.shape)
    types = (g.sum(1) % 2).astype(np.int32)
    return W.system(np.mod(pos, edge), types, np.array([edge] * 3), pot, 300.0, 1e-3), pot


def _check(qtb, oracle, s, pot, precision, **kw):
    ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=precision, **kw)
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
    finally:
        qtb.qtb_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("side,spacing", [(5, 2.7), (4, 2.7)])
def test_nearly_full_rows(qtb, oracle, precision, side, spacing):
    edge, r_list = 25.0, 8.8
    s, pot = _cluster(edge, side, spacing)
    # the case the test is for: rows of n + m entries within a capacity that cannot park m
    x = s["pos"][0]
    dd = x[None] - x[:, None]
    r = np.sqrt(((dd - edge * np.round(dd / edge)) ** 2).sum(-1)) + 99.0 * np.eye(len(x))
    n, tot = (r < 8.0).sum(1), (r < r_list).sum(1)
    cap = -(-int(np.ceil(1.5 * len(x) / edge ** 3 * 4.0 / 3.0 * np.pi * r_list ** 3 + 64.0)) // 64) * 64
    assert tot.max() <= cap
    assert (-(-n // 64) * 64 > cap - (tot - n)).any() == (side == 5)
    _check(qtb, oracle, s, pot, precision)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("ncell", [3, 5])
def test_thick_skin(qtb, oracle, precision, ncell):
    s, pot = W.mgo_system(ncell, 300.0, sigma=0.06, seed=60 + ncell)
    assert len(s["types"]) / s["box"].prod() * 4.0 / 3.0 * np.pi * (10.0 ** 3 - 8.0 ** 3) > 160
    _check(qtb, oracle, s, pot, precision, skin=2.0)
