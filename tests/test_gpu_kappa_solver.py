"""The kappa_P solver and the learned model's gradient at the edges of their tiles:
collocation grids below, at and above multiples of the 32-column tiles (one tile, two,
many; terms formed in place on small grids), and sample counts around the 64 of a CTA.
Tolerances: 1e-10 relative per node, as the solver's parity test (the refined
solution's error is ~cond(A) eps <= 1e-11); gradient 1e-4 of its RMS, as the model's."""
import numpy as np
import pytest

from oracle import mlp as OM
from oracle import spectra as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def qtb():
    import torch
    assert torch.cuda.is_available()
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb as q
    return q


@pytest.mark.parametrize("P,n", [(2, 8), (5, 31), (3, 32), (32, 33), (7, 64), (4, 65), (8, 130), (16, 333)])
def test_solver_over_grid_sizes(qtb, P, n):
    F = qtb.qtb_kappa_solve(P, n, 1000.0, 1.0)
    ref = S.kappa_solve(P, n=n, ymax=1000.0, y0=1.0).F
    assert np.abs(F / ref - 1.0).max() < 1e-10


@pytest.mark.parametrize("n", [1, 63, 64, 65, 1000])
def test_gradient_over_sample_counts(qtb, n):
    m = qtb.qtb_kappa_model_create(seed=4)
    try:
        w = qtb.qtb_kappa_model_get_weights(m).astype(np.float64)
        rng = np.random.default_rng(n)
        x = OM.features(np.sinh(rng.uniform(0, np.arcsinh(1000.0), n)), rng.integers(2, 33, n))
        t = rng.uniform(0.2, 1.0, n)
        loss, g = qtb.qtb_kappa_model_grad(m, x, t)
        loss_o, g_o = OM.loss_and_grad(w, x.astype(np.float32).astype(np.float64), t.astype(np.float32))
        assert loss == pytest.approx(loss_o, rel=1e-5)
        assert np.abs(g - g_o).max() < 1e-4 * np.sqrt((g_o ** 2).mean())
    finally:
        qtb.qtb_kappa_model_destroy(m)
