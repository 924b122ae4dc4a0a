"""External potentials: records against sums over the state read back, for system sizes of
part of a unit (32 atoms), one, and thousands of units.  K, <x^2>, momentum and the trace of
the virial are sums in FP64 of the stored values: 1e-12 relative of the sum of their terms'
sizes; V holds a rounding of each FP32 term in the mixed form: 1e-6."""
import numpy as np
import pytest

from helpers import gpu_ctx
from paper_1905_02521_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,P", [(1, 1), (33, 1), (31, 5), (40, 8), (200001, 1), (50001, 2), (20001, 8)])
def test_records_are_the_states_sums(precision, n, P):
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb
    s = W.oscillators(n, 120.0, 4e-3, n_beads=P, x0=0.4, spread=0.1, seed=5)[0]
    V0, a, m = 0.1, 0.5, 1.008
    ctx = gpu_ctx(qtb, [s], W.well_potential(), 0.5, precision=precision, filter_prec=1, seed=3,
                  potential=qtb.POT_DOUBLEWELL, ext={"V0": V0, "a": a}, obs_stride=3, max_records=8)
    try:
        qtb.qtb_step_n(ctx, 9)
        x, v = qtb.qtb_get_state(ctx, 0, P, n)
        rec = qtb.qtb_get_series(ctx, 0, 8)[-1]
    finally:
        qtb.qtb_destroy(ctx)
    u = x * x / a ** 2 - 1
    f = -4 * V0 * u * x / a ** 2
    tol = 1e-12 if precision == 0 else 1e-6
    sums = {1: (0.5 * m * W.MVV2E * v * v, 1e-12), 2: (V0 * u * u / P, tol), 17: (x * x / P, 1e-12),
            14: (m * v[..., 0], 1e-12), 15: (m * v[..., 1], 1e-12), 16: (m * v[..., 2], 1e-12),
            5: (x[..., 0] * f[..., 0] / P, tol), 9: (x[..., 1] * f[..., 1] / P, tol), 13: (x[..., 2] * f[..., 2] / P, tol)}
    assert rec[0] == 9
    for q, (t, tl) in sums.items():
        assert abs(rec[q] - t.sum()) < tl * np.abs(t).sum(), (q, rec[q], t.sum())
    if P > 1:
        wP = np.sqrt(P) * W.KB * 120.0 / 0.6582119569
        assert rec[3] == pytest.approx((0.5 * m * W.MVV2E * wP ** 2 * (x - np.roll(x, -1, 0)) ** 2).sum(),
                                       rel=1e-8 if precision == 0 else 1e-4)
