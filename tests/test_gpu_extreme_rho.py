"""FP64 pair forces with Buckingham lengths at the ends of the exponent's range.

e^{-r/rho} of a tiny rho is zero at every distance (its exponent in units of ln 2 does not
fit 32 bits below rho ~ 5e-9 A), that of a negative rho grows with distance.  Both are
accepted, and the forces are the oracle's (tests/tolerances.py).
"""
import numpy as np
import pytest

from helpers import gpu_ctx, rel_inf
from paper_1905_02521_gb300 import workloads as W
from tolerances import F64_TOL

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rho", [1e-12, 1e-10, 3e-9, 6e-9, 1e-3, -0.05, -1.0])
def test_forces_over_lengths(oracle, rho):
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb
    s, pot = W.mgo_system(3, 300.0, sigma=0.06, seed=51)
    r = pot["buck_rho"].copy()
    r[0, 1] = r[1, 0] = rho
    A = pot["buck_A"].copy()
    if rho < 0:
        A[0, 1] = A[1, 0] = 1e-3 * np.exp(8.0 / rho)   # (a term of the size of the others)
    pot = dict(pot, buck_rho=r, buck_A=A)
    ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=0)
    try:
        N = len(s["types"])
        x, _ = qtb.qtb_get_state(ctx, 0, 1, N)
        fo, eo, _ = oracle.pair_forces(x[0], s["types"], s["box"], pot)
        assert rel_inf(qtb.qtb_get_forces(ctx, 0, 1, N)[0], fo) < F64_TOL
        assert qtb.qtb_observables(ctx, 0)[2] == pytest.approx(eo, rel=10 * F64_TOL)
    finally:
        qtb.qtb_destroy(ctx)
