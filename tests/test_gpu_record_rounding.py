"""FP32 form: rounding of the energy and virial records.

Both are sums over all pairs, in which the rounding of a constant does not average out.  The
form holds positions exactly, in units of the edge times 2^-30, and that unit in FP32: its
configuration is the oracle's at an edge changed by that rounding.  Against it
* the energy is within half a unit in the last place of an FP32 number, 2^-24 relative;
* the trace of the virial is within what a change of all lengths by 2^-26, a quarter of a
  unit, does to it (their terms are some 50 times their sum; a single constant of the pair
  term off by its rounding already does more).
"""
import numpy as np
import pytest

from helpers import gpu_ctx
from paper_1905_02521_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("make", [W.mgo_system, W.lih_system])
@pytest.mark.parametrize("ncell,P", [(4, 1), (5, 1), (3, 1), (4, 4)])
def test_energy_and_virial(oracle, make, ncell, P):
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb
    for seed in (1, 2, 3):
        s, pot = make(ncell, 300.0, n_beads=P, seed=seed)
        ctx = gpu_ctx(qtb, [s], pot, 1.0, precision=1)
        try:
            N = len(s["types"])
            x, _ = qtb.qtb_get_state(ctx, 0, P, N)
            rec = qtb.qtb_observables(ctx, 0)
            unit = s["box"] / 2.0 ** 30
            f = np.float32(unit).astype(np.float64) / unit
            h = 1e-6

            def ref(scale):
                out = [oracle.pair_forces(x[b] * scale, s["types"], s["box"] * scale, pot)[1:] for b in range(P)]
                return np.mean([e for e, _ in out]), np.mean([np.trace(np.reshape(v, (3, 3))) for _, v in out])

            (E, T), Tp, Tm = ref(f), ref(1 + h)[1], ref(1 - h)[1]
            sens = abs((Tp - Tm) / (2 * h) / T)
            dE, dT = rec[2] / E - 1, (rec[5] + rec[9] + rec[13]) / T - 1
            print("V %+.1e  W %+.1e of %.1e" % (dE, dT, sens * 2.0 ** -26))
            assert abs(dE) < 2.0 ** -24, (seed, dE)
            assert abs(dT) < sens * 2.0 ** -26, (seed, dT)
        finally:
            qtb.qtb_destroy(ctx)
