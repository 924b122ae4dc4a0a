"""kappa_P solver where a block's elimination ends after 8 columns: grids whose last block
holds 8 nodes, one more and one less.  Tolerance as the solver's parity test."""
import numpy as np
import pytest

from oracle import spectra as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("P,n", [(2, 8), (2, 9), (8, 39), (3, 40), (4, 41), (8, 72)])
def test_last_block_of_eight(P, n):
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb
    F = qtb.qtb_kappa_solve(P, n, 1000.0, 1.0)
    ref = S.kappa_solve(P, n=n, ymax=1000.0, y0=1.0).F
    assert np.abs(F / ref - 1.0).max() < 1e-10
