"""The FP64 fast convolution and the tiled FP32 filter at the edges of their blocks:
taps around the lengths where either takes over, around multiples of a 256-step part
and of the 16 taps of a tile, ragged dof counts, and two systems of different length
(one of them short) in a context.  Tolerances: those of the coloured-noise parity test
(1e-12 of the RMS in FP64; FP32: 1e-5, the rounding of a sum of up to 2049 terms)."""
import numpy as np
import pytest

from helpers import gpu_ctx, rel_inf
from oracle import spectra as S
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


@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-5)])
@pytest.mark.parametrize("K", [7, 8, 15, 16, 63, 64, 255, 256, 257, 1024])
def test_noise_blocks_match_oracle_over_tap_counts(qtb, oracle, precision, tol, K):
    sizes = (7, 43)                          # 21 and 129 dofs: part of a tile, one past a padding
    lengths = (2 * K + 1, 2 * (K // 3) + 1)  # the second often below the take-over
    systems = []
    for n, T in zip(sizes, (100.0, 400.0)):
        s, pot = W.oscillators(n, T, 1e-3)
        systems.append(s)
    ctx = gpu_ctx(qtb, systems, pot, 1.0, precision=precision, filter_prec=1, seed=99, potential=qtb.POT_HARMONIC,
                  ext={"omega": 0.02}, obs_stride=512, max_records=1)
    try:
        for k, L in enumerate(lengths):
            qtb.qtb_set_filter(ctx, k, qtb.NOISE_QTB, L, 0.3)
        for n0 in (0, 512):
            qtb.qtb_step_n(ctx, n0 - qtb.qtb_get_step(ctx))
            for k, (n, L) in enumerate(zip(sizes, lengths)):
                eta, blk = qtb.qtb_get_noise(ctx, k, 3 * n)
                assert blk == n0 // 256
                ref = oracle.colored_block(99, k, 3 * n, n0, 256, S.taps(L, 1.0, systems[k]["T"], 0.3))
                assert rel_inf(eta, ref.T) < tol, (k, n0, rel_inf(eta, ref.T))
    finally:
        qtb.qtb_destroy(ctx)
