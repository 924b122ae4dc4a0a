"""The tuner tries the lane count by size with every skin it tries.

A small FP64 context takes 128 lanes by size and then holds a table of one force unit (8
bytes) per bead-atom, a size that no other array of an 61-ion context has; the other lane
counts hold less.  Counted through the allocator the library is given: the default and
each of the four skins.  At constant pressure, where the lane count is not a choice, only the
skins are tried."""
import pytest

from helpers import gpu_params
from paper_1905_02521_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npt", [None, dict(pressure=0.0, mass=1e5, gamma=1e-3)])
def test_every_skin_meets_the_lanes_by_size(monkeypatch, npt):
    from paper_1905_02521_gb300 import build
    build.build()
    from paper_1905_02521_gb300 import qtb
    s, pot = W.mgo_system(2, 300.0)
    s = dict(s, pos=s["pos"][:, 3:], vel=s["vel"][:, 3:], types=s["types"][3:])
    sizes = []
    alloc, free = qtb._torch_allocator()
    cb = (qtb.ALLOC_FN(lambda n, user: (sizes.append(n), alloc(n, user))[1]), free)
    monkeypatch.setattr(qtb, "_torch_allocator", lambda: cb)
    _, info = qtb.qtb_autotune([s], gpu_params(pot, 1.0, precision=0, obs_stride=256, npt=npt), qtb.NOISE_WHITE, 1, 0.0,
                               n_blocks=1, equil_blocks=0)
    assert sizes.count(8 * 61) == 1 + 4
    assert info["n_tried"] == (1 + 4 if npt else 1 + 4 * 3)
