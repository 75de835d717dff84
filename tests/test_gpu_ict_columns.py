"""The drop-tolerance IC's level sweeps on volumes of one to three voxels a column: their blocks follow
the (y, z) columns, up to one per SM and more, so there are far more of them than blocks of 256 voxels.
The kept fill goes beyond level 1, so that the pattern grows and the level sweeps run; per-iteration cost
and map against the oracle as in test_gpu_ict.py."""
import numpy as np
import pytest

from gpu_util import open_fm, to_np
from oracle import Oracle
from synth import make_volume

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 76, 64), (3, 80, 40)])
def test_more_columns_than_voxel_blocks(dims):
    vol = make_volume(*dims, ncoil=2, te=(0.0, 1.0, 2.3), snr_db=20.0, seed=14, fmax_hz=150.0, nblobs=3)
    o = Oracle.from_volume(vol)
    o.set_droptol(1e-2)
    ref = o.solve(niter=3, nls=5, precond=4)
    with open_fm(vol, "fp64", precond="ict", droptol=1e-2) as fm:
        w, cost = fm.solve(niter=3)
        assert len(fm.ict_pattern(planes=False)[0]) > 6
    np.testing.assert_allclose(cost, ref["cost"], rtol=1e-10)
    np.testing.assert_allclose(to_np(w), ref["w"], rtol=0, atol=1e-9)
