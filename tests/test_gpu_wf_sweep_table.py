"""The voxel-wise water-fat sweep at the edges of its table of field values (256 entries filled by a
block at a time) and with more mask voxels than threads in the grid, against the FP64 oracle.

FP64 mode's choices are the oracle's except where the two candidates' costs tie to rounding (1e-11
of the cost, as for the sweep of 100 values)."""
import numpy as np
import pytest

from gpu_util import dev_inputs, to_np
from oracle import Oracle, wf_gamma
from synth import make_wf_volume

pytestmark = pytest.mark.gpu


def _check(nx, ny, nz, ncoil, counts):
    from paper_2005_08661_gb300 import FieldMap
    vol = make_wf_volume(nx, ny, nz, ncoil=ncoil, seed=71, snr_db=20.0, fmax_hz=150.0, nblobs=3)
    amps, freqs = vol.meta["fat_amps"], vol.meta["fat_freqs_khz"]
    o = Oracle.from_volume(vol)
    o.set_gamma(wf_gamma(vol.te, amps, freqs)[1])
    fm = FieldMap(nx, ny, nz, ncoil=ncoil, necho=vol.necho, precision="fp64")
    fm.set_fat_model(amps, freqs)
    y, s, m = dev_inputs(vol, "fp64")
    fm.set_data(y, s, vol.te, m, vol.beta)
    m = vol.mask > 0
    for n in counts:
        ws, wt = to_np(fm.wf_sweep(n, -1.1, 1.4)), o.wf_sweep(n, -1.1, 1.4)
        assert np.all(ws[~m] == 0)
        d = m & (np.abs(ws - wt) > 1e-14)
        assert d.sum() <= max(1, m.sum() // 1000)
        pg, po = o.phi_vox(ws), o.phi_vox(wt)
        assert np.all(np.abs(pg[d] - po[d]) <= 1e-11 * np.abs(po[d]) + 1e-14)
    fm.close()
    return int(m.sum())


@pytest.mark.parametrize("ncoil", [1, 2])
def test_counts_around_the_table(ncoil):
    _check(23, 17, 5, ncoil, (1, 2, 255, 256, 257, 513))


def test_more_voxels_than_threads():
    assert _check(160, 128, 32, 1, (3, 258)) > 4 * 152 * 256
