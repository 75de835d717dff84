"""The drop-tolerance IC's base pattern where the factor, or both sweeps, go by levels: volumes with many
planes of several row groups.  As test_gpu_ict_rows.py, whose shapes go by rows: masks that leave groups and
planes empty, two factorisations of each, against the oracle's factor with its tolerances."""
import numpy as np
import pytest

from test_gpu_ict_rows import test_row_wavefront_matches_the_oracle_factor as matches_the_oracle_factor

pytestmark = pytest.mark.gpu

# nx, ny, nz: 64 (nz + 2) + nx steps by rows, nx + 2 ny + 3 nz levels
FACTOR_BY_LEVELS = [(5, 33, 40), (24, 40, 60)]
BY_LEVELS = [(3, 33, 150), (9, 34, 120)]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", FACTOR_BY_LEVELS + BY_LEVELS)
def test_levels_match_the_oracle_factor(prec, shape):
    matches_the_oracle_factor(prec, shape)


@pytest.mark.parametrize("fraction", [1.0, 0.125])
def test_a_batch_of_every_form_gives_each_volume_its_own_solve(fraction):
    from gpu_util import dev_inputs, open_fm
    from paper_2005_08661_gb300 import FieldMapBatch
    from synth import make_volume

    vols = [make_volume(*dims, ncoil=2, te=(0.0, 1.0, 2.3), snr_db=20.0, seed=20, fmax_hz=150.0, nblobs=3)
            for dims in ((40, 33, 3), FACTOR_BY_LEVELS[1], BY_LEVELS[1])]
    refs = []
    for v in vols:
        with open_fm(v, "fp64", precond="ict", droptol=1e-2) as fm:
            refs.append(fm.solve(niter=3)[1])
    b = FieldMapBatch([(v.nx, v.ny, v.nz, v.ncoil, v.necho) for v in vols], precision="fp64", precond="ict",
                      droptol=1e-2)
    b.set_fraction(fraction)
    keep = [dev_inputs(v, "fp64") for v in vols]
    for k, (v, (y, s, m)) in enumerate(zip(vols, keep)):
        b.set_data(k, y, s, v.te, m, v.beta)
    for _ in range(2):
        for cost, ref in zip(b.solve(niter=3)[1], refs):
            np.testing.assert_allclose(cost, ref, rtol=1e-10)
    b.close()
