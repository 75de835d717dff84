"""The batch reports the back substitution's blocks per SM that run: FP64 tiles take more than half of an
SM's shared memory and run one, FP32 one or two; the autotuner names no count that does not fit."""
import numpy as np
import pytest

from gpu_util import dev_inputs, to_np
from synth import make_volume

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,most", [("fp64", 1), ("fp32", 2)])
def test_reported_blocks_fit(prec, most):
    from paper_2005_08661_gb300 import FieldMapBatch
    vols = [make_volume(nx, ny, nz, ncoil=1, snr_db=20.0, seed=5 + nx, fmax_hz=120.0, nblobs=3)
            for nx, ny, nz in ((40, 34, 9), (64, 48, 16))]
    b = FieldMapBatch([(v.nx, v.ny, v.nz, 1, v.necho) for v in vols], precision=prec)
    keep = [dev_inputs(v, prec) for v in vols]
    for k, (v, (y, s, m)) in enumerate(zip(vols, keep)):
        b.set_data(k, y, s, v.te, m, v.beta)
    ref = [to_np(w) for w in b.solve(niter=3)[0]]
    assert b.bwd_blocks_per_sm() == 1
    b.set_fraction(0.25)
    assert b.bwd_blocks_per_sm() == most
    for _ in range(4):
        b.autotune(niter_probe=2)
        assert 1 <= b.bwd_blocks_per_sm() <= most
    for w, r in zip(b.solve(niter=3)[0], ref):
        np.testing.assert_allclose(to_np(w), r, rtol=0, atol=(1e-9 if prec == "fp64" else 1e-3) * np.abs(r).max())
    b.close()
