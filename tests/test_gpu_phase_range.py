"""FP32 literal curvature at field values of up to 2^24 turns between echoes.  Three coils (padded pairs)
and nine (lanes sharing a voxel) of which all but two are empty give the curvature of those two alone,
whose evaluator takes the phase through a 64-bit integer: the same fixed-point phase, so the values differ
by the rounding of their sums (1e-5 of the largest, as in test_gpu_many_coils.py)."""
import numpy as np
import pytest
import torch

from gpu_util import dev_inputs, to_np
from paper_2005_08661_gb300 import FieldMap
from synth import make_volume

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nc", [3, 9])
def test_curvature_far_from_zero_turns(nc):
    nx, ny, nz, te = 11, 9, 4, (0.0, 1.0, 2.3)
    vol = make_volume(nx, ny, nz, ncoil=2, te=te, snr_db=20.0, seed=8, fmax_hz=150.0, nblobs=3)
    y, s, m = dev_inputs(vol, "fp32")
    rng = np.random.default_rng(2)
    for turns in (0.3, 2.0 ** 21, 1.2 * 2.0 ** 22, 1.5 * 2.0 ** 23):  # over the longest spacing, at most
        w = torch.from_numpy((2 * np.pi * turns / 2.3 * rng.uniform(0.8, 1.0, (nz, ny, nx))).astype(np.float32)).cuda()
        d = []
        for n in (2, nc):
            yn = torch.zeros((3, n, nz, ny, nx), dtype=y.dtype, device="cuda")
            sn = torch.zeros((n, nz, ny, nx), dtype=s.dtype, device="cuda")
            yn[:, :2], sn[:2] = y, s
            with FieldMap(nx, ny, nz, ncoil=n, precision="fp32") as fm:
                fm.set_data(yn, sn, te, m, vol.beta)
                d.append(to_np(fm.cost_grad(w)[2]))
        assert np.abs(d[0]).max() > 0
        np.testing.assert_allclose(d[1], d[0], rtol=0, atol=1e-5 * np.abs(d[0]).max(), err_msg=f"{turns} turns")
