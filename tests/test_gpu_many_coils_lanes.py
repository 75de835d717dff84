"""FP32 literal curvature of more than eight coils on either side of the mask size up to which eight
lanes share a voxel (2432 voxels for each coil above five, half as many with two echoes): every voxel
once, in a last group that is not whole too.  Against the FP64 mode with the tolerances of
test_gpu_many_coils.py."""
import numpy as np
import pytest

from gpu_util import open_fm, to_dev, to_np
from synth import make_volume

pytestmark = pytest.mark.gpu

TE = {2: (0.0, 2.5), 3: (0.0, 1.0, 2.3), 4: (0.0, 1.5, 4.0, 9.5)}


@pytest.mark.parametrize("size,nc,L", [((32, 19, 16), 9, 3), ((37, 263, 1), 9, 3), ((28, 19, 16), 12, 2),
                                       ((8513, 1, 1), 12, 2), ((120, 100, 7), 13, 3), ((131, 47, 13), 11, 4)])
def test_both_sides_of_the_shared_lanes(size, nc, L):
    vol = make_volume(*size, ncoil=nc, te=TE[L], snr_db=20.0, seed=40 + nc, fmax_hz=150.0, nblobs=3)
    vol.mask = np.ones_like(vol.mask)
    rng = np.random.default_rng(1)
    with open_fm(vol, "fp32") as fm, open_fm(vol, "fp64") as ref:
        w0 = to_np(ref.init_omega())
        w = (w0 + 0.05 * rng.standard_normal(w0.shape)).astype(np.float32)
        c, g, d = fm.cost_grad(to_dev(w, "fp32"))
        c_ref, g_ref, d_ref = ref.cost_grad(to_dev(w, "fp64"))
        g_ref, d_ref = to_np(g_ref), to_np(d_ref)
        assert c == pytest.approx(c_ref, rel=2e-6, abs=1e-6 * np.abs(d_ref).max())
        np.testing.assert_allclose(to_np(g), g_ref, rtol=0, atol=3e-5 * np.abs(g_ref).max())
        np.testing.assert_allclose(to_np(d), d_ref, rtol=0, atol=1e-5 * np.abs(d_ref).max())
        a, b = (to_np(t.solve(niter=2)[0]) for t in (fm, ref))
        atol = 1e-4 * np.abs(b - w0).max() + 2e-6 * max(np.abs(w0).max(), 1.0)
        np.testing.assert_allclose(a, b, rtol=0, atol=atol)
