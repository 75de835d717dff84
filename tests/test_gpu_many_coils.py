"""FP32 literal curvature outside the register-resident coil counts: up to eight coils padded to
an even count (any number of echoes), and more than eight with eight lanes per voxel.  Coil counts
and mask sizes sit where the padding, the blocks of eight and four coils and the groups of four
voxels leave remainders.  Cost, gradient and curvature against the oracle with the FP32 tolerances
of test_gpu_parity.py; the line search through the map after two iterations, against the FP64 mode:
a step is a ratio of sums whose terms carry the gradient's 3e-5, so the map agrees to 1e-4 of the
distance moved, beside the start map's 2e-6."""
import numpy as np
import pytest

from gpu_util import open_fm, to_dev, to_np
from oracle import Oracle
from synth import make_volume

pytestmark = pytest.mark.gpu

TE = {2: (0.0, 2.5), 3: (0.0, 1.0, 2.3), 4: (0.0, 1.5, 4.0, 9.5)}
CASES = [
    # nx, ny, nz, coils, echoes
    (13, 9, 10, 3, 2),
    (11, 7, 5, 4, 4),
    (9, 8, 7, 5, 3),
    (7, 6, 5, 6, 4),
    (10, 9, 3, 7, 2),
    (9, 7, 5, 8, 4),
    (8, 7, 6, 9, 3),
    (33, 5, 4, 12, 3),
    (6, 5, 5, 13, 4),
    (17, 9, 4, 16, 2),
    (10, 9, 6, 32, 3),
    (1, 1, 1, 31, 3),
    (2, 3, 1, 20, 4),
]


def _vol(nx, ny, nz, nc, L):
    v = make_volume(nx, ny, nz, ncoil=nc, te=TE[L], snr_db=20.0, seed=40 + nc, fmax_hz=150.0, nblobs=3)
    rng = np.random.default_rng(nc)
    v.mask = (rng.uniform(size=v.mask.shape) < 0.8).astype(np.uint8)
    v.mask[0, 0, 0] = 1
    return v


@pytest.mark.parametrize("case", CASES)
def test_data_term_and_line_search_for_any_coil_count(case):
    vol = _vol(*case)
    o = Oracle.from_volume(vol)
    rng = np.random.default_rng(1)
    w = (o.init() + 0.05 * rng.standard_normal(vol.mask.shape)) * vol.mask
    with open_fm(vol, "fp32") as fm, open_fm(vol, "fp64") as ref:
        cost, g, d = fm.cost_grad(to_dev(w, "fp32"))
        g_ref, d_ref = o.grad(w), o.curv(w)
        assert cost == pytest.approx(o.cost(w), rel=2e-6, abs=1e-6 * np.abs(d_ref).max())
        np.testing.assert_allclose(to_np(g), g_ref, rtol=0, atol=3e-5 * np.abs(g_ref).max())
        np.testing.assert_allclose(to_np(d), d_ref, rtol=0, atol=1e-5 * np.abs(d_ref).max())
        a, b, w0 = (to_np(t) for t in (fm.solve(niter=2)[0], ref.solve(niter=2)[0], ref.init_omega()))
        atol = 1e-4 * np.abs(b - w0).max() + 2e-6 * max(np.abs(w0).max(), 1.0)
        np.testing.assert_allclose(a, b, rtol=0, atol=atol)
