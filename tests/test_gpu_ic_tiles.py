"""The IC(0) sweeps on support masks that leave tiles and hyperplanes empty, against the
oracle's factor: one context goes through a list of masks (fm_set_data lists its non-empty
tiles anew each time), and each mask is factored and applied twice, so that a face entry left
behind by one launch would show in the next.  Tolerances as in test_gpu_parity.py: FP64 differs
by summation order only; FP32 carries the pivots as hi + lo floats and substitutes in float."""
import numpy as np
import pytest

from gpu_util import dev_inputs, to_dev, to_np
from oracle import ic0_factor, ic0_solve
from paper_2005_08661_gb300 import FieldMap
from synth import make_volume

pytestmark = pytest.mark.gpu

TOL = {"fp64": (1e-11, 1e-10), "fp32": (3e-5, 2e-4)}
SHAPES = [(97, 70, 35), (64, 33, 16), (31, 100, 9)]  # nx, ny, nz: ragged and exact 64 x 16 x 8 tiles


def _masks(nx, ny, nz):
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    rng = np.random.default_rng(5)
    one = np.zeros((nz, ny, nx), bool)
    one[nz // 2, ny // 2, nx // 2] = True
    corners = np.zeros_like(one)
    corners[::max(nz - 1, 1), ::max(ny - 1, 1), ::max(nx - 1, 1)] = True
    return {
        "one voxel": one,
        "corners": corners,
        "all": np.ones_like(one),
        "two slabs": (x < 5) | (x >= nx - 5),
        "layers": (z == 0) | (z == nz - 1) | (y % 16 == 15) | (x == 64),
        "staircase": np.abs(x * ny - y * nx) < 2 * nx,
        "sparse": rng.uniform(size=one.shape) < 0.01,
        "holes": rng.uniform(size=one.shape) < 0.9,
        "ball": (x - nx / 2) ** 2 / nx ** 2 + (y - ny / 2) ** 2 / ny ** 2 + (z - nz / 2) ** 2 / nz ** 2 < 0.12,
        "empty": np.zeros_like(one),
    }


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_sweeps_on_masks_with_empty_tiles_match_the_oracle(prec, shape):
    nx, ny, nz = shape
    vol = make_volume(nx, ny, nz, seed=3)
    y, s, _ = dev_inputs(vol, prec)
    rng = np.random.default_rng(11)
    tip, tp = TOL[prec]
    with FieldMap(nx, ny, nz, precision=prec) as fm:
        for name, m in _masks(*shape).items():
            mask = m.astype(np.uint8)
            fm.set_data(y, s, vol.te, to_dev(mask, "fp64").byte(), 0.5)
            for rep in range(2):
                d = rng.uniform(0.05, 2.0, size=mask.shape).astype(np.float32).astype(np.float64) * mask
                g = rng.standard_normal(mask.shape).astype(np.float32).astype(np.float64) * mask
                ip = to_np(fm.ic_factor_curv(to_dev(d, prec))).reshape(-1)
                p = to_np(fm.ic_apply(to_dev(g, prec))).reshape(-1)
                ip_ref, p_ref = np.zeros(mask.size), np.zeros(mask.size)
                if mask.any():
                    colptr, rowidx, val, umap = ic0_factor(mask.shape, mask, d, 0.5)
                    ip_ref[umap] = 1.0 / val[colptr[:-1]] ** 2
                    p_ref[umap] = ic0_solve(colptr, rowidx, val, g.reshape(-1)[umap])
                np.testing.assert_allclose(ip, ip_ref, rtol=tip, atol=0, err_msg=name)
                np.testing.assert_allclose(p, p_ref, rtol=0, atol=tp * max(np.abs(p_ref).max(), 1e-300), err_msg=name)
