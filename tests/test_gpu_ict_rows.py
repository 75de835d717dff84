"""The row wavefront of the drop-tolerance IC (base fill pattern) at the edges of its row groups of
32: shapes with whole, ragged and single groups, masks that leave groups and planes empty, one
context through all of them and two factorisations of each mask, so that a record left behind by
one launch would show in the next.  Against the oracle's factor; tolerances as in test_gpu_ict.py
(FP64 differs by summation order only, FP32 rounds d, g and p to float)."""
import numpy as np
import pytest
import scipy.sparse as sp
from scipy.sparse.linalg import spsolve_triangular

from gpu_util import dev_inputs, to_dev, to_np
from oracle import ict_factor
from paper_2005_08661_gb300 import FieldMap
from synth import make_volume

pytestmark = pytest.mark.gpu

SHAPES = [(9, 70, 4), (40, 33, 3), (5, 32, 6), (66, 3, 2)]  # nx, ny, nz
BETA, DROP = 0.3, 0.007  # level-1 fill kept, none deeper


def _masks(nx, ny, nz):
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    rng = np.random.default_rng(7)
    one = np.zeros((nz, ny, nx), bool)
    one[nz - 1, ny - 1, nx // 2] = True
    return {
        "all": np.ones_like(one),
        "one voxel": one,
        "no middle rows": (y < 20) | (y >= 64),
        "planes apart": (z == 0) | (z == nz - 1),
        "sparse": rng.uniform(size=one.shape) < 0.1,
        "holes": rng.uniform(size=one.shape) < 0.85,
        "diagonal": np.abs(x - y % nx) < 2,
        "empty": np.zeros_like(one),
    }


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape", SHAPES)
def test_row_wavefront_matches_the_oracle_factor(prec, shape):
    nx, ny, nz = shape
    vol = make_volume(nx, ny, nz, seed=4)
    y, s, _ = dev_inputs(vol, prec)
    rng = np.random.default_rng(13)
    tol = 1e-11 if prec == "fp64" else 2e-4
    with FieldMap(nx, ny, nz, precision=prec, precond="ict", droptol=DROP) as fm:
        for name, m in _masks(*shape).items():
            mask = m.astype(np.uint8)
            fm.set_data(y, s, vol.te, to_dev(mask, "fp64").byte(), BETA)
            cnt = np.zeros(mask.shape)
            for ax in range(3):
                e = m & np.roll(m, -1, ax)
                e[tuple(slice(-1, None) if k == ax else slice(None) for k in range(3))] = False
                cnt += e.astype(int) + np.roll(e, 1, ax)
            for _ in range(2):
                d = rng.uniform(0.3, 3.0, size=mask.shape).astype(np.float32).astype(np.float64) * m
                g = rng.standard_normal(mask.shape).astype(np.float32).astype(np.float64) * m
                ip = to_np(fm.ic_factor_curv(to_dev(d, prec))).reshape(-1)
                p = to_np(fm.ic_apply(to_dev(g, prec))).reshape(-1)
                ip_ref, p_ref = np.zeros(mask.size), np.zeros(mask.size)
                if m.any():
                    tau = DROP * max((d + BETA * cnt)[m].max(), BETA if cnt.any() else 0.0)
                    colptr, rowidx, val, umap = ict_factor(mask.shape, mask, d, BETA, tau)
                    L = sp.csc_matrix((val, rowidx, colptr), shape=(umap.size, umap.size)).tocsr()
                    ip_ref[umap] = 1.0 / L.diagonal() ** 2
                    v = spsolve_triangular(L, g.reshape(-1)[umap], lower=True)
                    p_ref[umap] = spsolve_triangular(L.T.tocsr(), v, lower=False)
                assert np.max(np.abs(ip - ip_ref)) <= tol * max(np.abs(ip_ref).max(), 1e-300), name
                assert np.max(np.abs(p - p_ref)) <= tol * max(np.abs(p_ref).max(), 1e-300), name
                assert len(fm.ict_pattern(planes=False)[0]) == 6, name  # the base pattern held
