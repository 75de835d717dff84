"""The adjoint solve on support masks that leave one of the two IC(0) tiles of a dot-product unit (32
rows) empty.  The preconditioner's sweeps write no p there, so the sums must not read it: the context
first runs a solve on non-finite images under the full mask, which leaves NaN in its work buffers.
Against the oracle's direct solve.  The Hessians' condition numbers are at most 2.6e3: FP64 with a
relative residual of 1e-13 is within 3e-10 (1e-9 here), FP32 with 1e-6, and as much again from the
rounding of its phases, within 5e-3."""
import numpy as np
import pytest
import torch

from gpu_util import dev_inputs, to_dev, to_np
from oracle import Oracle
from paper_2005_08661_gb300 import FieldMap, FmError
from synth import make_volume

pytestmark = pytest.mark.gpu

NX, NY, NZ = 20, 40, 6  # tiles of 64 x 16 x 8: rows 0-15 and 16-31 are one unit, 32-39 the next


@pytest.fixture(scope="module")
def cases():
    vol = make_volume(NX, NY, NZ, ncoil=1, snr_db=20.0, seed=43, fmax_hz=120.0, nblobs=3)
    y = np.arange(NY)[None, :, None]
    out = []
    for rows in (y < 16, (y >= 16) & (y < 32), (y < 16) | (y >= 32), (y >= 16)):
        v = make_volume(NX, NY, NZ, ncoil=1, snr_db=20.0, seed=43, fmax_hz=120.0, nblobs=3)
        v.mask = (v.mask * rows).astype(np.uint8)
        o = Oracle.from_volume(v)
        w = o.solve(niter=150, nls=8)["w"]
        b = 2.0 * (w - vol.omega_true * v.mask) * v.mask
        out.append((v, w, b, o.implicit_gradient(w, b)[0]))
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_adjoint_reads_no_p_of_an_empty_tile(cases, prec):
    full = np.ones((NZ, NY, NX), np.uint8)
    with FieldMap(NX, NY, NZ, precision=prec) as fm:
        for vol, w, b, ref in cases:
            y, s, m = dev_inputs(vol, prec)
            fm.set_data(torch.full_like(y, float("nan")), s, vol.te, torch.from_numpy(full).cuda(), vol.beta)
            with pytest.raises(FmError):
                fm.solve(niter=2)
            fm.set_data(y, s, vol.te, m, vol.beta)
            tol = 1e-13 if prec == "fp64" else 1e-6
            lam, it, rr = fm.adjoint_solve(to_dev(w, prec), to_dev(b, prec), tol=tol, maxiter=3000)
            assert rr <= tol and it > 0
            err = np.linalg.norm(to_np(lam) - ref)
            assert err <= (1e-9 if prec == "fp64" else 5e-3) * np.linalg.norm(ref)
