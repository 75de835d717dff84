"""Device memory of the drop-tolerance IC.  The row wavefront's exchange buffer serves the base pattern
only and for speed alone, so it goes when the pattern grows, or when another of the context's buffers
would not fit beside it."""
import contextlib
import gc

import numpy as np
import pytest
import torch

from gpu_util import dev_inputs, open_fm, to_np
from paper_2005_08661_gb300 import FieldMap
from synth import make_volume

pytestmark = pytest.mark.gpu

MB = 1 << 20
TE = (0.0, 1.0, 2.3)


def _free():
    gc.collect()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


@contextlib.contextmanager
def _left(nbytes):
    """All device memory but about nbytes is taken."""
    hog = [torch.empty(_free() - nbytes, dtype=torch.uint8, device="cuda")]
    try:
        yield
    finally:
        hog.clear()
        _free()  # out of torch's cache too


def _grow_a_pattern():
    """Loads the level sweeps, and with them the device's local memory for their rows of 64 entries."""
    vol = make_volume(45, 33, 9, ncoil=4, te=TE, snr_db=20.0, seed=11, fmax_hz=150.0, nblobs=3)
    with open_fm(vol, "fp64", precond="ict", droptol=1e-3) as fm:
        fm.ic_factor(fm.init_omega())
        assert len(fm.ict_pattern(planes=False)[0]) > 6


def test_a_grown_pattern_gives_the_exchange_buffer_back():
    _grow_a_pattern()
    vol = make_volume(128, 96, 32, ncoil=2, te=TE, snr_db=20.0, seed=11, fmax_hz=150.0, nblobs=3)
    nv = vol.mask.size
    with open_fm(vol, "fp32", precond="ict", droptol=1e-3) as fm:  # its factor keeps 25 offsets
        w = fm.init_omega()
        before = _free()
        fm.ic_factor(w, want_pivots=False)
        took = before - _free()
        nh = len(fm.ict_pattern(planes=False)[0])
    assert nh > 6
    # a plane of doubles per offset more, and at least one record of six doubles a voxel less
    assert took <= (nh - 6) * 8 * nv - 48 * nv + 8 * MB


def test_the_exchange_buffer_makes_room_for_the_start_map():
    """A solve from a given map keeps a copy of it (the pattern may grow and the solve run again), here
    twice as large as what is left beside the context."""
    vol = make_volume(128, 128, 128, ncoil=1, snr_db=20.0, seed=12, fmax_hz=150.0, nblobs=3)
    y, s, m = dev_inputs(vol, "fp64")
    with FieldMap(vol.nx, vol.ny, vol.nz, precision="fp64", precond="ict") as fm:
        fm.set_data(y, s, vol.te, m, vol.beta)
        start = 1.01 * fm.init_omega()
    with FieldMap(vol.nx, vol.ny, vol.nz, precision="fp64", precond="ict") as fm:
        fm.set_data(y, s, vol.te, m, vol.beta)
        ref = to_np(fm.solve(start.clone(), niter=2)[0])
    with FieldMap(vol.nx, vol.ny, vol.nz, precision="fp64", precond="ict") as fm:
        fm.set_data(y, s, vol.te, m, vol.beta)
        fm.solve(niter=2)
        inout = start.clone()
        _grow_a_pattern()
        with _left(8 * MB):
            fm.solve_into(inout, False, 2)
        w = to_np(inout)
    # the two routes of the factor differ by the order of their sums
    np.testing.assert_allclose(w, ref, rtol=0, atol=1e-9)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_without_room_for_the_exchange_buffer_the_level_sweeps_hold_the_base_pattern(prec):
    """A context that opens with too little memory for the exchange buffer gives the factor and the
    substitutions of one that has it, alone and in a solve.  Tolerances as in test_gpu_ict_rows.py."""
    nx, ny, nz, beta, drop = 160, 128, 64, 0.3, 0.007  # level-1 fill kept, none deeper
    vol = make_volume(nx, ny, nz, ncoil=1, snr_db=20.0, seed=4, fmax_hz=120.0, nblobs=3)
    y, s, m = dev_inputs(vol, prec)
    rng = np.random.default_rng(13)
    dt = torch.float64 if prec == "fp64" else torch.float32
    d = torch.from_numpy(rng.uniform(0.3, 3.0, size=vol.mask.shape)).cuda().to(dt)
    g = torch.from_numpy(rng.standard_normal(vol.mask.shape)).cuda().to(dt)

    def run(fm):
        fm.set_data(y, s, vol.te, m, beta)
        ip = to_np(fm.ic_factor_curv(d))
        p = to_np(fm.ic_apply(g))
        assert len(fm.ict_pattern(planes=False)[0]) == 6
        return ip, p, to_np(fm.solve(niter=2)[0])

    _grow_a_pattern()
    before = _free()
    with FieldMap(nx, ny, nz, precision=prec, precond="ict", droptol=drop) as fm:
        whole = before - _free()
        ref = run(fm)
    short = whole - 40 * vol.mask.size  # the exchange buffer has at least 48 bytes a voxel
    with _left(short):
        fm = FieldMap(nx, ny, nz, precision=prec, precond="ict", droptol=drop)
    got = run(fm)
    fm.close()
    tol = 1e-11 if prec == "fp64" else 2e-4
    for a, b in zip(got[:2], ref[:2]):
        assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b))
    move = np.abs(ref[2] - to_np(_start(vol, y, s, m, beta, prec))).max()
    assert np.max(np.abs(got[2] - ref[2])) <= (1e-9 if prec == "fp64" else 1e-4 * move)


def _start(vol, y, s, m, beta, prec):
    with FieldMap(vol.nx, vol.ny, vol.nz, precision=prec) as fm:
        fm.set_data(y, s, vol.te, m, beta)
        return fm.init_omega()
