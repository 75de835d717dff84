"""The line search's grid barrier over launches: its three counts take turns and its number runs on
from launch to launch, so a context that has already run any number of barriers (nls per launch)
must give bit for bit what a fresh one gives.  One block, and more blocks than SMs."""
import numpy as np
import pytest

from gpu_util import open_fm, to_np
from synth import make_volume

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [(9, 7, 2), (96, 80, 24)])
@pytest.mark.parametrize("nls", [1, 2, 3, 4])
def test_used_context_equals_fresh(size, nls):
    vol = make_volume(*size, ncoil=1, seed=5)
    fresh = open_fm(vol, "fp32", nls=nls)
    want = to_np(fresh.solve(niter=3)[0])
    fresh.close()
    used = open_fm(vol, "fp32", nls=nls)
    for first in (1, 2, 5):
        used.solve(niter=first)
        assert np.array_equal(to_np(used.solve(niter=3)[0]), want)
    used.close()
