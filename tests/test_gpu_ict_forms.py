"""The drop-tolerance IC's base pattern where the factor, or both sweeps, go by levels: volumes with many
planes of several row groups.  As test_gpu_ict_rows.py, whose shapes go by rows: masks that leave groups and
planes empty, two factorisations of each, against the oracle's factor with its tolerances."""
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
