"""What cd_detect_contacts_noalloc answers for what its kernel left behind (no
GPU needed: the function is called with the values themselves).  A barrier that
ran out is an error, not a contact set."""
import ctypes as C

import pytest

from paper_1104_3516_gb300 import _build, cd

# the device's values: grid laid out, or refused for the radius, a periodic axis, its cells;
# errors none, timeout, colours, candidates
GRID = [0, 1, 2, 3]
NONE, TIMEOUT, COLOURS, CANDIDATES = 0, 1, 2, 3


def outcome(grid, error, overflow, needed):
    f = C.CDLL(_build.build()).cd_noalloc_outcome
    n = C.c_int64(-7)
    return f(grid, error, overflow, needed, C.byref(n)), n.value


@pytest.mark.parametrize("error, overflow, status, count", [
    (NONE, 0, cd.CD_OK, 5), (NONE, 1, cd.CD_ERR_CAPACITY, 5), (CANDIDATES, 0, cd.CD_ERR_CAPACITY, 5),
    (CANDIDATES, 1, cd.CD_ERR_CAPACITY, 5), (TIMEOUT, 0, cd.CD_ERR_TIMEOUT, -7), (TIMEOUT, 1, cd.CD_ERR_TIMEOUT, -7),
    (COLOURS, 0, cd.CD_ERR_STATE, 5)])
def test_what_the_kernel_left(error, overflow, status, count):
    assert outcome(0, error, overflow, 5) == (status, count)


@pytest.mark.parametrize("grid", GRID[1:])
@pytest.mark.parametrize("error", [NONE, TIMEOUT])
def test_a_refused_grid_comes_first(grid, error):
    assert outcome(grid, error, 0, 5) == (cd.CD_ERR_INVALID_ARG, -7)
