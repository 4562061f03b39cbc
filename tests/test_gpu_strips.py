"""Set-up kernels that split their rows by size: the 9-point assembly in strips of two and eight rows
(grids just past the thresholds and ending inside a strip; strips of one row are the small grids of
test_gpu_setup_passes.py, whose checks are run here)."""
import pytest

import test_gpu_setup_passes as passes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(123, 1217, 0), (123, 1301, 1), (123, 7297, 0), (123, 7303, 1)])
def test_assembly(libmg, cuda, shape):
    passes.test_nine_point_assembly(libmg, cuda, shape)
