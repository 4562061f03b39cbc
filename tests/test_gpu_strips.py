"""Set-up kernels that split their rows by size: the 9-point assembly in strips of two and eight rows
and the row-collapsed Galerkin product in strips of two and eight coarse rows (grids just past the
thresholds and ending inside a strip; strips of one row are the small grids of
test_gpu_setup_passes.py, whose checks are run here)."""
import pytest

import test_gpu_setup_passes as passes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(123, 1217, 0), (123, 1301, 1), (123, 7297, 0), (123, 7303, 1)])
def test_assembly(libmg, cuda, shape):
    passes.test_nine_point_assembly(libmg, cuda, shape)


@pytest.mark.parametrize("shape", [(121, 1217, 0), (121, 1235, 1), (121, 12977, 0), (121, 12981, 1)])
@pytest.mark.parametrize("five", [0, 1])
def test_galerkin(libmg, oracle, cuda, shape, five):
    passes.test_row_collapsed_galerkin(libmg, oracle, cuda, shape, five)
