"""Set-up kernels that split their rows, or choose their arithmetic, by size: the 9-point assembly in
strips of two and eight rows and the row-collapsed Galerkin product in strips of two and eight coarse
rows (grids just past the thresholds and ending inside a strip; strips of one row are the small grids of
test_gpu_setup_passes.py, whose checks are run here), and operator copies large enough for the
integer conversion (test_gpu_conversions.py's values)."""
import ctypes as C

import numpy as np
import pytest

import test_gpu_conversions as conversions
import test_gpu_setup_passes as passes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(123, 1217, 0), (123, 1301, 1), (123, 7297, 0), (123, 7303, 1)])
def test_assembly(libmg, cuda, shape):
    passes.test_nine_point_assembly(libmg, cuda, shape)


@pytest.mark.parametrize("shape", [(121, 1217, 0), (121, 1235, 1), (121, 12977, 0), (121, 12981, 1)])
@pytest.mark.parametrize("five", [0, 1])
def test_galerkin(libmg, oracle, cuda, shape, five):
    passes.test_row_collapsed_galerkin(libmg, oracle, cuda, shape, five)


@pytest.mark.parametrize("nx,ny", [(401, 250), (401, 249)])
def test_conversion(libmg, cuda, nx, ny):
    torch = cuda
    with np.errstate(all="ignore"):
        host = [conversions._values(ny * nx, 30 + k).reshape(ny, nx) for k in range(6)]
        ref = [h.astype(np.float32) for h in host]
    src = [torch.from_numpy(h).cuda() for h in host]
    f32 = [torch.zeros((ny, nx), dtype=torch.float32, device="cuda") for _ in range(6)]
    a, b = libmg.op_struct(src, nx, ny, 0), libmg.op_struct(f32, nx, ny, 0, f32=True)
    libmg.mgk("mgk_op_to_f32", C.byref(a), C.byref(b), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for k in range(6):
        got, nan = f32[k].cpu().numpy(), np.isnan(ref[k])
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got.view(np.uint32)[~nan], ref[k].view(np.uint32)[~nan])
