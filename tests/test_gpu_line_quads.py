"""Stored factors of long FP32 rows read as 16-byte quads or, from a factor buffer that does not start
on 16 bytes, one by one: the same operations per unknown, so the same bits."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4097, 8191, 8192, 8193])
@pytest.mark.parametrize("five", [0, 1])
def test_factor_alignment_changes_no_bit(libmg, cuda, n, five):
    torch = cuda
    nx, ny = n + 2, 7
    rng = np.random.default_rng(n)
    c = [-rng.uniform(0.5, 1.5, (ny, nx)) for _ in range(2)]
    c += [(np.zeros((ny, nx)) if five else rng.uniform(-0.2, 0.2, (ny, nx))) for _ in range(2)]
    diag = rng.uniform(6.0, 7.0, (ny, nx))
    t = [torch.from_numpy(a).to("cuda", torch.float32) for a in (*c, diag, 1.0 / diag)]
    op = libmg.op_struct(t, nx, ny, False, f32=True, five_point=five)
    elems = libmg.lib().mgk_line_factor_elems(nx, ny, 0)
    phi, b = (torch.from_numpy(rng.standard_normal((ny, nx))).to("cuda", torch.float32) for _ in range(2))
    s = torch.cuda.current_stream().cuda_stream
    out = []
    for shift in (0, 1):
        f = torch.zeros(elems + shift, dtype=torch.float32, device="cuda")[shift:]
        libmg.mgk("mgk_line_factor_f32", C.byref(op), f.data_ptr(), s)
        x = phi.clone()
        libmg.mgk("mgk_line_smooth_f32", C.byref(op), f.data_ptr(), x.data_ptr(), b.data_ptr(), 1, 0, s)
        torch.cuda.synchronize()
        assert torch.isfinite(x).all()
        out.append(x)
    assert torch.equal(*out)
