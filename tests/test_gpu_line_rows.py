"""FP32 line half-sweeps that factor their rows as they solve them (k_line_row): row lengths at and
after each power of two up to the longest (4096 unknowns; 4097 use stored factors), against the
oracle's Thomas solves.  Square cells keep the row systems' condition numbers small; the bound is
that of the other FP32 line tests (operator, data and solve rounded to FP32: 2e-5 relative)."""
import ctypes as C

import numpy as np
import pytest

from paper_2602_01888_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 63, 64, 65, 128, 129, 256, 257, 512, 513, 1024, 1025, 2048, 2049, 4096, 4097])
@pytest.mark.parametrize("five", [0, 1])
def test_row_lengths(libmg, oracle, cuda, n, five):
    torch = cuda
    nx, ny = n + 2, 9
    mp = I.MapSpec("identity") if five else I.MapSpec("sine_warp", (0.05,))
    inst = I.Instance("r", I.Grid(nx, ny, 0.0, 0.0, 1.0, 8.0 / (nx - 1)), mp, np.ones((ny, nx)))
    A = oracle.prepare(inst).A
    t = [torch.from_numpy(np.ascontiguousarray(a)).to("cuda", torch.float32)
         for a in (A.cE, A.cN, A.cNE, A.cNW, A.diag, 1.0 / A.diag)]
    op = libmg.op_struct(t, nx, ny, False, f32=True, five_point=five)
    f = torch.zeros(libmg.lib().mgk_line_factor_elems(nx, ny, 0), dtype=torch.float32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    libmg.mgk("mgk_line_factor_f32", C.byref(op), f.data_ptr(), s)
    rng = np.random.default_rng(n)
    phi, b = rng.standard_normal((ny, nx)), rng.standard_normal((ny, nx)) * np.abs(A.diag).max()
    bd = torch.from_numpy(b).to("cuda", torch.float32)
    for par in (0, 1):
        x = torch.from_numpy(phi).to("cuda", torch.float32)
        libmg.mgk("mgk_line_rows_f32", C.byref(op), f.data_ptr(), x.data_ptr(), bd.data_ptr(), par, s)
        torch.cuda.synchronize()
        got, ref = x.double().cpu().numpy(), oracle.line_rows(A, phi, b, par)
        assert np.abs(got - ref).max() < 2e-5 * np.abs(ref).max(), par
        still = np.ones((ny, nx), bool)
        still[par:-1:2, 1:-1] = False
        still[0] = True
        assert np.array_equal(got[still], phi.astype(np.float32).astype(np.float64)[still]), par
