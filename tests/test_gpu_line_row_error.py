"""Error of FP32 line half-sweeps whose rows are dominated by their own couplings (x couplings R times
the y ones: the systems' condition number is about 4 R), against FP64 Thomas solves of the same
FP32 numbers, with the other rows at zero so that the right-hand side is exact.

The elimination carries each equation's surplus (diagonal minus its two couplings) and forms its
pivots by sums of positive terms, so its relative errors do not grow with the condition number: in a
CPU emulation the rms errors are at most 1.1, 2.2, 2.8, 3.7 and 5.0 units of 2^-24 at R = 1, 30, 100, 300 and
1000 (with stored cyclic-reduction factors 1.2, 4, 9, 20 and 45).  The bounds are about 1.5 times these."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BOUND = {1.0: 1.6, 30.0: 3.3, 100.0: 4.4, 300.0: 6.0, 1000.0: 7.7}  # in units of 2^-24


def _thomas(a, b, c, d):
    """FP64 solves of rows (axis 0) of tridiagonal systems along axis 1."""
    n = b.shape[1]
    cp, dp = np.empty_like(b), np.empty_like(b)
    cp[:, 0], dp[:, 0] = c[:, 0] / b[:, 0], d[:, 0] / b[:, 0]
    for i in range(1, n):
        m = b[:, i] - a[:, i] * cp[:, i - 1]
        cp[:, i], dp[:, i] = c[:, i] / m, (d[:, i] - a[:, i] * dp[:, i - 1]) / m
    for i in range(n - 2, -1, -1):
        dp[:, i] -= cp[:, i] * dp[:, i + 1]
    return dp


@pytest.mark.parametrize("n", [2, 7, 31, 63, 64, 95, 127, 128, 255, 511, 1023, 1151, 2048, 3071, 4096])
@pytest.mark.parametrize("R", sorted(BOUND))
def test_dominant_rows(libmg, cuda, n, R):
    torch = cuda
    nx, ny = n + 2, 129
    rng = np.random.default_rng(n)
    f32 = lambda a: a.astype(np.float32)
    E = f32(-R * rng.uniform(0.5, 1.5, (ny, nx)))
    N = f32(-rng.uniform(0.5, 1.5, (ny, nx)))
    E64, N64 = E.astype(np.float64), N.astype(np.float64)
    diag = np.ones((ny, nx), np.float32)
    diag[1:-1, 1:-1] = f32(-(E64[1:-1, 1:-1] + E64[1:-1, :-2] + N64[1:-1, 1:-1] + N64[:-2, 1:-1]))
    b = f32(rng.standard_normal((ny, nx)))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    zero = np.zeros((ny, nx), np.float32)
    arr = [dev(a) for a in (E, N, zero, zero, diag, f32(1.0 / diag))]
    op = libmg.op_struct(arr, nx, ny, False, f32=True, five_point=True)
    fac = torch.zeros(libmg.lib().mgk_line_factor_elems(nx, ny, 0), dtype=torch.float32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    libmg.mgk("mgk_line_factor_f32", C.byref(op), fac.data_ptr(), s)
    x, bd = dev(zero), dev(b)
    libmg.mgk("mgk_line_rows_f32", C.byref(op), fac.data_ptr(), x.data_ptr(), bd.data_ptr(), 1, s)
    torch.cuda.synchronize()
    got = x.cpu().numpy().astype(np.float64)[1:-1:2, 1:-1]
    a, c = E64[1:-1:2, :-2].copy(), E64[1:-1:2, 1:-1].copy()
    a[:, 0] = 0.0
    c[:, -1] = 0.0
    ref = _thomas(a, diag.astype(np.float64)[1:-1:2, 1:-1], c, b.astype(np.float64)[1:-1:2, 1:-1])
    err = np.sqrt((((got - ref) ** 2).sum(1) / (ref ** 2).sum(1)).mean()) * 2.0 ** 24
    print(f"n {n} R {R}: {err:.2f}")
    assert err <= BOUND[R]
