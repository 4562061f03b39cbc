"""Polar map with a material: eps' / det J of Eqs. 12-15 is rounded once, like the division.  On the
row y = 0 every other factor is exact (cos 0 = 1, sin 0 = 0, so det J = x and Eq. 15 is s / x),
so eps_yy there is the quotient, bit for bit; elsewhere it is within the roundings of
det J, the row's sum of squares and the product (four) of the formula."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,x0,hx", [(1025, 1.0, 2.0 ** -10), (4097, 0.125, 2.0 ** -9), (515, 3.0, 0.375)])
def test_one_rounding_of_the_quotient(libmg, cuda, nx, x0, hx):
    torch = cuda
    ny = 9
    s = np.exp(np.random.default_rng(nx).uniform(-3.0, 3.0, (ny, nx)))
    eps = torch.from_numpy(s).cuda()
    out = [torch.zeros((ny, nx), dtype=torch.float64, device="cuda") for _ in range(4)]
    folded = torch.zeros(1, dtype=torch.int32, device="cuda")
    libmg.mgk("mgk_eps_analytic", 2, (C.c_double * 4)(), nx, ny, 0, x0, 0.0, hx, 0.125, eps.data_ptr(), nx,
              *[v.data_ptr() for v in out], folded.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert int(folded.item()) == 0
    D, exx, exy, eyy = (v.cpu().numpy() for v in out)
    x = x0 + hx * np.arange(nx)
    assert np.array_equal(D[0], x)
    assert np.array_equal(eyy[0], s[0] / x)
    assert np.abs(eyy * x / s - 1.0).max() <= 6 * 2.0 ** -53  # and two of this line
