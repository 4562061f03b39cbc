"""Smoothing reads the reciprocal diagonal only, so a diagonal array that does not start on 16 bytes
is no obstacle to mgk_smooth_march_* and the marching variants; a cycle, whose restriction reads it,
gives the same bits too."""
import ctypes as C

import numpy as np
import pytest

from _hier import operator, place, sizes, vcycle

pytestmark = pytest.mark.gpu

OFF = (0, 0, 0, 0, 1, 0)  # the diagonal starts one element late


@pytest.mark.parametrize("shape", [(213, 177, 0), (129, 129, 1)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_smoothing(libmg, cuda, shape, prec):
    torch = cuda
    nx, ny, per = shape
    dt = torch.float32 if prec == "f32" else torch.float64
    pitch = (nx + 31) // 32 * 32
    rng = np.random.default_rng(nx)
    phi, b = rng.standard_normal((2, ny - per, nx))
    s = torch.cuda.current_stream().cuda_stream
    names = [(None, None)] + [(v, n) for v, _, n in libmg.smooth_variants(prec == "f32", 4)]
    for v, _ in names:
        out = []
        for shift in ((0,) * 6, OFF):
            keep, op, unk = operator(libmg, torch, dt, nx, ny, per, 0, pitch, shift)
            x, bd = place(torch, phi, dt, pitch), place(torch, b, dt, pitch)
            y = torch.full_like(x, float("nan"))
            args = (x.data_ptr(), y.data_ptr(), bd.data_ptr(), 0, None, 0)
            if v is None:
                libmg.mgk(f"mgk_smooth_march_{prec}", C.byref(op), *args, s)
            else:
                libmg.mgk(f"mgk_smooth_variant_{prec}", C.byref(op), 4, v, *args, None, s)
            torch.cuda.synchronize()
            out.append(y[:, :nx])
        assert torch.isfinite(out[0]).all() and torch.equal(*out), v


@pytest.mark.parametrize("shape", [(65, 33, 0), (213, 177, 0), (129, 129, 1)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 1)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_cycles(libmg, cuda, shape, nu, prec):
    nx, ny, per = shape
    a, b = (vcycle(libmg, cuda, prec, sizes(nx, ny, per), per, nu, shift=s) for s in ((0,) * 6, OFF))
    assert cuda.isfinite(a).all()
    assert cuda.equal(a, b)
