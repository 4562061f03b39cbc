"""Mixed solves of very small and very large sources: beyond 2^60 the power of two between the FP64
residual and the FP32 cycle is applied in FP64, below in FP32.  Scaling the source by a power of two scales
every FP64 quantity exactly, and the cycle's right-hand side but for entries more than 2^60 below the rms (lost in
FP32 either way), so iteration counts are the same and solutions agree to rounding."""
import numpy as np
import pytest

from paper_2602_01888_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("outer", ["fcg", "vcycle"])
def test_powers_of_two(libmg, cuda, outer):
    inst = I.Instance("s", I.Grid(257, 257), I.MapSpec("sine_warp", (0.08,)), np.ones((257, 257)))
    rng = np.random.default_rng(9)
    rho = rng.standard_normal(inst.grid.shape)
    ctx = libmg.Context(0)
    opts = libmg.make_opts("mixed", outer, rtol=1e-10, max_iters=100)
    p = libmg.Problem(ctx, inst, opts)
    ref = np.zeros(inst.grid.shape)
    iters = libmg.mg_solve(p.h, rho, None, ref, opts).iters
    for k in (-900 // 8, -80, -61, -59, 59, 61, 80, 900 // 8):
        phi = np.zeros_like(ref)
        st = libmg.mg_solve(p.h, np.ascontiguousarray(np.ldexp(rho, k)), None, phi, opts)
        assert st.iters == iters, k
        assert np.abs(np.ldexp(phi, -k) - ref).max() <= 1e-13 * np.abs(ref).max(), k
    p.close()
    ctx.close()
