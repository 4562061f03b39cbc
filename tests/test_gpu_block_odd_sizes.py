"""Point-smoothed mgk_vcycle_* on levels whose sides are not 2 m + 1 (the last unknown column or row
then lies on the coarse grid's boundary): rows of 16-byte multiples, whose levels the register blocks
smooth, give the bits of rows of an odd pitch, which the per-colour and tile kernels smooth."""
import pytest

from _hier import sizes, vcycle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(12, 10), (40, 33), (41, 34), (62, 60), (200, 151)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 1), (2, 0)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_even_sides(libmg, cuda, shape, nu, prec):
    shapes = sizes(*shape, 0, coarsest=60)
    a, b = (vcycle(libmg, cuda, prec, shapes, 0, nu, pitch=p) for p in (lambda n: (n + 31) // 32 * 32, lambda n: n | 1))
    assert cuda.isfinite(a).all()
    assert cuda.equal(a, b)
