"""mgk_vcycle_* start every coarse iterate from zero, boundary nodes included, whatever the
caller's arrays hold: cycles whose coarse arrays and scratch hold NaN equal, bit for bit, cycles on
cleared ones.  Two levels (no tail kernel), the FP64 line cycle (never a tail), an FP32 line
cycle with a tail below two levels, point cycles on aligned and unaligned rows."""
import pytest

from _hier import sizes, vcycle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,levels", [((33, 17), 2), ((65, 33), 3), ((129, 65), 4)])
@pytest.mark.parametrize("nu", [(1, 1), (2, 1), (0, 1), (1, 0)])
@pytest.mark.parametrize("per", [0, 1])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("line", [False, True])
def test_stale_coarse_arrays_change_nothing(libmg, cuda, shape, levels, nu, per, prec, line):
    shapes = sizes(*shape, per, levels)
    for five in (0, 1) if line else (0,):
        for pitch in (lambda n: (n + 31) // 32 * 32, lambda n: n | 1):
            a, b = (vcycle(libmg, cuda, prec, shapes, per, nu, line=line, five=five, pitch=pitch, stale=v)
                    for v in (0.0, float("nan")))
            assert cuda.isfinite(a).all()
            assert cuda.equal(a, b), (five, pitch(2))
