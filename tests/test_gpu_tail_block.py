"""The tail kernel in registers (k_tail_block) against the cycle written out in numpy on the same
numbers: hierarchies of at most 1200 nodes, which it runs whole.  Coarsest levels of 12 to 256 unknowns
(from 129 up the inverse is read from global memory), periodic and not, sides that are not 2 m + 1,
cycles with and without pre- or post-smoothing.

Tolerance: a node's value passes at most 4 sweeps on each of 3 levels on the way down and up, each some ten
operations on a diagonally dominant row (which damps what comes in), and one dense row: below 300
roundings, 300 2^-24 = 1.8e-5 and 300 2^-53 = 3.3e-14 of the largest value."""
import numpy as np
import pytest

from _hier import couplings, inverse, sizes, start, vcycle

pytestmark = pytest.mark.gpu

ORDER = [(0, 0), (1, 1), (1, 0), (0, 1)]  # (i mod 2, j mod 2) of the colours
SH = lambda a, dj, di: np.roll(a, (-dj, -di), (0, 1))  # value at (j + dj, i + di); wraps hit no unknown but a periodic one


def _offdiag(c, x):
    E, N, NE, NW = c[:4]
    return (E * SH(x, 0, 1) + SH(E * 1.0, 0, -1) * SH(x, 0, -1) + N * SH(x, 1, 0) + SH(N, -1, 0) * SH(x, -1, 0)
            + NE * SH(x, 1, 1) + SH(NE, -1, -1) * SH(x, -1, -1) + NW * SH(x, 1, -1) + SH(NW, -1, 1) * SH(x, -1, 1))


def _smooth(c, unk, x, b, sweeps, rev):
    j, i = np.indices(x.shape)
    for _ in range(sweeps):
        for ci, cj in ORDER[::-1] if rev else ORDER:
            m = unk & (i % 2 == ci) & (j % 2 == cj)
            x = np.where(m, (b - _offdiag(c, x)) / c[4], x)
    return x


def _cycle(levels, per, inv, x, b, nu, l=0):
    c, unk = levels[l]
    if l == len(levels) - 1:
        x = np.zeros_like(b)
        x[unk] = inv.T @ b[unk]
        return x
    x = _smooth(c, unk, x, b, nu[0], False)
    r = np.where(unk, b - c[4] * x - _offdiag(c, x), 0.0)
    unkc = levels[l + 1][1]
    full = (4 * r + 2 * (SH(r, 0, 1) + SH(r, 0, -1) + SH(r, 1, 0) + SH(r, -1, 0))
            + SH(r, 1, 1) + SH(r, 1, -1) + SH(r, -1, 1) + SH(r, -1, -1)) / 16
    bc = np.where(unkc, full[::2, ::2][: unkc.shape[0], : unkc.shape[1]], 0.0)
    e = _cycle(levels, per, inv, np.zeros_like(bc), bc, nu, l + 1)
    up = np.vstack([e, e[:1] if per else 0 * e[:1]])
    up = np.hstack([up, 0 * up[:, :1]])
    p = np.zeros((2 * e.shape[0], 2 * e.shape[1]))
    p[::2, ::2], p[::2, 1::2] = up[:-1, :-1], (up[:-1, :-1] + up[:-1, 1:]) / 2
    p[1::2, ::2], p[1::2, 1::2] = (up[:-1, :-1] + up[1:, :-1]) / 2, (up[:-1, :-1] + up[:-1, 1:] + up[1:, :-1] + up[1:, 1:]) / 4
    x = np.where(unk, x + p[: x.shape[0], : x.shape[1]], x)
    return _smooth(c, unk, x, b, nu[1], True)


@pytest.mark.parametrize("shape,levels", [((9, 7, 0), 2), ((35, 19, 0), 2), ((27, 25, 0), 2), ((33, 33, 0), 2), ((33, 33, 0), 3),
                                          ((35, 33, 1), 2), ((33, 17, 1), 3), ((30, 33, 0), 2), ((21, 16, 0), 2)])
@pytest.mark.parametrize("nu", [(2, 2), (1, 1), (0, 1), (2, 0)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_cycle(libmg, cuda, shape, levels, nu, prec):
    nx, ny, per = shape
    shapes = sizes(nx, ny, per, levels)
    got = vcycle(libmg, cuda, prec, shapes, per, nu).double().cpu().numpy()
    dt = np.float32 if prec == "f32" else np.float64
    r = lambda a: a.astype(dt).astype(np.float64)
    lv = [([r(a) for a in c], unk) for c, unk in (couplings(n, m, per, 0) for n, m in shapes)]
    x, b = (r(a) for a in start(lv[0][1]))
    ref = _cycle(lv, per, inverse(*shapes[-1], per), x, b, nu)
    e = np.abs(got - ref).max() / np.abs(ref).max()
    assert e <= (1.8e-5 if prec == "f32" else 3.3e-14), e
