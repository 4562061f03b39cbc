"""Set-up kernels that do in one pass what several did: the 9-point assembly (a warp owns 30
columns and marches strips of 8 rows), its couplings and its diagonal (four terms, the cross ones
cancel) bit for bit and against the sum over all eight couplings; the row-collapsed FP64 Galerkin
product (30 coarse columns a warp) against the direct product, which rows of an odd pitch take;
and the analytic maps with factors of one coordinate (tiles of 32 x 32) against the general
formula.  Sizes around those edges."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(5, 5, 0), (31, 9, 0), (33, 17, 0), (61, 33, 0), (63, 65, 0), (119, 37, 0), (123, 131, 0), (257, 129, 1), (125, 65, 1)]


def _fields(nx, nyr, seed):
    rng = np.random.default_rng(seed)
    return [rng.uniform(0.5, 1.5, (nyr, nx)), rng.uniform(-0.3, 0.3, (nyr, nx)), rng.uniform(0.5, 1.5, (nyr, nx))]


@pytest.mark.parametrize("shape", SHAPES)
def test_nine_point_assembly(libmg, cuda, shape):
    torch = cuda
    nx, ny, per = shape
    nyr, hx, hy = (ny - 1 if per else ny), 0.01, 0.013
    pitch = (nx + 31) // 32 * 32
    put = lambda a: torch.nn.functional.pad(torch.from_numpy(a), (0, pitch - nx)).contiguous().cuda()
    exx, exy, eyy = (put(a) for a in _fields(nx, nyr, nx))
    ops = [torch.full((nyr, pitch), 7.0, dtype=torch.float64, device="cuda") for _ in range(6)]
    st = libmg.op_struct(ops, nx, ny, per)
    libmg.mgk("mgk_assemble", C.byref(st), hx, hy, exx.data_ptr(), exy.data_ptr(), eyy.data_ptr(),
              torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    E, N, NE, NW, dg, di = (a[:, :nx].cpu().numpy() for a in ops)
    xx, xy, yy = (a[:, :nx].cpu().numpy() for a in (exx, exy, eyy))
    up = lambda a: np.roll(a, -1, 0)
    has_up = np.ones((nyr, 1), bool)
    if not per:
        has_up[-1] = False
    e, n = np.zeros_like(xx), np.zeros_like(xx)
    ne, nw = np.zeros_like(xx), np.zeros_like(xx)
    e[:, :-1] = (xx[:, :-1] + xx[:, 1:]) * (-0.5 * (1.0 / (hx * hx)))
    n[:] = np.where(has_up, (yy + up(yy)) * (-0.5 * (1.0 / (hy * hy))), 0.0)
    q = 1.0 / (4.0 * hx * hy)
    ne[:, :-1] = np.where(has_up, -(xy[:, 1:] + up(xy)[:, :-1]) * q, 0.0)
    nw[:, 1:] = np.where(has_up, (xy[:, :-1] + up(xy)[:, 1:]) * q, 0.0)
    for a, b in ((E, e), (N, n), (NE, ne), (NW, nw)):
        assert np.array_equal(a, b)
    dn, w, r = (lambda a: np.roll(a, 1, 0)), (lambda a: np.roll(a, 1, 1)), (lambda a: np.roll(a, -1, 1))
    s = e + w(e) + n + dn(n)
    d = np.ones_like(s)
    unk = (slice(None) if per else slice(1, -1), slice(1, -1))
    d[unk] = -s[unk]
    assert np.array_equal(dg, d) and np.array_equal(di, 1.0 / d)
    # zero row sums: eight couplings of at most 1.5 / h^2, rounded once, and seven additions
    full = (s + ne + dn(w(ne)) + nw + dn(r(nw)))[unk]
    assert np.abs(dg[unk] + full).max() <= 32 * 1.5 / hx ** 2 * 2.0 ** -53 * 4


@pytest.mark.parametrize("shape", [s for s in SHAPES if (s[0] - 1) % 2 == 0 and (s[1] - 1) % 2 == 0])
@pytest.mark.parametrize("five", [0, 1])
def test_row_collapsed_galerkin(libmg, oracle, cuda, shape, five):
    torch = cuda
    nx, ny, per = shape
    nyr, nxc, nyc = (ny - 1 if per else ny), (nx - 1) // 2 + 1, (ny - 1) // 2 + 1
    rng = np.random.default_rng(nx)
    fine = [rng.uniform(-1.5, -0.5, (nyr, nx)) for _ in range(2)]
    fine += [(np.zeros((nyr, nx)) if five else rng.uniform(-0.4, 0.4, (nyr, nx))) for _ in range(2)]
    fine += [rng.uniform(6.0, 8.0, (nyr, nx))]
    fine += [1.0 / fine[4]]
    got = []
    for pad in (True, False):  # aligned pairs of columns; odd pitch: the direct product
        pf, pc = ((nx + 31) // 32 * 32, (nxc + 31) // 32 * 32) if pad else (nx, nxc | 1)
        put = lambda a, p: torch.nn.functional.pad(torch.from_numpy(a), (0, p - a.shape[1])).contiguous().cuda()
        F = [put(a, pf) for a in fine]
        H = [torch.full((nyc - 1 if per else nyc, pc), 7.0, dtype=torch.float64, device="cuda") for _ in range(6)]
        sf, sh = libmg.op_struct(F, nx, ny, per, five_point=five), libmg.op_struct(H, nxc, nyc, per)
        libmg.mgk("mgk_galerkin", C.byref(sf), C.byref(sh), torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        got.append([a[:, :nxc].cpu().numpy() for a in H])
    # both sum the same products of magnitude up to 8 in different orders: 1e-14 absolute
    for a, b in zip(*got):
        assert np.abs(a - b).max() <= 1e-14


MAPS = {"identity": (0, (0.0,) * 4), "polar": (2, (0.0,) * 4), "sinh": (3, (0.7, 1.3, 0.0, 0.0)),
        "scaled": (4, (1.5, 0.0, 0.0, 0.75)), "sheared": (4, (1.1, 0.2, -0.1, 0.9))}


@pytest.mark.parametrize("name", list(MAPS))
@pytest.mark.parametrize("nx,ny,per,physical", [(5, 5, 0, 1), (31, 33, 0, 0), (32, 65, 1, 1), (67, 31, 0, 1)])
def test_separable_maps(libmg, cuda, name, nx, ny, per, physical):
    torch = cuda
    kind, prm = MAPS[name]
    nyr, pitch, x0, y0, hx, hy = (ny - 1 if per else ny), nx + 3, 1.0, 0.25, 1.0 / (nx - 1), 2.0 / (ny - 1)
    s = np.random.default_rng(nx).uniform(0.5, 8.0, (nyr, nx)) if physical else np.ones((nyr, nx))
    x, y = (x0 + np.arange(nx) * hx)[None, :] + np.zeros((nyr, 1)), (y0 + np.arange(nyr) * hy)[:, None] + np.zeros((1, nx))
    p, one, zero = prm, np.ones_like(x), np.zeros_like(x)
    a, b, c, d = {0: (one, zero, zero, one), 2: (np.cos(y), -x * np.sin(y), np.sin(y), x * np.cos(y)),
                  3: (p[0] * p[1] * np.cosh(p[1] * x), zero, zero, p[0] * p[1] * np.cosh(p[1] * y)),
                  4: (p[0] * one, p[1] * one, p[2] * one, p[3] * one)}[kind]
    det = a * d - b * c
    ref = [det, s / det * (d * d + b * b), s / det * (-d * c - b * a), s / det * (c * c + a * a)]
    put = lambda v: torch.nn.functional.pad(torch.from_numpy(v), (0, pitch - nx)).contiguous().cuda()
    eps = put(s) if physical else None
    out = [torch.full((nyr, pitch), 7.0, dtype=torch.float64, device="cuda") for _ in range(4)]
    folded = torch.zeros(1, dtype=torch.int32, device="cuda")
    libmg.mgk("mgk_eps_analytic", kind, (C.c_double * 4)(*prm), nx, ny, per, x0, y0, hx, hy,
              eps.data_ptr() if physical else None, pitch, *[v.data_ptr() for v in out], folded.data_ptr(),
              torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert int(folded.item()) == 0
    got = [v.cpu().numpy() for v in out]
    emag = max(np.abs(ref[1]).max(), np.abs(ref[3]).max())
    # at most 16 roundings a side (two of them cosh's two units), none in a cancelling sum but exy's
    for v, r, m in zip(got, ref, (det.max(), emag, emag, emag)):
        assert np.abs(v[:, :nx] - r).max() <= 32 * 2.0 ** -53 * m
        assert (v[:, nx:] == 7.0).all()
    if name != "sheared":
        assert (got[2][:, :nx] == 0.0).all()
