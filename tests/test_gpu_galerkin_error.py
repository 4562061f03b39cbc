"""Error of the row-collapsed FP64 Galerkin product against exact sums, coupling by coupling, relative to
the largest coupling: not larger than that of the direct product (which rows of an odd pitch take), on
operators assembled from smooth and from rough tensors.  A CPU emulation of both orders has ratios of
0.5-0.95 on such operators; 1 is the bound, with the statistics of some 4000 nodes."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W = {0: 1.0, 1: 0.5, -1: 0.5}


def _operator(kind, n):
    h, rng = 1.0 / (n - 1), np.random.default_rng(3)
    y, x = np.meshgrid(np.arange(n) * h, np.arange(n) * h, indexing="ij")
    pi = np.pi
    a, b = 1 + 0.1 * pi * np.cos(pi * x) * np.sin(pi * y), 0.1 * pi * np.sin(pi * x) * np.cos(pi * y)
    c, d = 0.2 * pi * np.cos(2 * pi * x) * np.sin(pi * y), 1 + 0.1 * pi * np.sin(2 * pi * x) * np.cos(pi * y)
    s = {"smooth": np.ones_like(x), "material": np.where((x - 0.5) ** 2 + (y - 0.5) ** 2 < 0.06, 10.0, 1.0),
         "rough": rng.uniform(0.5, 1.5, x.shape), "stretched": np.ones_like(x)}[kind] / (a * d - b * c)
    xx, xy, yy = s * (d * d + b * b), s * (-d * c - b * a), s * (c * c + a * a)
    if kind == "stretched":
        xx, xy = 30 * xx, 0.1 * xy
    E, N, NE, NW, D = (np.zeros((n, n)) for _ in range(5))
    E[:, :-1] = -0.5 * (xx[:, :-1] + xx[:, 1:]) / h ** 2
    N[:-1] = -0.5 * (yy[:-1] + yy[1:]) / h ** 2
    NE[:-1, :-1] = -(xy[:-1, 1:] + xy[1:, :-1]) / (4 * h * h)
    NW[:-1, 1:] = (xy[:-1, :-1] + xy[1:, 1:]) / (4 * h * h)
    D[:] = 1.0
    D[1:-1, 1:-1] = -(E[1:-1, 1:-1] + E[1:-1, :-2] + N[1:-1, 1:-1] + N[:-2, 1:-1])
    return [E, N, NE, NW, D, 1.0 / D]


def _exact(E, N, NE, NW, D, _):
    r = lambda a, dj, di: np.roll(a, (-dj, -di), (0, 1))
    ld = [v.astype(np.longdouble) for v in (E, N, NE, NW, D)]
    E, N, NE, NW, D = ld
    entry = {(1, 0): E, (-1, 0): r(E, 0, -1), (0, 1): N, (0, -1): r(N, -1, 0), (1, 1): NE, (-1, -1): r(NE, -1, -1),
             (-1, 1): NW, (1, -1): r(NW, -1, 1), (0, 0): D}
    out = []
    for oi, oj in ((1, 0), (0, 1), (1, 1), (-1, 1), (0, 0)):
        v = np.zeros(D[::2, ::2].shape, np.longdouble)
        for ki in (-1, 0, 1):
            for kj in (-1, 0, 1):
                for (li, lj), a in entry.items():
                    w = 0.25 * W[ki] * W[kj] * W.get(ki + li - 2 * oi, 0.0) * W.get(kj + lj - 2 * oj, 0.0)
                    if w:
                        v += w * r(a, kj, ki)[::2, ::2]
        out.append(v)
    return out


@pytest.mark.parametrize("kind", ["smooth", "material", "rough", "stretched"])
def test_not_larger_than_the_direct_product(libmg, cuda, kind):
    torch = cuda
    nx = 129
    fine = _operator(kind, nx)
    for level in (0, 1):
        nxc = (nx - 1) // 2 + 1
        ref, err, got = _exact(*fine), [], None
        for pf, pc in (((nx + 31) // 32 * 32, (nxc + 31) // 32 * 32), (nx, nxc)):
            put = lambda a, p: torch.nn.functional.pad(torch.from_numpy(np.ascontiguousarray(a)), (0, p - a.shape[1])).contiguous().cuda()
            F = [put(a, pf) for a in fine]
            H = [torch.zeros((nxc, pc), dtype=torch.float64, device="cuda") for _ in range(6)]
            sf, sh = libmg.op_struct(F, nx, nx, 0), libmg.op_struct(H, nxc, nxc, 0)
            libmg.mgk("mgk_galerkin", C.byref(sf), C.byref(sh), torch.cuda.current_stream().cuda_stream)
            torch.cuda.synchronize()
            got = [v[:, :nxc].cpu().numpy() for v in H]
            inner = (slice(2, -2), slice(2, -2))
            big = np.abs(ref[4][inner]).max()
            err.append([float(np.sqrt((((g - e)[inner] / big) ** 2).mean())) for g, e in zip(got, ref)])
        print(kind, level, [f"{a / b:.2f}" for a, b in zip(*err)], [f"{v:.2e}" for v in err[1]])
        for a, b in zip(*err):
            assert a <= b
        fine, nx = got, nxc
