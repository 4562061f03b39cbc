"""The register-block smoother (k_block.cu): sweeps, coarse correction and the fused residual
restriction against the per-colour and tile kernels, bit for bit (both do the same operations
per node in the same order; those kernels are checked against the oracle elsewhere).

The tile of a pass owns 52 x 48 nodes (FP32, two sweeps; 52 x 16 on small levels), 48 x 46 /
48 x 14 with the restriction, 56 x 56 / 56 x 24 for one FP32 sweep; in FP64 22 x 16, 18 x 14 with
the restriction, 26 x 24 for one sweep: the shapes below end one node before, at and after such edges, and wrap a periodic seam."""
import ctypes as C

import numpy as np
import pytest

from paper_2602_01888_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = [(17, 9, 0), (23, 17, 0), (45, 29, 0), (49, 33, 0), (53, 49, 0), (57, 25, 0), (105, 17, 0), (113, 57, 0), (209, 177, 0), (833, 385, 0),
          (129, 129, 1), (513, 257, 1)]


def _operator(libmg, torch, dt, nx, ny, per, five, pitch):
    """Random symmetric diagonally dominant couplings: every term of the sums matters."""
    nyr = ny - 1 if per else ny
    rng = np.random.default_rng(nx * 1000 + ny)
    c = [-rng.uniform(0.5, 1.5, (nyr, nx)) for _ in range(2)] + [
        (np.zeros((nyr, nx)) if five else rng.uniform(-0.2, 0.2, (nyr, nx))) for _ in range(2)]
    diag = rng.uniform(6.0, 7.0, (nyr, nx))
    unk = np.zeros((nyr, nx), bool)
    unk[(slice(None) if per else slice(1, -1)), 1:-1] = True
    diag[~unk] = 1.0

    def put(a, p):
        t = torch.zeros((nyr, p), dtype=dt, device="cuda")
        t[:, :nx] = torch.from_numpy(a).to("cuda", dt)
        return t

    arr = [put(a, pitch) for a in (*c, diag, 1.0 / diag)]
    return arr, libmg.op_struct(arr, nx, ny, per, f32=dt == torch.float32, five_point=five), put, unk, nyr, rng


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("five", [0, 1])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_sweeps_equal_the_per_colour_kernels(libmg, cuda, shape, five, prec):
    torch = cuda
    nx, ny, per = shape
    dt = torch.float32 if prec == "f32" else torch.float64
    pitch = (nx + 31) // 32 * 32
    keep, op, put, unk, nyr, rng = _operator(libmg, torch, dt, nx, ny, per, five, pitch)
    ns = 2
    var = [v for v, t, n in libmg.smooth_variants(prec == "f32", 4) if t[0] == (52 if prec == "f32" else 22)][0]
    phi, b = rng.standard_normal((nyr, nx)), rng.standard_normal((nyr, nx))
    nxc, nyc = (nx - 1) // 2 + 1, (ny - 1) // 2 + 1
    pc = (nxc + 31) // 32 * 32
    eH = torch.zeros((nyc - 1 if per else nyc, pc), dtype=dt, device="cuda")
    lo = 0 if per else 1
    eH[lo:(None if per else -1), 1:nxc - 1] = torch.from_numpy(
        rng.standard_normal((eH.shape[0] - 2 * lo, nxc - 2))).to("cuda", dt)
    s = torch.cuda.current_stream().cuda_stream
    for rev in (0, 1):
        for corr in (None, eH):
            x, bd = put(phi, pitch), put(b, pitch)
            out = torch.full_like(x, float("nan"))
            libmg.mgk(f"mgk_smooth_variant_{prec}", C.byref(op), 4, var, x.data_ptr(), out.data_ptr(), bd.data_ptr(), rev,
                      None if corr is None else corr.data_ptr(), pc, None, s)
            if corr is not None:
                libmg.mgk(f"mgk_prolong_add_{prec}", C.byref(op), x.data_ptr(), corr.data_ptr(), pc, s)
            libmg.mgk(f"mgk_smooth_{prec}", C.byref(op), x.data_ptr(), bd.data_ptr(), ns, rev, s)
            torch.cuda.synchronize()
            assert torch.equal(out[:, :nx], x[:, :nx]), (rev, corr is not None)


@pytest.mark.parametrize("shape", [s for s in SHAPES if s[0] > 17])
@pytest.mark.parametrize("five", [0, 1])
@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nu", [(1, 1), (2, 2), (3, 2), (0, 1)])
def test_cycles_equal_the_unaligned_path(libmg, cuda, shape, five, prec, nu):
    """A V-cycle from a nonzero iterate on rows of 16-byte multiples (register blocks with the
    fused restriction in FP32) and on rows of an odd pitch (the other kernels)."""
    torch = cuda
    nx, ny, per = shape
    dt = torch.float32 if prec == "f32" else torch.float64
    got = []
    for pad in (True, False):
        ops, X, B, T, keep = [], [], [], [], []
        n, m = nx, ny
        for l in range(8):
            pitch = (n + 31) // 32 * 32 if pad else n | 1
            arr, op, put, unk, nyr, rng = _operator(libmg, torch, dt, n, m, per, five if l == 0 else 0, pitch)
            keep.append(arr)
            ops.append(op)
            r = rng.standard_normal((nyr, n)) * unk
            B.append(put(r if l == 0 else 0 * r, pitch))
            X.append(put(rng.standard_normal((nyr, n)) * unk if l == 0 else 0 * r, pitch))
            T.append(put(0 * r, pitch))
            if (n - 2) * (m - (1 if per else 2)) <= 250 or (n - 1) % 2 or (m - 1) % 2:
                break
            n, m = (n - 1) // 2 + 1, (m - 1) // 2 + 1
        mc = (n - 2) * (m - 1 if per else m - 2)
        assert mc <= 256
        inv = torch.from_numpy(np.random.default_rng(5).standard_normal((mc, mc)) / mc).cuda()
        arr = ((libmg.mgk_op_f32 if prec == "f32" else libmg.mgk_op_f64) * len(ops))(*ops)
        ptrs = lambda L: (C.c_void_p * len(L))(*[t.data_ptr() for t in L])
        libmg.mgk(f"mgk_vcycle_{prec}", len(ops), arr, ptrs(X), ptrs(B), ptrs(T), inv.data_ptr(), nu[0], nu[1], 0,
                  torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        got.append(X[0][:, :nx].clone())
    assert torch.isfinite(got[0]).all()
    assert torch.equal(got[0], got[1])
