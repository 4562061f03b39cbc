"""Hierarchies of random symmetric, diagonally dominant operators in caller-owned arrays, for the
mgk_vcycle_* tests: every term of every sum matters, and no level is the coarsening of another."""
import ctypes as C

import numpy as np


def couplings(nx, ny, per, five):
    """cE cN cNE cNW diag and the mask of the unknowns, as numpy arrays; the same numbers every time."""
    nyr = ny - 1 if per else ny
    rng = np.random.default_rng(nx * 1000 + ny)
    c = [-rng.uniform(0.5, 1.5, (nyr, nx)) for _ in range(2)] + [
        (np.zeros((nyr, nx)) if five else rng.uniform(-0.2, 0.2, (nyr, nx))) for _ in range(2)]
    diag = rng.uniform(6.0, 7.0, (nyr, nx))
    unk = np.zeros((nyr, nx), bool)
    unk[(slice(None) if per else slice(1, -1)), 1:-1] = True
    diag[~unk] = 1.0
    return [*c, diag], unk


def operator(libmg, torch, dt, nx, ny, per, five, pitch, shift=(0,) * 6):
    """Arrays cE cN cNE cNW diag 1/diag of row pitch `pitch`, array k starting shift[k] elements past
    a 16-byte boundary, and the operator struct."""
    c, unk = couplings(nx, ny, per, five)
    arr = [place(torch, a, dt, pitch, s) for a, s in zip((*c, 1.0 / c[4]), shift)]
    return arr, libmg.op_struct(arr, nx, ny, per, f32=dt == torch.float32, five_point=five), unk


def start(unk, seed=5):
    """Iterate and right-hand side of the finest level."""
    return np.random.default_rng(seed).standard_normal((2,) + unk.shape) * unk


def inverse(nx, ny, per):
    """A stand-in for the coarsest inverse."""
    m = (nx - 2) * (ny - 1 if per else ny - 2)
    return np.random.default_rng(m).standard_normal((m, m)) / m


def place(torch, a, dt, pitch, shift=0, fill=0.0):
    """The rows of `a` at a row pitch, the array starting `shift` elements into its storage."""
    n = a.shape[0] * pitch
    t = torch.full((n + shift,), fill, dtype=dt, device="cuda")[shift:].view(a.shape[0], pitch)
    t[:, : a.shape[1]] = torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    return t


def sizes(nx, ny, per, levels=None, coarsest=250):
    """Level sizes: `levels` of them, or down to at most `coarsest` unknowns."""
    out = [(nx, ny)]
    while (len(out) < levels) if levels else ((nx - 2) * (ny - (1 if per else 2)) > coarsest):
        nx, ny = (nx - 1) // 2 + 1, (ny - 1) // 2 + 1
        out.append((nx, ny))
    return out


def vcycle(libmg, torch, prec, shapes, per, nu, line=False, five=0, pitch=lambda n: (n + 31) // 32 * 32, stale=0.0,
           shift=(0,) * 6, seed=5):
    """One cycle from a random iterate; the coarse iterates, right-hand sides and all scratch arrays
    hold `stale` beforehand.  Returns the result's nodes."""
    dt = torch.float32 if prec == "f32" else torch.float64
    ops, X, B, T, F, keep = [], [], [], [], [], []
    s = torch.cuda.current_stream().cuda_stream
    for l, (n, m) in enumerate(shapes):
        p = pitch(n)
        arr, op, unk = operator(libmg, torch, dt, n, m, per, five if l == 0 else 0, p, shift)
        keep.append(arr)
        ops.append(op)
        r = start(unk, seed)
        old = np.full(unk.shape, stale)
        X.append(place(torch, r[0] if l == 0 else old, dt, p))
        B.append(place(torch, r[1] if l == 0 else old, dt, p))
        T.append(place(torch, old, dt, p))
        if line and l < len(shapes) - 1:
            F.append(torch.zeros(libmg.lib().mgk_line_factor_elems(n, m, per), dtype=dt, device="cuda"))
            libmg.mgk(f"mgk_line_factor_{prec}", C.byref(op), F[-1].data_ptr(), s)
    inv = torch.from_numpy(inverse(*shapes[-1], per)).cuda()
    arr = ((libmg.mgk_op_f32 if prec == "f32" else libmg.mgk_op_f64) * len(ops))(*ops)
    ptrs = lambda L: (C.c_void_p * len(L))(*[t.data_ptr() for t in L])
    if line:
        libmg.mgk(f"mgk_vcycle_line_{prec}", len(ops), arr, ptrs(X), ptrs(B), ptrs(T), inv.data_ptr(), ptrs(F), nu[0], nu[1], s)
    else:
        libmg.mgk(f"mgk_vcycle_{prec}", len(ops), arr, ptrs(X), ptrs(B), ptrs(T), inv.data_ptr(), nu[0], nu[1], 0, s)
    torch.cuda.synchronize()
    return X[0][:, : shapes[0][0]].clone()
