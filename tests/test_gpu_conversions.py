"""FP64 -> FP32 conversion of an operator's arrays on the integer pipe: the bits of the cast, over
every exponent, ties, the edges of both normal ranges, subnormal results, infinities and NaN."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _values(n, seed):
    rng = np.random.default_rng(seed)
    bits = rng.integers(0, 2 ** 64, n, dtype=np.uint64)
    near = rng.integers(850, 1170, n // 2, dtype=np.uint64) << np.uint64(52)  # around the FP32 range
    bits[: n // 2] = bits[: n // 2] & np.uint64(0x800FFFFFFFFFFFFF) | near
    ties = rng.integers(0, 2 ** 32, n // 4, dtype=np.uint64).astype(np.uint32).view(np.float32)
    ties = np.where(np.isfinite(ties), ties, np.float32(1.0))
    up = np.nextafter(ties, np.float32(np.inf)).astype(np.float64)
    mid = 0.5 * (ties.astype(np.float64) + np.where(np.isfinite(up), up, 0.0))
    v = bits.view(np.float64).copy()
    v[n // 2: n // 2 + mid.size] = mid
    edge = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, 2.0 ** -149, 2.0 ** -150, 1.5 * 2.0 ** -150,
                     2.0 ** -151, 3.4028235677973366e38, 3.4028235677973362e38, 1e308, 5e-324, 1.0, 1.0 + 2.0 ** -24])
    v[-2 * edge.size:] = np.concatenate([edge, -edge])
    return v


@pytest.mark.parametrize("seed", [0, 1])
def test_operator_copies_convert_like_casts(libmg, cuda, seed):
    torch = cuda
    nx = ny = 65
    with np.errstate(all="ignore"):
        host = [_values(ny * nx, 10 * seed + k).reshape(ny, nx) for k in range(6)]
        ref = [h.astype(np.float32) for h in host]
    stream = torch.cuda.current_stream().cuda_stream
    src = [torch.from_numpy(h).cuda() for h in host]
    f32 = [torch.zeros((ny, nx), dtype=torch.float32, device="cuda") for _ in range(6)]
    a, b = libmg.op_struct(src, nx, ny, 0), libmg.op_struct(f32, nx, ny, 0, f32=True)
    libmg.mgk("mgk_op_to_f32", C.byref(a), C.byref(b), stream)
    torch.cuda.synchronize()
    for k in range(6):
        got, nan = f32[k].cpu().numpy(), np.isnan(ref[k])
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got.view(np.uint32)[~nan], ref[k].view(np.uint32)[~nan])
