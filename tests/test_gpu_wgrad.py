"""The conv weight gradient (coulps_cv_conv3d_wgrad) against FP64 sums of the
same BF16 values, at sizes around its 16 x 16 tiles, on one site, and from
addresses aligned to 2 bytes only.  Tolerance: the FP32 sums' rounding, at most
2^-23 of the sum of magnitudes per step over the 16 MMAs of a tile and the
tiles and CTAs added after, < 1e-5 of it."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def _ref(torch, a, d):
    n, Z, Y, X, _ = a.shape
    ap = torch.nn.functional.pad(a.double(), (0, 0, 1, 1, 1, 1, 1, 1))
    d2 = d.double().reshape(-1, 16)
    out = torch.empty(16, 16, 3, 3, 3, dtype=torch.float64, device=a.device)
    for k in range(27):
        z, y, x = k // 9, k // 3 % 3, k % 3
        out[:, :, z, y, x] = d2.T @ ap[:, z:z + Z, y:y + Y, x:x + X].reshape(-1, 16)
    return out


@pytest.mark.parametrize("shape", [(1, 1, 1, 1), (2, 5, 6, 37), (1, 3, 17, 15), (3, 2, 33, 16),
                                   (1, 1, 3, 70), (64, 14, 14, 14), (2, 16, 16, 16)])
@pytest.mark.parametrize("shift", [0, 1])
def test_wgrad_matches_fp64(shape, shift):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps
    _build.build()
    lib = coulps.load()
    n, Z, Y, X = shape
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    size = n * Z * Y * X * 16

    def rnd():
        return torch.randn(size + shift, generator=g, device="cuda").to(torch.bfloat16)[shift:]

    a, d = rnd(), rnd()
    nblk = min(1024, (n * Z * Y * ((X + 63) // 64) + 31) // 32)
    scratch = torch.full((nblk * 27 * 256,), float("nan"), device="cuda")
    dW = torch.full((16 * 16 * 27,), float("nan"), device="cuda")
    vp = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    args = (n, X, Y, Z, vp(scratch))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    assert lib.coulps_cv_conv3d_wgrad(vp(a), vp(d), vp(dW), *args, scratch.numel() - 1, stream) == coulps.EINVAL
    assert lib.coulps_cv_conv3d_wgrad(vp(a), vp(d), vp(dW), *args, scratch.numel(), stream) == coulps.OK
    got = dW.view(16, 16, 3, 3, 3).double()
    a5, d5 = a.view(n, Z, Y, X, 16), d.view(n, Z, Y, X, 16)
    ref, mag = _ref(torch, a5, d5), _ref(torch, a5.abs(), d5.abs())
    assert bool(((got - ref).abs() <= 1e-5 * mag + 1e-30).all())
