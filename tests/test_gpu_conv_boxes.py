"""Convolutions of many narrow boxes, which share tiles side by side, against
the boxes one by one: bitwise, both epilogues, on a range of rows too, at
widths around the rule's edges (a box as wide as a tile stays by itself)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,Z,Y,X", [(5, 3, 4, 14), (300, 2, 3, 1), (3, 2, 2, 127), (2, 2, 2, 128),
                                      (7, 4, 5, 63), (9, 1, 1, 129), (2, 3, 3, 64), (130, 5, 6, 2)])
def test_boxes_side_by_side_bitwise(nb, Z, Y, X):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps, stein
    _build.build()
    lib = coulps.load()
    g = torch.Generator(device="cuda").manual_seed(nb + X)
    a = torch.randn(nb, Z, Y, X, 16, generator=g, device="cuda").to(torch.bfloat16)
    W = 0.2 * torch.randn(16, 16, 3, 3, 3, generator=g, device="cuda")
    b = torch.randn(16, generator=g, device="cuda")
    h = stein.conv3d_tc(a, W, b)
    act, der = stein.conv3d_tanh_tc(a, W, b)
    wp, err = stein.pack_weights(W), torch.zeros(1, dtype=torch.int32, device="cuda")
    vp = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    part, pder = torch.zeros_like(act), torch.zeros_like(der)
    y0, z0 = Y // 2, Z // 2
    assert lib.coulps_cv_conv3d_tanh_rows(vp(a), vp(wp), vp(b), vp(part), vp(pder), nb, X, Y, Z, 0, y0, Y, z0, Z,
                                          vp(err), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == 0
    for n in range(nb):
        one = stein.conv3d_tc(a[n:n + 1].contiguous(), W, b)
        assert torch.equal(h[n:n + 1], one), n
        t1, d1 = stein.conv3d_tanh_tc(a[n:n + 1].contiguous(), W, b)
        assert torch.equal(act[n:n + 1], t1) and torch.equal(der[n:n + 1], d1), n
    assert torch.equal(part[:, z0:, y0:], act[:, z0:, y0:]) and torch.equal(pder[:, z0:, y0:], der[:, z0:, y0:])
    assert not part[:, :z0].any() and not part[:, :, :y0].any() and int(err) == 0
