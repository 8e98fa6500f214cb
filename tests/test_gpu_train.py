"""The training kernels of the learned control variate against the framework
operations that they stand for, bitwise: packed weights, the activations and
their backward with either gradient missing, and the neighbours' gather and
its backward for regions inside the box, clipped by its faces and one site
thick, and for sample counts around the kernels' groups of 8."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps, stein
    _build.build()
    return torch, coulps.load(), stein


def test_pack_weights_equals_host(env):
    torch, lib, stein = env
    W = torch.randn(16, 16, 3, 3, 3, generator=torch.Generator().manual_seed(1))
    W.view(-1)[:4] = torch.tensor([0.0, -0.0, float("inf"), 1e-42])
    ref = np.zeros(27 * 256, dtype=np.uint16)
    w = W.numpy()
    assert lib.coulps_cv_pack_weights(w.ctypes.data_as(ctypes.POINTER(ctypes.c_float)),
                                      ref.ctypes.data_as(ctypes.POINTER(ctypes.c_uint16))) == 0
    for v in (W.cuda(), W.cuda().transpose(0, 1).contiguous().transpose(0, 1)):
        assert np.array_equal(stein.pack_weights(v).cpu().numpy().view(np.uint16), ref)


@pytest.mark.parametrize("use", ["both", "a", "s"])
def test_act_equals_operations(env, use):
    torch, lib, stein = env
    g = torch.Generator(device="cuda").manual_seed(2)
    h = 3 * torch.randn(3, 5, 4, 7, 16, generator=g, device="cuda")
    h.view(-1)[:5] = torch.tensor([0.0, -0.0, 30.0, -30.0, 1e-30], device="cuda")
    u = torch.randn(h.shape, generator=g, device="cuda").to(torch.bfloat16)
    v = torch.randn(h.shape, generator=g, device="cuda")
    h1, h2 = h.clone().requires_grad_(), h.clone().requires_grad_()
    a, s = stein._Act.apply(h1)
    t = torch.tanh(h2)
    st = 1.0 - t * t
    at = t.to(torch.bfloat16)
    st = st + (st.to(torch.bfloat16).float() - st).detach()
    assert torch.equal(a, at) and torch.equal(s, st)
    out = {"both": ((a, s), (at, st), (u, v)), "a": ((a,), (at,), (u,)), "s": ((s,), (st,), (v,))}[use]
    torch.autograd.backward(out[0], out[2])
    torch.autograd.backward(out[1], out[2])
    assert torch.equal(h1.grad, h2.grad)


@pytest.mark.parametrize("n", [1, 8, 11])
@pytest.mark.parametrize("E,lo,hi", [((9, 8, 7), (2, 2, 2), (6, 5, 4)), ((6, 5, 4), (0, 0, 0), (6, 5, 4)),
                                     ((5, 9, 3), (0, 4, 0), (5, 5, 2)), ((1, 1, 1), (0, 0, 0), (1, 1, 1)),
                                     ((24, 22, 20), (2, 2, 2), (22, 20, 18))])
def test_neighbours_equal_operations(env, E, lo, hi, n):
    torch, lib, stein = env
    ex, ey, ez = E
    g = torch.Generator(device="cuda").manual_seed(sum(E) + n)
    s = torch.randn(n, ez, ey, ex, 16, generator=g, device="cuda")
    s1, s2 = s.clone().requires_grad_(), s.clone().requires_grad_()
    got = stein._Neighbours.apply(s1 * 1.0, lo, hi)
    q = torch.tensor([(z, y, x) for z in range(lo[2], hi[2]) for y in range(lo[1], hi[1])
                      for x in range(lo[0], hi[0])], device="cuda")
    p = torch.nn.functional.pad(s2 * 1.0, (0, 0, 1, 1, 1, 1, 1, 1))
    ref = torch.stack([p[:, q[:, 0] + 1 + o[0], q[:, 1] + 1 + o[1], q[:, 2] + 1 + o[2]]
                       for o in stein.OFFS], dim=2)
    assert torch.equal(got, ref)
    d = torch.randn(ref.shape, generator=g, device="cuda")
    got.backward(d)
    ref.backward(d)
    assert torch.equal(s1.grad, s2.grad)
