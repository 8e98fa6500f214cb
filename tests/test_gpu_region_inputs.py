"""Inputs of LocalSteinCV.region_divergence that the gather kernel must not take
as they are: another number of channels is refused as by the framework
operations (the kernel reads 16 whatever the tensor holds), no samples give no
values, and a tensor that starts off a 16-byte boundary gives what an aligned
one does, in the values and in the gradient."""
import pytest

pytestmark = pytest.mark.gpu

L, LO, HI = (10, 9, 8), (3, 3, 2), (6, 5, 6)


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps, stein
    _build.build()
    coulps.load()
    return torch, stein, stein.LocalSteinCV(L, LO, HI, seed=2, w3_scale=0.3)


def _s(torch, cv, n=3, c=16, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ex, ey, ez = cv.edims
    return torch.rand(n, ez, ey, ex, c, generator=g, device="cuda")


@pytest.mark.parametrize("channels", [8, 15, 17, 32])
def test_other_channel_counts_are_refused(env, channels):
    torch, stein, cv = env
    with pytest.raises(RuntimeError):
        cv.region_divergence(_s(torch, cv, c=channels), _s(torch, cv))
    with pytest.raises(ValueError):
        stein._Neighbours.apply(_s(torch, cv, c=channels), [1, 1, 1], [3, 3, 3])


def test_no_samples(env):
    torch, stein, cv = env
    assert cv.region_divergence(_s(torch, cv, n=0), _s(torch, cv, n=0)).shape == (0,)


def test_unaligned_start(env):
    torch, stein, cv = env
    a, s2 = _s(torch, cv), _s(torch, cv, seed=1)
    out = []
    for off in (0, 1):
        base = torch.zeros(a.numel() + 4, device="cuda")
        s1 = base[off:off + a.numel()].view(a.shape)
        s1.copy_(a)
        s1.requires_grad_()
        d = cv.region_divergence(s1, s2)
        d.backward(torch.linspace(1, 2, len(d), device="cuda"))
        out.append((d.detach(), s1.grad))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
