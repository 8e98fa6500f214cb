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


def test_derivatives_of_any_kind(env):
    """Double backward, forward-mode and vmap of the region divergence, as through
    the framework operations (the ones that a double-precision input takes); FP32
    against FP64: sums of 27 x 16 x 16 products per site over some hundred sites,
    1e-4 of the largest value."""
    torch, stein, cv = env
    a, b = _s(torch, cv), _s(torch, cv, seed=1)
    ta, tb = _s(torch, cv, seed=2), _s(torch, cv, seed=3)
    ws = [p.detach().clone() for p in cv.parameters()]

    def second(dtype):
        s1, s2 = a.to(dtype).requires_grad_(), b.to(dtype).requires_grad_()
        d = cv.region_divergence(s1, s2)
        g1, = torch.autograd.grad((d * d).sum(), s1, create_graph=True)
        return torch.autograd.grad((g1 * ta.to(dtype)).sum(), (s1, s2))

    def forward_mode(dtype):
        with torch.autograd.forward_ad.dual_level():
            dual = [torch.autograd.forward_ad.make_dual(x.to(dtype), t.to(dtype))
                    for x, t in ((a, ta), (b, tb))]
            return torch.autograd.forward_ad.unpack_dual(cv.region_divergence(*dual)).tangent

    def mapped(dtype):
        x = torch.stack([a, ta]).to(dtype), torch.stack([b, tb]).to(dtype)
        return torch.func.vmap(cv.region_divergence)(*x)

    def functional(dtype):
        f = lambda s: cv.region_divergence(s, b.to(dtype)).sum()  # noqa: E731
        return torch.func.grad(f)(a.to(dtype))

    for f in (second, forward_mode, mapped, functional):
        got = f(torch.float32)
        for p in cv.parameters():
            p.data = p.data.double()
        ref = f(torch.float64)
        for p, w in zip(cv.parameters(), ws):
            p.data = w.clone()
        for x, y in zip(got if isinstance(got, tuple) else (got,),
                        ref if isinstance(ref, tuple) else (ref,)):
            assert x.dtype == torch.float32 and float(y.abs().max()) > 0
            assert float((x.double() - y).abs().max()) <= 1e-4 * float(y.abs().max())
