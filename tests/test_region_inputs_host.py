"""Which tensors the region gather takes (the choice made before any pointer is
passed on), with stand-ins for CUDA tensors."""
import types

import pytest

torch = pytest.importorskip("torch")


def _t(shape, dtype=torch.float32, is_cuda=True):
    return types.SimpleNamespace(shape=shape, dtype=dtype, is_cuda=is_cuda, dim=lambda: len(shape))


def test_only_rows_of_16_float32_channels():
    from paper_1403_0711_gb300 import stein
    lo, hi = [1, 1, 1], [5, 4, 3]
    assert stein._gatherable(_t((2, 6, 7, 8, 16)), lo, hi)
    for bad in (_t((2, 6, 7, 8, 8)), _t((2, 6, 7, 8, 17)), _t((0, 6, 7, 8, 16)),
                _t((2, 6, 7, 8, 16), torch.float64), _t((2, 6, 7, 8, 16), is_cuda=False),
                _t((6, 7, 8, 16))):
        assert not stein._gatherable(bad, lo, hi)
    # the scatter's limit, 56320 sites of the box grown by one
    assert stein._gatherable(_t((1, 90, 90, 90, 16)), [0, 0, 0], [38, 30, 42])   # 40 x 32 x 44
    assert not stein._gatherable(_t((1, 90, 90, 90, 16)), [0, 0, 0], [38, 30, 43])


def test_neighbours_refuse_what_they_would_misread():
    from paper_1403_0711_gb300 import stein
    for t in (torch.zeros(1, 4, 4, 4, 8), torch.zeros(1, 4, 4, 4, 16)):  # 8 channels; not CUDA
        with pytest.raises(ValueError):
            stein._Neighbours.apply(t, [1, 1, 1], [2, 2, 2])


def test_transforms_and_tracers_keep_the_framework_operations():
    from paper_1403_0711_gb300 import stein
    x = torch.ones(2, 3)
    seen = []

    def f(t):
        seen.append(stein._plain(t))
        return (t * t).sum()

    f(x)
    f(torch.nn.Parameter(x))
    assert seen == [True, True]
    seen.clear()
    torch.func.grad(f)(x)
    torch.func.vmap(f)(x)
    torch.func.jvp(f, (x,), (x,))
    torch.jit.trace(f, x, check_trace=False)
    with torch.autograd.forward_ad.dual_level():
        f(torch.autograd.forward_ad.make_dual(x, x))
    from torch.fx.experimental.proxy_tensor import make_fx
    make_fx(f)(x)
    assert len(seen) == 6 and not any(seen)
