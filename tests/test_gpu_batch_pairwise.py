"""Batches alive side by side: their kernels share one limit of dynamic shared
memory, so a batch of small tiles made (or laid out again) later must leave the
one of large tiles able to launch, in every fused mode and for every mix, directly
and as the recorded step of a run.  Fields bitwise those of the batch on its own."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LARGE = [(200, 40, 40), (96, 64, 30)]
SMALL = [(5, 4, 6), (8, 3, 3)]


@pytest.fixture(scope="module")
def cl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps
    _build.build()
    coulps.load()
    coulps.use_torch_allocator()
    return coulps


def _batch(cl, dims, prec, mode):
    import torch
    from paper_1403_0711_gb300 import inputs
    b = cl.Batch(dims, precision=prec, seed=3, stream=torch.cuda.Stream())
    b.set_fused(mode)
    b.set_charges([inputs.uniform_q(d, 6, seed=k) for k, d in enumerate(dims)], log_capacity=8)
    return b


@pytest.mark.parametrize("prec", ["F32", "F64"])
@pytest.mark.parametrize("mode", [0, 1, 2, 3])
def test_small_tiles_do_not_stop_large_ones(cl, prec, mode):
    p, out = getattr(cl, prec), []
    for beside in (False, True):
        a = _batch(cl, LARGE, p, mode)
        for mix in ((1, 0), (1, 3), (0, 2)):
            a.sweep(1, *mix)
            if beside:
                b = _batch(cl, SMALL, p, mode)
                assert b.info()["smem"] < a.info()["smem"]
                b.sweep(1, *mix)
            a.sweep(1, *mix)
            a.run(1, 3, *mix)
            if beside:
                b.run(0, 2, *mix)
                b.close()
        out.append((a.samples(), [a.field(k) for k in range(len(LARGE))]))
        a.close()
    assert np.array_equal(out[0][0], out[1][0])
    for x, y in zip(out[0][1], out[1][1]):
        assert np.array_equal(x, y)
