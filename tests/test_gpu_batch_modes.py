"""The fused mode of an FP64 batch is what it says: from 2^19 sites on it is
created with fused passes (mode 1, no pair tiles laid out), set_fused(2) and
set_pair_tiles bring pass pairs, and every one of them gives bitwise the fields
of the half-sweeps."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LARGE = [(90, 70, 50), (37, 53, 71), (17, 95, 45), (48, 31, 20)]  # 557,000 sites
SMALL = [(20, 18, 16), (33, 20, 14)]


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


@pytest.mark.parametrize("prec,dims,default", [("F64", LARGE, 1), ("F64", SMALL, 2), ("F32", LARGE, 2)])
def test_mode_is_what_runs(cl, prec, dims, default):
    import torch
    from paper_1403_0711_gb300 import inputs
    charges = [inputs.uniform_q(d, 20, seed=5 + k) for k, d in enumerate(dims)]

    def run(prepare):
        b = cl.Batch(dims, precision=getattr(cl, prec), seed=3, stream=torch.cuda.Stream())
        mode = prepare(b)
        assert b.fused() == mode and (b.info()["pair_grid"] > 0) == (mode >= 2)
        b.set_charges(charges, log_capacity=8)
        b.sweep(2, 1, 4)
        b.run(1, 3, 1, 3)
        out = b.samples(), [b.field(k) for k in range(len(dims))]
        b.close()
        return out

    def tiles(b):
        b.set_pair_tiles([(min(d[1], 4), 9) for d in dims])
        return 2

    def given(mode, then=None):
        def prepare(b):
            b.set_fused(mode)
            if then:
                then(b)
            return mode
        return prepare

    ref = run(given(0))
    for prepare in (lambda b: default, given(1), given(2), given(3), tiles, given(1, tiles),
                    given(2, tiles)):
        s, f = run(prepare)
        assert np.abs(s - ref[0]).max() <= 1e-13 * np.abs(ref[0]).max()
        assert all(np.array_equal(x, y) for x, y in zip(f, ref[1]))


def test_many_small_fp64_systems(cl):
    """One pass tile per system, about four to an SM: their CTAs take them in turn."""
    import torch
    from paper_1403_0711_gb300 import inputs
    rng = np.random.default_rng(4)
    dims = [tuple(int(v) for v in rng.choice([12, 17, 25], 3)) for _ in range(500)]
    charges = [inputs.uniform_q(d, 9, seed=k % 5) for k, d in enumerate(dims)]
    out = []
    for mode in (0, 1):
        b = cl.Batch(dims, precision=cl.F64, seed=3, stream=torch.cuda.Stream())
        b.set_fused(mode)
        b.set_charges(charges, log_capacity=8)
        b.sweep(1, 1, 0)
        b.run(1, 3, 0, 2)
        b.run(0, 2, 1, 3)
        out.append((b.samples(), [b.field(k) for k in range(0, 500, 83)]))
        b.close()
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-13 * np.abs(out[0][0]).max()
    assert all(np.array_equal(x, y) for x, y in zip(out[0][1], out[1][1]))
