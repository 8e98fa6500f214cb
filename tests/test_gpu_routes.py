"""Which kernels the bitwise comparisons run: resident cases that the estimate
does take resident (asked, not assumed), with several heatbath passes in FP32 and
boxes up to the largest that fit, and FP64 pass pairs, which no default takes,
with tiles of their own (counted by the kernel timers).  Fields bitwise those of
the half-sweeps, samples up to the order of the FP64 sums (1e-13)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


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


def _run(cl, L, chains, prec, mix, prepare):
    import torch
    from paper_1403_0711_gb300 import inputs
    lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=11,
                     stream=torch.cuda.Stream())
    prepare(lat)
    n = max(1, min(40, L[0] * L[1] * L[2] // 2))
    c = cl.Charges(lat, *inputs.uniform_q(L, n, seed=3), log_capacity=8)
    lat.sweep(2, *mix)
    c.run(0, 3, *mix)
    out = c.samples(), [lat.field(k) for k in {0, chains - 1}], lat.info()["pass"]
    c.close()
    lat.close()
    return out


def _same(a, b):
    assert np.abs(a[0] - b[0]).max() <= 1e-13 * max(np.abs(b[0]).max(), 1e-300)
    assert all(np.array_equal(x, y) for x, y in zip(a[1], b[1])) and a[2] == b[2]


@pytest.mark.parametrize("L,chains,prec,mix", [
    ((64, 64, 64), 8, "F32", (2, 5)),
    ((64, 64, 64), 30, "F32", (2, 3)),
    ((200, 40, 40), 2, "F32", (2, 2)),
    ((80, 80, 80), 4, "F32", (1, 3)),
    ((61, 47, 53), 30, "F32", (1, 3)),
    ((13, 7, 5), 40, "F64", (2, 1)),
    ((257, 5, 6), 2, "F64", (1, 3)),
])
def test_resident_cases_run_resident(cl, L, chains, prec, mix):
    def resident(lat):
        assert lat.resident(*mix)[0] > 0

    def half_sweeps(lat):
        lat.set_fused(0)
        assert lat.resident(*mix)[0] == 0

    _same(_run(cl, L, chains, prec, mix, resident), _run(cl, L, chains, prec, mix, half_sweeps))


@pytest.mark.parametrize("mode", [3, 4])
@pytest.mark.parametrize("L,mix,tile", [
    ((21, 18, 12), (2, 3), (18, 12)),
    ((16, 16, 16), (2, 2), (16, 16)),
    ((16, 16, 16), (1, 4), (5, 3)),
    ((9, 1, 1), (1, 2), (1, 1)),
    ((61, 47, 53), (1, 3), (10, 16)),
    ((130, 37, 20), (0, 4), (9, 20)),
])
def test_fp64_pairs(cl, L, mix, tile, mode):
    import torch

    def pairs(lat):
        lat.set_fused(mode)
        lat.set_pair_tile(*tile)
        assert lat.pair_tile() == tile

    def half_sweeps(lat):
        lat.set_fused(0)

    _same(_run(cl, L, 2, "F64", mix, pairs), _run(cl, L, 2, "F64", mix, half_sweeps))
    lat = cl.Lattice(L, n_chains=2, precision=cl.F64, seed=1, stream=torch.cuda.Stream())
    pairs(lat)
    lat.set_profiling(True)
    lat.sweep(1, *mix)
    t = lat.kernel_times()
    assert t["pair_or_n"] + t["pair_hb_n"] > 0
    lat.close()
