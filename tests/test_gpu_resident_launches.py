"""The length of a resident launch: as many compound sweeps as last about 0.1 s,
whatever the lattice and the mix (twice that is allowed here, for the estimate's
error), and none for a mix whose single sweep would last longer.  Runs of several
launches are bitwise those of the march kernels in their fields and one by one
the same samples up to the order of the FP64 sums (1e-13)."""
import time

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


def _lattice(cl, L, chains, prec):
    import torch
    return cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=11,
                      stream=torch.cuda.Stream())


@pytest.mark.parametrize("L,chains,prec,mix,on", [
    ((64, 64, 64), 64, "F32", (1, 3), True),
    ((32, 32, 32), 100, "F64", (1, 3), True),
    ((16, 16, 16), 1, "F32", (1, 300), True),
    ((16, 16, 16), 1, "F64", (40, 0), True),
    ((8, 8, 8), 20000, "F32", (1, 3), False),
    ((5, 4, 3), 2, "F32", (1, 0), True),
])
def test_a_launch_lasts_a_tenth_of_a_second(cl, L, chains, prec, mix, on):
    lat = _lattice(cl, L, chains, prec)
    cluster, sweeps = lat.resident(*mix)
    assert (cluster > 0) == on and 1 <= sweeps <= (2048 if on else 1)
    lat.sweep(1, *mix)
    lat.sync()
    t = time.perf_counter()
    lat.sweep(sweeps, *mix)
    lat.sync()
    assert time.perf_counter() - t < 0.2
    lat.close()


def test_mixes_longer_than_a_launch_stay_with_the_march_kernels(cl):
    lat = _lattice(cl, (16, 16, 16), 1, "F32")
    for n_sweeps in (0, 1, 100):
        assert lat.resident(1, 3, n_sweeps)[0] > 0
        assert lat.resident(1, 10 ** 6, n_sweeps) == (0, 1)
    lat.close()


@pytest.mark.parametrize("L,chains,prec,mix", [((32, 32, 32), 100, "F64", (1, 3)),
                                               ((16, 16, 16), 3, "F32", (1, 60))])
def test_runs_of_several_launches(cl, L, chains, prec, mix):
    from paper_1403_0711_gb300 import inputs
    out = []
    for march in (False, True):
        lat = _lattice(cl, L, chains, prec)
        if not march:
            n = 2 * lat.resident(*mix)[1] + 3
        else:
            lat.set_fused(3)
            assert lat.resident(*mix) == (0, 1)
        c = cl.Charges(lat, *inputs.uniform_q(L, 50, seed=3), log_capacity=n)
        c.run(2, n, *mix)
        out.append((c.samples(), [lat.field(k) for k in {0, chains - 1}], lat.info()["pass"]))
        c.close()
        lat.close()
    assert out[0][0].shape == out[1][0].shape and out[0][2] == out[1][2]
    assert np.abs(out[0][0] - out[1][0]).max() <= 1e-13 * np.abs(out[1][0]).max()
    for x, y in zip(out[0][1], out[1][1]):
        assert np.array_equal(x, y)
