"""Resident sweeps of small lattices (resident.cu) against the march kernels
(selected by set_fused): bitwise the same fields, pass counter and estimates
up to the order of the FP64 sums over the charges (1e-13, as between the march
kernels' tiles), over box shapes that leave remainders in every direction, one
and several CTAs per chain, both precisions, chains in several waves, more
charges than the measuring threads' registers hold, mixes without heatbath or
over-relaxation passes, and runs longer than one launch."""
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


def _run(cl, L, chains, prec, n, mix, meas, march, split=False, streams=1):
    import torch
    from paper_1403_0711_gb300 import inputs
    lat = cl.Lattice(L, n_chains=chains, precision=prec, seed=11, stream=torch.cuda.Stream())
    if march:
        lat.set_fused(3)
    lat.set_streams(streams)
    ch = cl.Charges(lat, *inputs.uniform_q(L, n, seed=3), log_capacity=2 * meas)
    lat.sweep(2, *mix)
    if split:
        for _ in range(meas):
            ch.run(0, 1, *mix)
    else:
        ch.run(0, meas, *mix)
    ch.measure()
    out = (ch.samples(), [lat.field(k) for k in {0, chains // 2, chains - 1}], ch.chain_stats(),
           lat.info()["pass"])
    ch.close()
    lat.close()
    return out


def _same(a, b):
    scale = np.abs(a[0]).max()
    assert np.abs(a[0] - b[0]).max() <= 1e-13 * max(scale, 1e-300)
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)
    assert a[3] == b[3]


@pytest.mark.parametrize("L,chains,prec,n,mix,meas", [
    ((1, 1, 1), 2, "F32", 1, (1, 1), 4),
    ((2, 3, 4), 3, "F64", 3, (1, 2), 4),
    ((13, 7, 5), 2, "F32", 30, (1, 3), 6),
    ((13, 7, 5), 40, "F64", 30, (2, 1), 6),
    ((16, 16, 16), 1, "F64", 8, (1, 0), 70),
    ((8, 8, 8), 200, "F32", 64, (1, 3), 6),
    ((20, 31, 9), 4, "F64", 400, (0, 2), 5),
    ((61, 47, 53), 12, "F32", 501, (1, 2), 5),
    ((61, 47, 53), 30, "F32", 2, (1, 3), 4),
    ((40, 23, 19), 2, "F32", 6000, (1, 3), 5),
    ((40, 23, 19), 3, "F64", 6000, (1, 1), 5),
    ((257, 5, 6), 2, "F32", 40, (0, 1), 5),
    ((257, 5, 6), 2, "F64", 40, (1, 3), 5),
    ((9, 100, 16), 3, "F32", 50, (0, 2), 5),
    ((64, 64, 64), 64, "F32", 4096, (1, 3), 3),
    ((80, 80, 80), 4, "F32", 64, (2, 5), 3),
    ((5, 4, 3), 2, "F32", 6, (1, 1), 2100),
])
def test_resident_equals_march(cl, L, chains, prec, n, mix, meas):
    p = getattr(cl, prec)
    _same(_run(cl, L, chains, p, n, mix, meas, True), _run(cl, L, chains, p, n, mix, meas, False))


@pytest.mark.parametrize("prec", ["F32", "F64"])
def test_resident_split_runs_bitwise(cl, prec):
    """Call by call and in one call, and with the streams of the march kernels asked for."""
    p = getattr(cl, prec)
    a = _run(cl, (21, 18, 14), 5, p, 60, (1, 3), 9, False)
    for b in (_run(cl, (21, 18, 14), 5, p, 60, (1, 3), 9, False, split=True),
              _run(cl, (21, 18, 14), 5, p, 60, (1, 3), 9, False, streams=2)):
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[2], b[2]) and a[3] == b[3]
        for x, y in zip(a[1], b[1]):
            assert np.array_equal(x, y)


def test_streams_with_sets_and_global_cv_on_march_kernels(cl):
    """The march kernels' stream split under multi-set runs and the global control variate."""
    import torch
    from paper_1403_0711_gb300 import inputs
    L, out = (20, 18, 16), []
    for n in (1, 2, 4):
        lat = cl.Lattice(L, n_chains=4, precision=cl.F32, seed=43, stream=torch.cuda.Stream())
        lat.set_fused(3)
        lat.set_streams(n)
        cs = [cl.Charges(lat, *inputs.uniform_q(L, 33, seed=k), log_capacity=6) for k in (1, 2)]
        cl.run_sets(lat, cs, 2, 6, 1, 3)
        g = cl.GlobalCV(cs[0], R=0)
        g.run(8, 1, 3, 1.0)
        out.append(([c.samples() for c in cs], cs[0].cv_chain_stats(), lat.field(3)))
        g.close()
        for c in cs:
            c.close()
        lat.close()
    for b in out[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(out[0][0], b[0]))
        assert np.array_equal(out[0][1], b[1]) and np.array_equal(out[0][2], b[2])
