"""Runs of a few sweeps on lattices that count as resident: by the resident
kernel or by the march kernels with the resident kernel's sums from memory,
whichever is the sooner, bitwise the same samples, statistics and fields however
a run is divided into calls.  Lattices around the line between the two, with
several waves of clusters, charge counts of one and of several measuring warps,
planes without charges, no charges, two streams and a change of the mix between."""
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


def _charges(L, n):
    from paper_1403_0711_gb300 import inputs
    if n > L[0] * L[1] * L[2] // 2 or n == 0:  # repeated sites
        rng = np.random.default_rng(n)
        return np.stack([rng.integers(0, v, n) for v in L], axis=1).astype(np.int32), rng.uniform(-1, 1, n)
    return inputs.uniform_q(L, n, seed=3)


@pytest.mark.parametrize("L,chains,prec,mix,n", [
    ((40, 40, 40), 100, "F32", (1, 0), 200),
    ((40, 40, 40), 100, "F32", (1, 0), 6000),
    ((80, 80, 80), 4, "F32", (1, 3), 64),
    ((80, 80, 80), 4, "F32", (1, 3), 5000),
    ((35, 13, 81), 94, "F32", (1, 3), 3),
    ((119, 8, 68), 105, "F32", (1, 1), 700),
    ((10, 45, 67), 89, "F32", (1, 0), 0),
    ((65, 15, 20), 112, "F64", (0, 2), 300),
    ((30, 100, 23), 6, "F64", (0, 2), 2500),
    ((21, 18, 14), 5, "F64", (1, 3), 9000),
])
def test_divided_runs_bitwise(cl, L, chains, prec, mix, n):
    import torch
    sites, q = _charges(L, n)
    out = []
    for calls, streams in (((13,), 1), ((1,) * 13, 1), ((2, 1, 3, 1, 4, 2), 2), ((1, 9, 1, 2), 1)):
        lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=7,
                         stream=torch.cuda.Stream())
        lat.set_streams(streams)
        assert lat.resident(*mix)[0] > 0
        c = cl.Charges(lat, sites, q, log_capacity=13)
        lat.sweep(2, 1, 1)
        for k in calls:
            c.run(0, k, *mix)
        out.append((c.samples(), c.chain_stats(), [lat.field(k) for k in {0, chains - 1}],
                    lat.info()["pass"]))
        c.close()
        lat.close()
    a = out[0]
    for b in out[1:]:
        assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1]) and a[3] == b[3]
        assert all(np.array_equal(x, y) for x, y in zip(a[2], b[2]))


def test_short_runs_after_other_schedules_and_sets(cl):
    """The recorded step of a short run is its own: changes of the schedule, the
    charges, the set and the route in between leave the samples those of a lattice
    that does nothing else."""
    import torch
    L, chains, mix = (40, 40, 40), 100, (1, 0)
    sa, qa = _charges(L, 200)
    sb, qb = _charges(L, 77)

    def run(busy):
        lat = cl.Lattice(L, n_chains=chains, precision=cl.F32, seed=7, stream=torch.cuda.Stream())
        a = cl.Charges(lat, sa, qa, log_capacity=16)
        b = cl.Charges(lat, sb, qb)
        for k in range(6):
            a.run(0, 1, *mix)
            if busy and k == 1:
                b.run(0, 1, *mix)
            elif k == 1:
                lat.sweep(1, *mix)
            if busy and k == 2:
                lat.set_schedule(cl.SCHEDULE_SHIFTED)
                b.run(0, 1, *mix)
                lat.set_schedule(cl.SCHEDULE_ALIGNED)
            elif k == 2:
                lat.sweep(1, *mix)
            if busy and k == 3:
                lat.set_resident(False)
                b.run(0, 1, *mix)
                lat.set_resident()
            elif k == 3:
                lat.sweep(1, *mix)
            if k == 4:
                a.update(sb, qb) if len(sb) == len(sa) else a.update(sa[::-1].copy(), qa)
        a.run(0, 9, *mix)
        out = a.samples(), lat.field(chains - 1)
        for o in (a, b, lat):
            o.close()
        return out

    x, y = run(False), run(True)
    assert np.array_equal(x[0], y[0]) and np.array_equal(x[1], y[1])
