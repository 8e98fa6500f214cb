"""Tuning never makes a lattice or a batch slower: a small lattice that runs
resident in shared memory goes on so, lattices and batches of chosen tiles keep
them where the tuned ones are slower.  Times are the best of several runs of
measured sweeps; 1.3 is allowed for what two such runs of one side differ by."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    import os

    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, autotune, coulps, inputs
    _build.build()
    coulps.load()
    coulps.use_torch_allocator()
    os.environ["COULPS_TUNE_CACHE"] = str(tmp_path_factory.mktemp("tune") / "tune.json")
    return torch, coulps, autotune, inputs


def _time(run, sync, n):
    run(3)
    sync()
    out = []
    for _ in range(7):
        t = time.perf_counter()
        run(n)
        sync()
        out.append((time.perf_counter() - t) / n)
    return min(out)


@pytest.mark.parametrize("L,chains,prec,mix,n", [((16, 16, 16), 1, "F32", (1, 3), 1000),
                                                 ((16, 16, 16), 1, "F64", (1, 0), 1000),
                                                 ((61, 47, 53), 12, "F32", (1, 2), 300),
                                                 ((96, 96, 96), 16, "F32", (1, 3), 100)])
def test_tuned_lattice_is_no_slower(env, L, chains, prec, mix, n):
    torch, cl, autotune, inputs = env
    out = []
    for tune in (False, True):
        lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=3,
                         stream=torch.cuda.Stream())
        if tune:
            best = autotune.tune_lattice(lat, *mix, reps=1)
            assert (lat.info()["ty"], lat.info()["dz"]) == best
        c = cl.Charges(lat, *inputs.uniform_q(L, 8, seed=1), log_capacity=4)
        c.run(0, 4, *mix)
        s, f = c.samples(), lat.field(chains - 1)
        out.append((_time(lambda k: c.run(0, k, *mix), lat.sync, n), s, f))
        c.close()
        lat.close()
    assert np.array_equal(out[0][2], out[1][2])
    assert np.abs(out[0][1] - out[1][1]).max() <= 1e-13 * np.abs(out[0][1]).max()
    assert out[1][0] <= 1.3 * out[0][0], (out[0][0], out[1][0])


def test_tuned_batch_is_no_slower(env):
    torch, cl, autotune, inputs = env
    dims = [(37 + 7 * (k % 5), 40 + 9 * (k % 4), 50 + 8 * (k % 6)) for k in range(20)]
    out = []
    for tune in (False, True):
        b = cl.Batch(dims, precision=cl.F32, seed=1, stream=torch.cuda.Stream())
        if tune:
            best = autotune.tune_batch(b, 1, 0, reps=1)
            assert b.tiles() == [tuple(best[d]) for d in dims]
        b.set_charges([inputs.uniform_q(d, 4, seed=k) for k, d in enumerate(dims)])
        out.append(_time(lambda k: b.run(0, k, 1, 0), b.sync, 100))
        b.close()
    assert out[1] <= 1.3 * out[0], out


def test_way_back_to_the_automatic_choice(env):
    torch, cl, autotune, inputs = env
    lat = cl.Lattice((16, 16, 16), n_chains=2, precision=cl.F32, seed=3, stream=torch.cuda.Stream())
    assert lat.resident_enabled() and lat.resident(1, 3)[0] > 0
    for pin in (lambda: lat.set_tile(4, 4), lambda: lat.set_pass_tile(4), lambda: lat.set_fused(3),
                lambda: lat.set_pair_tile(4), lambda: lat.set_resident(False)):
        pin()
        assert not lat.resident_enabled() and lat.resident(1, 3) == (0, 1)
        lat.set_resident()
        assert lat.resident_enabled() and lat.resident(1, 3)[0] > 0
    with pytest.raises(cl.CoulpsError):
        cl._check(cl.load().coulps_set_resident(lat.handle, 2), "coulps_set_resident")
    lat.close()


def test_user_set_tiles_stay_pinned(env):
    torch, cl, autotune, inputs = env
    lat = cl.Lattice((16, 16, 16), n_chains=1, precision=cl.F32, seed=3, stream=torch.cuda.Stream())
    lat.set_fused(2)
    autotune.tune_lattice(lat, reps=1)
    assert not lat.resident_enabled() and lat.info()["fused"] == 2
    lat.close()
