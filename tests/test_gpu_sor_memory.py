"""The control variates' solve where device memory has room for the arrays that
it leaves behind but not for its working copies: it runs all the same, and h, its
residual and h . rho are bitwise those of the solve with room."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture
def limited():
    """coulps with an allocator that refuses single requests above limit['bytes']
    (counted in limit['refused'])."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps as cl
    _build.build()
    limit = {"bytes": None, "refused": 0}

    def alloc(nbytes, stream, ctx):
        if limit["bytes"] is not None and nbytes > limit["bytes"]:
            limit["refused"] += 1
            return None
        return torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))

    def free(ptr, stream, ctx):
        torch.cuda.caching_allocator_delete(int(ptr))

    cl.load()
    a, f = cl._ALLOC_T(alloc), cl._FREE_T(free)
    cl._check(cl.load().coulps_set_allocator(a, f, None), "coulps_set_allocator")
    cl._keep.extend([a, f])
    yield cl, limit
    cl.use_torch_allocator()


@pytest.mark.parametrize("L,n_iter", [((33, 57, 29), 25), ((64, 40, 50), 60), ((127, 5, 64), 12)])
def test_solve_without_room(limited, L, n_iter):
    import torch
    cl, limit = limited
    n = L[0] * L[1] * L[2]
    rng = np.random.default_rng(sum(L))
    sites = np.stack([rng.integers(0, v, 9) for v in L], axis=1).astype(np.int32)
    sites[5:] = sites[:4]  # two charges a site
    q = rng.uniform(-1, 1, 9)
    lat = cl.Lattice(L, n_chains=1, precision=cl.F32, seed=1, stream=torch.cuda.Stream())
    ch = cl.Charges(lat, sites, q)
    b = cl.Batch([(8, 9, 10), L], precision=cl.F32, seed=1, stream=torch.cuda.Stream())
    b.set_charges([(sites[:1] * 0, q[:1]), (sites, q)])

    def make(cls, of, room):
        limit["bytes"], limit["refused"] = room, 0
        g = cls(of, n_iter=n_iter, R=1)
        limit["bytes"] = None
        assert (limit["refused"] > 0) == (room is not None)
        return g

    # room for arrays of one double a site; the working copies have ghosts besides
    for cls, of, room in ((cl.GlobalCV, ch, 8 * n), (cl.BatchGlobalCV, b, 8 * (720 + n))):
        with_room, without = make(cls, of, None), make(cls, of, room)
        for k in ((),) if cls is cl.GlobalCV else ((0,), (1,)):
            h = with_room.h(*k)
            assert np.array_equal(h, without.h(*k)) and np.abs(h).max() > 0
        a, c = with_room.info(), without.info()
        assert all(np.array_equal(a[key], c[key]) for key in a)
        with_room.close()
        without.close()
    for o in (ch, lat, b):
        o.close()
