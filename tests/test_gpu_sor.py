"""The control variates' SOR solve (sor.cu) iterate by iterate against a plain
FP64 red/black SOR, over edges that leave odd rows, boxes of one site and of
one plane, and charges that share a site.  h is u rounded to a grid of at most
13 max|u| 2^-23, half of which (8e-7 max|u|) is the tolerance."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _sor(L, rho, n_iter):
    Lx, Ly, Lz = L
    rj = sum(math.cos(math.pi / (n + 1)) for n in L) / 3.0
    w = 2.0 / (1.0 + math.sqrt(1.0 - rj * rj))
    u = np.zeros((Lz + 2, Ly + 2, Lx + 2))
    z, y, x = np.meshgrid(np.arange(Lz), np.arange(Ly), np.arange(Lx), indexing="ij")
    for _ in range(n_iter):
        for c in (0, 1):
            S = (u[:-2, 1:-1, 1:-1] + u[2:, 1:-1, 1:-1] + u[1:-1, :-2, 1:-1] + u[1:-1, 2:, 1:-1] +
                 u[1:-1, 1:-1, :-2] + u[1:-1, 1:-1, 2:])
            i = u[1:-1, 1:-1, 1:-1]
            i[...] = np.where((x + y + z) % 2 == c, (1 - w) * i + w * (S - rho) / 6.0, i)
    return u[1:-1, 1:-1, 1:-1]


@pytest.mark.parametrize("n_iter", [0, 1, 7, 60])
@pytest.mark.parametrize("L", [(1, 1, 1), (2, 3, 1), (9, 1, 17), (33, 17, 9), (300, 5, 2), (16, 64, 64)])
def test_iterates(L, n_iter):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps as cl
    _build.build()
    cl.use_torch_allocator()
    rng = np.random.default_rng(sum(L))
    n = 12
    sites = np.stack([rng.integers(0, v, n) for v in L], axis=1).astype(np.int32)
    sites[n // 2:] = sites[:n - n // 2]
    q = rng.uniform(-1, 1, n)
    rho = np.zeros(L[::-1])
    np.add.at(rho, (sites[:, 2], sites[:, 1], sites[:, 0]), q)
    ref = _sor(L, rho, n_iter)
    lat = cl.Lattice(L, n_chains=1, precision=cl.F32, seed=1, stream=torch.cuda.Stream())
    ch = cl.Charges(lat, sites, q)
    g = cl.GlobalCV(ch, n_iter=n_iter, R=0)
    b = cl.Batch([(5, 4, 3), L], precision=cl.F32, seed=1, stream=torch.cuda.Stream())
    b.set_charges([(sites[:1] * 0, q[:1]), (sites, q)])
    gb = cl.BatchGlobalCV(b, n_iter=n_iter, R=0)
    for h in (g.h(), gb.h(1)):
        assert np.abs(h - ref).max() <= 8e-7 * np.abs(ref).max()
    assert np.array_equal(g.h(), gb.h(1))
    for o in (g, gb, ch, b, lat):
        o.close()


@pytest.mark.parametrize("systems", [1, 3, 300])
def test_boxes_of_one_site(systems):
    """Colour 1 of such boxes has no site: its launches take part in the chain of
    dependent launches all the same.  h = -q / 6 for any number of iterations."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps as cl
    _build.build()
    cl.use_torch_allocator()
    q = np.random.default_rng(systems).uniform(-1, 1, systems)
    b = cl.Batch([(1, 1, 1)] * systems, precision=cl.F32, seed=1, stream=torch.cuda.Stream())
    b.set_charges([(np.zeros((1, 3), np.int32), q[k:k + 1]) for k in range(systems)])
    for n_iter in (1, 2, 400):
        g = cl.BatchGlobalCV(b, n_iter=n_iter, R=0)
        for k in {0, systems // 2, systems - 1}:
            assert abs(float(g.h(k).reshape(-1)[0]) + q[k] / 6.0) <= 8e-7 * abs(q[k] / 6.0)
        g.close()
    b.close()
