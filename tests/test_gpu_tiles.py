"""Tiles and plans taken by an estimate of the launch (lattices and batches from
2^19 sites, FP64 lattices of any size; FP64 without pass pairs; resident
launches of one sweep): whatever is taken, the fields are bitwise those of the
half-sweep kernels alone, and the samples agree up to the order of the FP64 sums
over the charges (1e-13, as between any two tiles).  Shapes that leave remainders
in every direction, rows of odd quads, few and many chains, one and two streams."""
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


def _same(a, b):
    assert np.abs(a[0] - b[0]).max() <= 1e-13 * np.abs(a[0]).max()
    for x, y in zip(a[1], b[1]):
        assert np.array_equal(x, y)
    assert a[2] == b[2]


@pytest.mark.parametrize("L,chains,prec,mix,streams", [
    ((90, 70, 110), 1, "F32", (1, 3), 1),
    ((37, 53, 71), 9, "F32", (1, 4), 2),
    ((300, 41, 59), 2, "F32", (1, 2), 1),
    ((20, 401, 31), 5, "F32", (0, 5), 1),
    ((96, 96, 96), 16, "F32", (1, 3), 2),
    ((290, 33, 64), 2, "F32", (1, 3), 1),
    ((61, 47, 53), 6, "F64", (1, 3), 2),
    ((130, 37, 120), 1, "F64", (1, 2), 1),
    ((9, 200, 5), 1, "F64", (0, 3), 1),
])
def test_chosen_tiles_equal_half_sweeps(cl, L, chains, prec, mix, streams):
    import torch
    from paper_1403_0711_gb300 import inputs
    out = []
    for fused in (0, None):
        lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=7,
                         stream=torch.cuda.Stream())
        lat.set_streams(streams)
        if fused is not None:
            lat.set_tile(min(L[1], 4), 5)
            lat.set_fused(fused)
        c = cl.Charges(lat, *inputs.uniform_q(L, 40, seed=2), log_capacity=8)
        lat.sweep(1, 1, 1)
        c.run(1, 4, *mix)
        out.append((c.samples(), [lat.field(k) for k in {0, chains - 1}], lat.info()["pass"]))
        c.close()
        lat.close()
    _same(*out)


@pytest.mark.parametrize("prec", ["F32", "F64"])
@pytest.mark.parametrize("dims", [
    [(90, 70, 50), (37, 53, 71), (17, 95, 45), (48, 31, 20)],
    [(33, 20, 14)] * 60 + [(14, 33, 20), (400, 9, 11)],
    [(64, 64, 64)] * 3 + [(5, 7, 300)],
])
def test_chosen_batch_tiles_equal_half_sweeps(cl, dims, prec):
    import torch
    from paper_1403_0711_gb300 import inputs
    assert sum(x * y * z for x, y, z in dims) >= 1 << 19
    charges = [inputs.uniform_q(d, 20, seed=5 + k) for k, d in enumerate(dims)]
    for mix in ((1, 0), (1, 3), (0, 4)):
        out = []
        for fused in (0, None):
            b = cl.Batch(dims, precision=getattr(cl, prec), seed=3, stream=torch.cuda.Stream())
            if fused is not None:
                b.set_fused(fused)
                b.set_tiles([(min(d[1], 3), 7) for d in dims])
            b.set_charges(charges, log_capacity=8)
            b.sweep(1, 1, 1)
            b.run(1, 3, *mix)
            out.append((b.samples(), [b.field(k) for k in (0, len(dims) // 2, len(dims) - 1)],
                        b.info()["pass"]))
            b.close()
        _same(*out)


@pytest.mark.parametrize("L,chains,prec", [((16, 16, 16), 3, "F32"), ((61, 47, 53), 12, "F32"),
                                           ((64, 64, 64), 1, "F32"), ((24, 25, 9), 30, "F64")])
def test_single_sweep_launches(cl, L, chains, prec):
    """One sweep per launch (off-lattice samples between): resident where its
    launch, load and store are counted in, bitwise the march kernels' fields
    and, the gather being the same kernel, their samples."""
    import torch
    out = []
    for pin in (True, False):
        lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=4,
                         stream=torch.cuda.Stream())
        if pin:
            lat.set_fused(3)
        rng = np.random.default_rng(1)
        pos = rng.uniform(2, np.array(L) - 3, size=(6, 3))
        c = cl.Charges.off_lattice(lat, pos, np.array([1.0, -1.0] * 3), log_capacity=16)
        c.run(1, 10, 1, 3)
        c.run(1, 2, 1, 0)
        out.append((c.samples(), [lat.field(k) for k in {0, chains - 1}], lat.info()["pass"]))
        c.close()
        lat.close()
    _same(*out)


@pytest.mark.parametrize("L,chains,prec,n,R", [
    ((23, 18, 15), 3, "F32", 30, 1),     # whole runs of 512 elements and a rest
    ((16, 16, 16), 40, "F32", 700, 2),   # several charges a warp, an odd count
    ((5, 4, 3), 2, "F32", 4, 4),         # a cube larger than the box
    ((40, 33, 20), 90, "F32", 801, 1),
    ((23, 18, 15), 40, "F64", 301, 1),
    ((9, 8, 7), 1, "F64", 5, 0),
])
def test_control_variate_sums(cl, L, chains, prec, n, R):
    """T g of the first and last chain against a direct evaluation in FP64 from
    the field and h.  Bound: FP32 fields round each product and each cube point's
    seven terms, |error| <= 32 * 2^-24 * (sum of magnitudes); FP64 fields 1e-12."""
    import torch
    from oracle import stein as ost
    from paper_1403_0711_gb300 import inputs
    sites, q = inputs.uniform_q(L, n, seed=6)
    lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=2,
                     stream=torch.cuda.Stream())
    lat.sweep(4, 1, 2)
    c = cl.Charges(lat, sites, q)
    g = cl.GlobalCV(c, n_iter=60, R=R)
    tg = torch.zeros(chains, dtype=torch.float64, device="cuda")
    g.eval(tg.data_ptr())
    lat.sync()
    h = g.h().astype(np.float64)
    v = ost.apply_A(h)
    k = ost.cube_green(R).astype(np.float32).astype(np.float64) if R > 0 else None
    rho = np.zeros(L[::-1])
    for (x, y, z), qi in zip(np.asarray(sites), q):
        rho[z, y, x] += qi
    eps = 32 * 2.0 ** -24 if prec == "F32" else 1e-12
    for ch in {0, chains - 1}:
        phi = np.asarray(lat.field(ch), dtype=np.float64)
        Q = float(np.sum(rho * phi))
        ref = g.info()["h_dot_rho"] - Q * float(np.sum(v * phi))
        scale = abs(g.info()["h_dot_rho"]) + abs(Q) * float(np.sum(np.abs(v * phi)))
        if R > 0:
            ref += ost.local_p_stein_term(phi, sites, q, k)
            amax = float(np.abs(phi).max())
            scale += 12 * amax * float(np.abs(k).sum()) * float(
                sum(qi * qi * abs(phi[z, y, x]) for (x, y, z), qi in zip(np.asarray(sites), q)))
        assert abs(float(tg[ch]) - ref) <= eps * scale, (ch, float(tg[ch]), ref, scale)
    g.close()
    c.close()
    lat.close()
