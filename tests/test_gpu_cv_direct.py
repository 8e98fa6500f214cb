"""T g of the control variates by both forms of the local term (a warp per charge;
charge neighbourhoods in shared memory), on either side of the line between them,
for every radius and precision, lattices and batches, against a direct evaluation in
FP64 from the field and h.  Bounds as for the control variate's sums elsewhere: FP32
fields round each product and each cube point's seven terms, |error| <= 32 * 2^-24 *
(sum of magnitudes); FP64 fields 1e-12."""
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


def _check(phi, h, sites, q, R, f32, got):
    from oracle import stein as ost
    phi, h = np.asarray(phi, np.float64), h.astype(np.float64)
    v = ost.apply_A(h)
    rho = np.zeros(phi.shape)
    np.add.at(rho, (sites[:, 2], sites[:, 1], sites[:, 0]), q)
    Q, hr = float(np.sum(rho * phi)), float(np.sum(h * rho))
    k = ost.cube_green(R).astype(np.float32).astype(np.float64)
    ref = hr - Q * float(np.sum(v * phi)) + ost.local_p_stein_term(phi, sites, q, k)
    scale = abs(hr) + abs(Q) * float(np.sum(np.abs(v * phi)))
    scale += 12 * float(np.abs(phi).max()) * float(np.abs(k).sum()) * float(
        np.sum(q * q * np.abs(phi[sites[:, 2], sites[:, 1], sites[:, 0]])))
    assert abs(got - ref) <= (32 * 2.0 ** -24 if f32 else 1e-12) * scale, (got, ref, scale)


@pytest.mark.parametrize("prec,R,chains,n", [
    ("F32", 1, 80, 299), ("F32", 1, 80, 301),     # 24000 charges in all
    ("F32", 2, 120, 399), ("F32", 2, 120, 401),   # 48000
    ("F32", 3, 160, 601), ("F32", 3, 2, 40), ("F32", 4, 3, 200),
    ("F64", 1, 25, 399), ("F64", 1, 25, 401),     # 10000
    ("F64", 2, 3, 40), ("F64", 3, 9, 33), ("F64", 4, 2, 500),
])
def test_lattice(cl, prec, R, chains, n):
    import torch
    from paper_1403_0711_gb300 import inputs
    L = (19, 14, 12)
    sites, q = inputs.uniform_q(L, n, seed=6)
    lat = cl.Lattice(L, n_chains=chains, precision=getattr(cl, prec), seed=2,
                     stream=torch.cuda.Stream())
    lat.sweep(4, 1, 2)
    c = cl.Charges(lat, sites, q)
    g = cl.GlobalCV(c, n_iter=60, R=R)
    tg = torch.zeros(chains, dtype=torch.float64, device="cuda")
    g.eval(tg.data_ptr())
    lat.sync()
    for k in {0, chains - 1}:
        _check(lat.field(k), g.h(), np.asarray(sites), q, R, prec == "F32", float(tg[k]))
    for o in (g, c, lat):
        o.close()


@pytest.mark.parametrize("prec,R,systems,n", [
    ("F32", 1, 100, 399), ("F32", 1, 100, 401),   # 40000 charges in all
    ("F32", 2, 200, 401), ("F32", 3, 5, 30), ("F32", 4, 320, 1001),
    ("F64", 1, 100, 399), ("F64", 1, 100, 401), ("F64", 2, 200, 401),
    ("F64", 3, 7, 100), ("F64", 4, 40, 301),
])
def test_batch(cl, prec, R, systems, n):
    import torch
    from paper_1403_0711_gb300 import inputs
    dims = [(13 + k % 3, 12, 15 - k % 4) for k in range(systems)]
    charges = [inputs.uniform_q(d, n, seed=k % 7) for k, d in enumerate(dims)]
    b = cl.Batch(dims, precision=getattr(cl, prec), seed=4, stream=torch.cuda.Stream())
    b.set_charges(charges)
    b.sweep(4, 1, 2)
    g = cl.BatchGlobalCV(b, n_iter=60, R=R)
    tg = torch.zeros(systems, dtype=torch.float64, device="cuda")
    g.eval(tg.data_ptr())
    b.sync()
    for k in {0, systems // 2, systems - 1}:
        _check(b.field(k), g.h(k), np.asarray(charges[k][0]), charges[k][1], R, prec == "F32",
               float(tg[k]))
    g.close()
    b.close()
