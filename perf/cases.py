"""Performance cases: what a user of the sampler runs, through the public Python binding.

kind        one pass
chains      n_meas measured compound sweeps of a Lattice (Charges.run), then the samples and the estimate
            (and, of a single small box, its field)
off         the same with off-lattice particles (trilinear weights, forces, near pairs left out)
batch       n_meas measured compound sweeps of many uneven systems (Batch.run), samples and estimates
gcv_run     n_meas measured compound sweeps with the global control variate recorded (GlobalCV.run)
gcv_setup   building the global control variate of a new charge set (GlobalCV: the SOR solve), h read back
batch_gcv   n_meas measured compound sweeps of a Batch with every system's control variate recorded
cv_eval     the learned local control variate of the current fields (LocalSteinCV.evaluate, as its graph)
cv_train    one training pass of the learned control variate: T g, the loss and every gradient

prepare() thermalises each lattice by `therm` compound sweeps from the zero field.  The sampler's draws
are keyed by (seed, chain, pass, site), so exact() replays the same chain in 64 bits with plain torch.
"""
import math
import random

import numpy as np
import torch

from paper_1403_0711_gb300 import coulps, inputs, stein

THERM = 2
_ready = False


def listed():
    return [
        # a single small box in double precision, heatbath only: the smallest run there is, all latency
        dict(name="plain16_f64", kind="chains", Lx=16, Ly=16, Lz=16, chains=1, f64=True, n=8, charges="pm",
             n_hb=1, n_or=0, n_meas=200, streams=1, field=True),
        # one chain of the paper's Fig. 2 geometry (a q = 1 cube in a 128^3 box): an ordinary small run
        dict(name="cube128_1chain", kind="chains", Lx=128, Ly=128, Lz=128, chains=1, f64=False, n=8,
             charges="cube", n_hb=1, n_or=3, n_meas=40, streams=1),
        # a few chains of an uneven box with odd edges and an even number of over-relaxation passes
        dict(name="ragged_12chains", kind="chains", Lx=61, Ly=47, Lz=53, chains=12, f64=False, n=501,
             charges="uniform", n_hb=1, n_or=2, n_meas=40, streams=1),
        # the headline workload: 64 chains of 128^3, 4096 charges of +-1, two streams as the benchmark runs it
        dict(name="main128_64chains", kind="chains", Lx=128, Ly=128, Lz=128, chains=64, f64=False, n=4096,
             charges="pm", n_hb=1, n_or=3, n_meas=8, streams=2),
        # the largest single system: one 512^3 chain with a million charges in blobs
        dict(name="large512_1chain", kind="chains", Lx=512, Ly=512, Lz=512, chains=1, f64=False, n=1000000,
             charges="blobs", n_hb=1, n_or=3, n_meas=6, streams=1),
        # particles off the lattice, with forces and the near-field correction
        dict(name="offlattice96_16chains", kind="off", Lx=96, Ly=96, Lz=96, chains=16, f64=False, n=512,
             rc=1.5, n_hb=1, n_or=3, n_meas=10),
        # 256 independent systems of uneven size in one batch
        dict(name="batch256", kind="batch", systems=256, edges="32,48,64,80,96", n_min=64, n_max=2048,
             dims_seed=11, f64=False, n_hb=1, n_or=3, n_meas=8),
        # production sampling of the headline system with its global control variate
        dict(name="gcv128_64chains", kind="gcv_run", Lx=128, Ly=128, Lz=128, chains=64, f64=False, n=4096,
             charges="pm", R=1, n_hb=1, n_or=3, n_meas=8, n_iter=400),
        # a new charge set's control variate: paid once per charge set
        dict(name="gcv_setup128", kind="gcv_setup", Lx=128, Ly=128, Lz=128, chains=2, f64=False, n=4096,
             charges="pm", R=1, n_iter=818),
        # control variates of many systems
        dict(name="batch_gcv64", kind="batch_gcv", systems=64, edges="32,48,64,80", n_min=64, n_max=2048,
             dims_seed=5, f64=False, R=1, n_hb=1, n_or=3, n_meas=8, n_iter=300),
        # the learned control variate evaluated on 64 chains' current fields (after every measured sweep)
        dict(name="cv_eval_64chains", kind="cv_eval", Lx=128, Ly=128, Lz=128, chains=64, halo=3, side=2),
        # one step of the learned control variate's training at the benchmark's batch size
        dict(name="cv_train_256", kind="cv_train", Lx=64, Ly=64, Lz=64, chains=64, halo=3, side=2, batch=256),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _edges(rng, lo, hi, most_sites):
    while True:
        L = [_loguniform(rng, lo, hi) for _ in range(3)]
        if L[0] * L[1] * L[2] <= most_sites:
            return L


def draw(rng):
    kind = rng.choices(["chains", "off", "batch", "gcv_run", "gcv_setup", "batch_gcv", "cv_eval", "cv_train"],
                       weights=[8, 2, 2, 2, 2, 1, 2, 2])[0]
    if kind in ("chains", "off", "gcv_run", "gcv_setup"):
        f64 = rng.random() < 0.25
        most = 3000000 if f64 else 60000000
        L = _edges(rng, 8, 200, most)
        sites = L[0] * L[1] * L[2]
        chains = _loguniform(rng, 1, min(64, max(1, most // sites)))
        n_hb, n_or = rng.choice([(1, 0), (1, 1), (1, 2), (1, 3), (1, 3), (1, 4), (2, 5)])
        n = _loguniform(rng, 2, max(2, min(4096, sites // 4)))
        c = dict(kind=kind, Lx=L[0], Ly=L[1], Lz=L[2], chains=chains, f64=f64, n=n, n_hb=n_hb, n_or=n_or)
        c["n_meas"] = max(4, min(100, int(4e8 / (sites * chains * (n_hb + n_or)))))
        if kind == "chains":
            # a single small box is also looked at as a whole
            c.update(charges=rng.choice(["pm", "uniform"]), streams=rng.choice([1, 2]),
                     field=chains == 1 and sites <= 40000)
            c["n"] += c["n"] % 2
        elif kind == "off":
            c.update(rc=rng.uniform(1.0, 2.5))
        else:
            c.update(charges="uniform", R=rng.choice([0, 1, 1, 2]))
            c["n_iter"] = rng.randint(2, 3) * max(L) + rng.randint(0, 20)
            if kind == "gcv_setup":
                c["chains"] = 1
                c = {k: v for k, v in c.items() if k not in ("n_hb", "n_or", "n_meas")}
        return c
    if kind in ("batch", "batch_gcv"):
        lo = rng.randint(12, 40)
        edges = sorted({lo + rng.randint(0, 56) for _ in range(4)})
        c = dict(kind=kind, systems=_loguniform(rng, 8, 200 if kind == "batch" else 64),
                 edges=",".join(map(str, edges)), n_min=8, n_max=1024, dims_seed=rng.randint(1, 10**6),
                 f64=False, n_hb=1, n_or=rng.randint(1, 4), n_meas=rng.randint(4, 8))
        if kind == "batch_gcv":
            c.update(R=rng.choice([0, 1, 2]), n_iter=2 * max(edges))
        return c
    E = rng.randint(24, 80)
    c = dict(kind=kind, Lx=E, Ly=E + rng.randint(-3, 3), Lz=E + rng.randint(-3, 3), chains=_loguniform(rng, 4, 64),
             halo=rng.randint(1, 3), side=rng.randint(1, 3))
    if kind == "cv_train":
        c["batch"] = c["chains"] * rng.randint(1, 3)
    return c


# ------------------------------------------------------------------- inputs
def _box(case):
    return (case["Lx"], case["Ly"], case["Lz"])


def _blobs(L, n, seed, n_blob=200, sigma=6.0, qmax=0.8):
    """n distinct sites in Gaussian blobs, q uniform with zero net charge."""
    rng = np.random.default_rng(seed)
    centre = rng.integers(0, L, size=(n_blob, 3))
    lin = np.empty(0, dtype=np.int64)
    while len(lin) < n:
        p = centre[rng.integers(0, n_blob, 2 * n)] + np.rint(rng.normal(0.0, sigma, (2 * n, 3))).astype(np.int64)
        p = p[((p >= 0) & (p < np.asarray(L))).all(axis=1)]
        lin = np.unique(np.concatenate([lin, p[:, 0] + L[0] * (p[:, 1] + L[1] * p[:, 2])]))
    lin = rng.permutation(lin)[:n]
    q = rng.uniform(-qmax, qmax, n)
    return (np.stack([lin % L[0], (lin // L[0]) % L[1], lin // (L[0] * L[1])], axis=1).astype(np.int32),
            q - q.mean())


def _charges(case, seed):
    L = _box(case)
    if case["charges"] == "cube":
        return inputs.cube(L, round(case["n"] ** (1 / 3)))
    if case["charges"] == "pm":
        return inputs.plus_minus(L, case["n"], seed + 1)
    if case["charges"] == "blobs":
        return _blobs(L, case["n"], seed + 1)
    return inputs.uniform_q(L, case["n"], seed + 1)


def _systems(case, seed):
    rng = random.Random(case["dims_seed"])
    edges = [int(v) for v in case["edges"].split(",")]
    out = []
    for i in range(case["systems"]):
        e = rng.choice(edges)
        n = _loguniform(rng, case["n_min"], min(case["n_max"], e ** 3 // 2))
        out.append(((e, e, e), *inputs.uniform_q((e, e, e), n, seed * 1009 + i)))
    return out


def _net(case, seed):
    """A small net's weights (W1 b1 W2 b2 W3 b3), of the size trained ones have."""
    g = torch.Generator().manual_seed(seed + 17)
    sizes = [((16, 3, 3, 3, 3), 0.3), ((16,), 0.1), ((16, 16, 3, 3, 3), 0.075), ((16,), 0.1),
             ((1, 16, 3, 3, 3), 0.075), ((1,), 0.1)]
    return [torch.randn(s, generator=g) * c for s, c in sizes]


def _cluster(case):
    """The charges of the learned control variate's cases (a q = 1 cube) and its box R."""
    sites, q = inputs.cube(_box(case), case["side"])
    return sites, q, sites.min(axis=0) - case["halo"], sites.max(axis=0) + 1 + case["halo"]


def _lattice(case, seed):
    global _ready
    if not _ready:
        coulps.use_torch_allocator()
        _ready = True
    return coulps.Lattice(_box(case), n_chains=case["chains"],
                          precision=coulps.F64 if case.get("f64") else coulps.F32, seed=seed, stream=torch.cuda.Stream())


def _mix(case):
    return case.get("n_hb", 1), case.get("n_or", 3)


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind in ("batch", "batch_gcv"):
        global _ready
        if not _ready:
            coulps.use_torch_allocator()
            _ready = True
        sys = _systems(case, seed)
        b = coulps.Batch([d for d, _, _ in sys], precision=coulps.F64 if case["f64"] else coulps.F32, seed=seed,
                         stream=torch.cuda.Stream())
        b.set_charges([(x, q) for _, x, q in sys], log_capacity=case["n_meas"])
        b.sweep(THERM, *_mix(case))
        if kind == "batch_gcv":
            s["cv"] = coulps.BatchGlobalCV(b, n_iter=case["n_iter"], R=case["R"])
            s["tg"] = torch.zeros(len(sys), dtype=torch.float64, device="cuda")
        b.sync()
        s["batch"] = b
        return s
    lat = _lattice(case, seed)
    s["lat"] = lat
    if kind in ("cv_eval", "cv_train"):
        sites, q, lo, hi = _cluster(case)
        rho = stein.charge_density(_box(case), sites, q)
        cv = stein.LocalSteinCV(_box(case), lo, hi)
        with torch.no_grad():
            for p, w in zip((cv.W1, cv.b1, cv.W2, cv.b2, cv.W3, cv.b3), _net(case, seed)):
                p.copy_(w.to(p.device))
        ch = coulps.Charges(lat, sites, q)
        torch.cuda.synchronize()
        lat.sweep(THERM, *_mix(case))
        s.update(cv=cv, rho=rho, ch=ch)
        if kind == "cv_eval":
            lat.sync()
            s["graph"], s["tg"] = cv.record_graph(lat, ch, rho)
        else:
            phis, Aphis, es = stein.collect_region(cv, lat, ch, rho, n_rounds=-(-case["batch"] // case["chains"]))
            s.update(phis=phis[:case["batch"]].contiguous(), Aphis=Aphis[:case["batch"]].contiguous(),
                     es=es[:case["batch"]].cuda())
            cv.set_density(rho)
            torch.cuda.synchronize()
        return s
    if kind == "off":
        pos, q = inputs.off_lattice(_box(case), case["n"], seed + 1)
        ch = coulps.Charges.off_lattice(lat, pos, q, log_capacity=case["n_meas"], forces=True)
        ch.near(case["rc"])
    else:
        ch = coulps.Charges(lat, *_charges(case, seed), log_capacity=case.get("n_meas", 0))
    s["ch"] = ch
    if kind == "gcv_setup":
        lat.sync()
        return s
    lat.set_streams(case.get("streams", 1))
    lat.sweep(THERM, *_mix(case))
    if kind == "gcv_run":
        s["cv"] = coulps.GlobalCV(ch, n_iter=case["n_iter"], R=case["R"])
        s["tg"] = torch.zeros(case["chains"], dtype=torch.float64, device="cuda")
    lat.sync()
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind in ("batch", "batch_gcv"):
        b = s["batch"]
        b.reset_stats()
        if kind == "batch":
            b.run(0, case["n_meas"], *_mix(case))
            return dict(samples=b.samples(), estimate=b.estimate())
        s["cv"].reset()
        s["cv"].run(case["n_meas"], *_mix(case))
        s["cv"].eval(s["tg"].data_ptr())
        return dict(samples=b.samples(), tg=s["tg"], cv=s["cv"].estimate())
    if kind == "cv_eval":
        with torch.cuda.stream(s["lat"]._stream):
            s["graph"].replay()
        return s["tg"]
    if kind == "cv_train":
        cv = s["cv"]
        par = [cv.W1, cv.b1, cv.W2, cv.b2, cv.W3, cv.b3]
        tg = cv.stein_term(stein.inputs_from(s["phis"], cv.rho_region(s["rho"])), s["Aphis"])
        r = s["es"].float() - tg
        loss = ((r - r.mean()) ** 2).mean() / (s["es"].float().var() + 1e-30)
        for p in par:
            p.grad = None
        loss.backward()
        return dict(tg=tg.detach(), loss=loss.detach(), grads=[p.grad for p in par])
    if kind == "gcv_setup":
        cv = coulps.GlobalCV(s["ch"], n_iter=case["n_iter"], R=case["R"])
        h, hr = cv.h(), cv.info()["h_dot_rho"]
        cv.close()
        return dict(h=h, h_dot_rho=hr)
    ch = s["ch"]
    ch.reset_stats()
    if kind == "gcv_run":
        ch.cv_reset()
        s["cv"].run(case["n_meas"], *_mix(case))
        s["cv"].eval(s["tg"].data_ptr())
        return dict(samples=ch.samples(), tg=s["tg"], cv=ch.cv_estimate())
    ch.run(0, case["n_meas"], *_mix(case))
    out = dict(samples=ch.samples(), estimate=ch.estimate())
    if case.get("field"):
        out["field"] = s["lat"].field(0)
    if kind == "off":
        out["force"], out["force_stderr"] = ch.forces()
    return out


# --------------------------------------------------------------------- work
def work(case):
    kind = case["kind"]
    if kind in ("batch", "batch_gcv"):
        sys = [d for d, _, _ in _systems(case, 0)]
        sites = sum(a * b * c for a, b, c in sys)
        es, n = 4, sites
    elif kind in ("cv_eval", "cv_train"):
        _, q, lo, hi = _cluster(case)
        L = _box(case)
        nb = case.get("batch", case["chains"])
        E = math.prod(min(int(h) + 3, n) - max(int(a) - 3, 0) for a, h, n in zip(lo, hi, L)) * nb
        R1 = math.prod(int(h - a) + 2 for a, h in zip(lo, hi)) * nb
        # two 16 -> 16 convolutions (the first with 3 input channels), the 16 x 16 x 27 divergence
        # contraction next to R; a training pass does each twice more for its gradients
        f = 2 * 27 * 16 * (3 * E + 16 * E + 16 * R1 + R1)
        # phi and A phi in, T g out
        return {"bytes": E * (4 if kind == "cv_eval" else 6), "flops": f * (3 if kind == "cv_train" else 1)}
    else:
        n = case["Lx"] * case["Ly"] * case["Lz"]
        es = 8 if case["f64"] else 4
        sites = n * case["chains"]
    if kind == "gcv_setup":
        # density in (its charges), h out; 9 operations per site and iteration
        return {"bytes": 4 * n + 12 * case["n"], "flops": 9 * n * case["n_iter"]}
    n_hb, n_or = _mix(case)
    # a compound sweep reads and writes every site once; 7 operations per update and about 40 per draw
    b, f = 2 * es * sites, sites * (7 * (n_hb + n_or) + 40 * n_hb)
    if kind in ("gcv_run", "batch_gcv"):
        b, f = b + es * sites, f + 2 * sites  # v . phi of every sample
    return {"bytes": b * case["n_meas"], "flops": f * case["n_meas"]}


# -------------------------------------------------------- the same in 64 bits
_M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wraps as the unsigned product does
        c0, c1, c2, c3 = (((p1 >> 32) & _M32) ^ c1 ^ k0, p1 & _M32, ((p0 >> 32) & _M32) ^ c3 ^ k1, p0 & _M32)
        k0, k1 = (k0 + 0x9E3779B9) & _M32, (k1 + 0xBB67AE85) & _M32
    return c0, c1, c2, c3


class _Replay:
    """The sampler's chains in FP64: phi (n, Z, Y, X) from 0, red/black heatbath and over-relaxation."""

    def __init__(self, L, ids, seed):
        X, Y, Z = L
        self.L, self.key, self.passes = L, (seed & _M32, (seed >> 32) & _M32), 0
        self.ids = torch.tensor(ids, dtype=torch.int64, device="cuda")
        self.phi = torch.zeros((len(ids), Z, Y, X), dtype=torch.float64, device="cuda")
        ar = [torch.arange(v, device="cuda") for v in (Z, Y, X)]
        self.colour = (ar[0][:, None, None] + ar[1][None, :, None] + ar[2][None, None, :]) & 1
        self.wq = (X + 7) // 8

    def S(self):
        p = self.phi
        s = torch.zeros_like(p)
        s[:, 1:] += p[:, :-1]
        s[:, :-1] += p[:, 1:]
        s[:, :, 1:] += p[:, :, :-1]
        s[:, :, :-1] += p[:, :, 1:]
        s[..., 1:] += p[..., :-1]
        s[..., :-1] += p[..., 1:]
        return s

    def noise(self, c):
        X, Y, Z = self.L
        out = torch.empty_like(self.phi)
        for z0 in range(0, Z, 64):  # in slabs, to bound the memory of the words
            z1 = min(z0 + 64, Z)
            qid = torch.arange(z0 * Y * self.wq, z1 * Y * self.wq, device="cuda")[None, :]
            full = lambda v: torch.full_like(qid, v)  # noqa: E731
            w = torch.stack(_philox(qid, full(self.passes), self.ids[:, None], full(c), *self.key), dim=-1)
            r = (w.double() + 0.5) * 2.0 ** -32
            w = torch.special.ndtri(r) / math.sqrt(6.0)  # = -erfc^-1(2 r) / sqrt(3)
            w = w.reshape(len(self.ids), z1 - z0, Y, 4 * self.wq).repeat_interleave(2, dim=3)
            out[:, z0:z1] = w[..., :X]
        return out

    def sweep(self, n, n_hb, n_or):
        for _ in range(n):
            for k in range(n_hb + n_or):
                for c in (0, 1):
                    new = self.S() / 6 + self.noise(c) if k < n_hb else self.S() / 3 - self.phi
                    self.phi = torch.where(self.colour == c, new, self.phi)
                self.passes += 1


def _sample(phi, sites, q):
    at = torch.as_tensor(np.asarray(sites, dtype=np.int64), device="cuda")
    t = phi[:, at[:, 2], at[:, 1], at[:, 0]] * torch.as_tensor(q, device="cuda")
    Q, P = t.sum(1), (t * t).sum(1)
    return torch.stack([Q, P, Q * Q - P], dim=1)


def _dst_solve(rho):
    """u with A u = -rho (A: 6 on the diagonal, -1 per neighbour, 0 outside)."""
    u, lam = -rho, 0.0
    S = []
    for d, n in enumerate(rho.shape):
        k = torch.arange(1, n + 1, dtype=torch.float64, device="cuda")
        S.append(torch.sin(math.pi / (n + 1) * k[:, None] * k[None, :]) * math.sqrt(2.0 / (n + 1)))
        lam = lam + (2 - 2 * torch.cos(math.pi * k / (n + 1))).reshape([-1 if i == d else 1 for i in range(3)])
    rot = lambda v: torch.einsum("zyx,za,yb,xc->abc", v, *S)  # noqa: E731
    return rot(rot(u) / lam)


def _apply_A(p):
    out = 6.0 * p
    for d in (-3, -2, -1):
        n = p.shape[d]
        out.narrow(d, 1, n - 1).sub_(p.narrow(d, 0, n - 1))
        out.narrow(d, 0, n - 1).sub_(p.narrow(d, 1, n - 1))
    return out


def _density(L, sites, q):
    rho = torch.zeros((L[2], L[1], L[0]), dtype=torch.float64, device="cuda")
    at = torch.as_tensor(np.asarray(sites, dtype=np.int64), device="cuda")
    rho[at[:, 2], at[:, 1], at[:, 0]] = torch.as_tensor(q, device="cuda")
    return rho


def _global_tg(phi, L, sites, q, R):
    """h.rho - Q (A h).phi for A h = -rho, plus the local term of P with the (2R+1)^3 cube's Green function."""
    rho = _density(L, sites, q)
    h = _dst_solve(rho)
    Q = (phi * rho).sum(dim=(1, 2, 3))
    tg = (h * rho).sum() - Q * (phi * _apply_A(h)).sum(dim=(1, 2, 3))
    if R > 0:
        m = 2 * R + 1
        e = torch.zeros((m, m, m), dtype=torch.float64, device="cuda")
        e[R, R, R] = -1.0
        k = _dst_solve(e).float().double()
        Ap = torch.nn.functional.pad(_apply_A(phi), (R,) * 6)
        at = torch.as_tensor(np.asarray(sites, dtype=np.int64), device="cuda")
        qq = torch.as_tensor(q, device="cuda") ** 2
        w = 0.0
        for dz in range(m):
            for dy in range(m):
                for dx in range(m):
                    w = w + k[dz, dy, dx] * Ap[:, at[:, 2] + dz, at[:, 1] + dy, at[:, 0] + dx]
        tg = tg + k[R, R, R] * qq.sum() - (qq * phi[:, at[:, 2], at[:, 1], at[:, 0]] * w).sum(1)
    return tg


def _groups(case):
    """Chains a few at a time, so that a replay's memory stays bounded."""
    step = max(1, 40000000 // (case["Lx"] * case["Ly"] * case["Lz"]))
    return [list(range(k, min(k + step, case["chains"]))) for k in range(0, case["chains"], step)]


def _shift(a, d):
    """a (n, Z, Y, X, C) at x + d, 0 outside."""
    for axis, v in enumerate(d):
        if v:
            n = a.shape[axis + 1]
            pad = [0, 0] * (3 - axis) + ([0, v] if v > 0 else [-v, 0])
            a = torch.nn.functional.pad(a, pad).narrow(axis + 1, max(v, 0), n)
    return a


_OFFS = [(z, y, x) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1)]


def _conv(a, W, b):
    return b + sum(_shift(a, d) @ W[:, :, d[0] + 1, d[1] + 1, d[2] + 1].T for d in _OFFS)


def _local_tg(phi16, Aphi, rho, mask, weights):
    """sum_{x in R} (dg_x/dphi_x - g_x (A phi)_x) of the net on (phi, rho, rho phi), by the chain rule;
    phi16, Aphi (n, Z, Y, X), rho and the mask of R (Z, Y, X) on E."""
    W1, b1, W2, b2, W3, b3 = weights
    x0 = torch.stack([phi16, rho.expand_as(phi16), (rho * phi16).bfloat16().double()], dim=-1)
    a1 = torch.tanh(_conv(x0, W1, b1))
    a2 = torch.tanh(_conv(a1, W2, b2))
    g = _conv(a2, W3, b3)[..., 0]
    s1, s2 = 1 - a1 * a1, 1 - a2 * a2
    zs, ys, xs = [(int(v[0]), int(v[-1]) + 1) for v in (mask.nonzero()[:, k].unique() for k in range(3))]
    cut = lambda a: a[:, zs[0]:zs[1], ys[0]:ys[1], xs[0]:xs[1]]  # noqa: E731
    r = cut(rho[None])[..., None]
    div = 0.0
    for f in _OFFS:
        w3s2 = cut(_shift(s2, f)) * W3[0, :, f[0] + 1, f[1] + 1, f[2] + 1]
        inner = 0.0
        for e in _OFFS:
            u = [-(a + b) + 1 for a, b in zip(f, e)]
            if min(u) < 0 or max(u) > 2:
                continue
            w1 = W1[:, 0, u[0], u[1], u[2]] + r * W1[:, 2, u[0], u[1], u[2]]
            se = cut(_shift(_shift(s1, e), f)) * w1
            inner = inner + se @ W2[:, :, e[0] + 1, e[1] + 1, e[2] + 1].T
        div = div + (w3s2 * inner).sum(dim=(1, 2, 3, 4))
    return div - (g * Aphi * mask).sum(dim=(1, 2, 3))


def _exact_learned(case, seed):
    L = _box(case)
    sites, q, lo, hi = _cluster(case)
    lo, hi = [int(v) for v in lo], [int(v) for v in hi]
    e_lo, e_hi = [max(v - 3, 0) for v in lo], [min(v + 3, n) for v, n in zip(hi, L)]
    cut = lambda a: a[..., e_lo[2]:e_hi[2], e_lo[1]:e_hi[1], e_lo[0]:e_hi[0]]  # noqa: E731
    rho = _density(L, sites, q)
    mask = torch.zeros_like(rho)
    mask[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = 1
    rho, mask = cut(rho).contiguous(), cut(mask).contiguous()
    train = case["kind"] == "cv_train"
    rounds = -(-case["batch"] // case["chains"]) if train else 0
    phi, Aphi, es = [], [], []
    for ids in _groups(case):
        c = _Replay(L, ids, seed)
        c.sweep(THERM, *_mix(case))
        for k in range(max(1, rounds)):
            if train:
                c.sweep(1, *_mix(case))
            phi.append((k, cut(c.phi).bfloat16().double()))
            Aphi.append((k, cut(_apply_A(c.phi)).contiguous()))
            es.append((k, _sample(c.phi, sites, q)[:, 2]))
    phi, Aphi, es = (torch.cat([v for _, v in sorted(x, key=lambda t: t[0])]) for x in (phi, Aphi, es))
    # the net's weights are held as BF16 values; its biases are not
    w = [(v.bfloat16() if v.dim() > 1 else v).double().cuda().requires_grad_(train) for v in _net(case, seed)]
    if not train:
        return _local_tg(phi, Aphi, rho, mask, w)
    n = case["batch"]
    tg = _local_tg(phi[:n], Aphi[:n], rho, mask, w)
    r = es[:n] - tg
    loss = ((r - r.mean()) ** 2).mean() / (es[:n].var() + 1e-30)
    loss.backward()
    return dict(tg=tg.detach(), loss=loss.detach(), grads=[p.grad for p in w])


def exact(case, seed):
    kind = case["kind"]
    if kind in ("cv_eval", "cv_train"):
        return _exact_learned(case, seed)
    L = _box(case) if "Lx" in case else None
    if kind == "gcv_setup":
        rho = _density(L, *_charges(case, seed))
        h = _dst_solve(rho)
        return dict(h=h, h_dot_rho=float((h * rho).sum()))
    if kind in ("batch", "batch_gcv"):
        sys = _systems(case, seed)
        samples = torch.zeros((case["n_meas"], len(sys), 3), dtype=torch.float64, device="cuda")
        tg = torch.zeros(len(sys), dtype=torch.float64, device="cuda")
        for dims in sorted({d for d, _, _ in sys}):
            ids = [i for i, (d, _, _) in enumerate(sys) if d == dims]
            c = _Replay(dims, ids, seed)
            c.sweep(THERM, *_mix(case))
            for k in range(case["n_meas"]):
                c.sweep(1, *_mix(case))
                for j, i in enumerate(ids):
                    samples[k, i] = _sample(c.phi[j:j + 1], *sys[i][1:])[0]
            if kind == "batch_gcv":
                for j, i in enumerate(ids):
                    tg[i] = _global_tg(c.phi[j:j + 1], *sys[i], case["R"])[0]
        if kind == "batch_gcv":
            return dict(samples=samples, tg=tg, cv=None)
        return dict(samples=samples, estimate=dict(mean=samples[:, :, 2].mean(0), stderr=None, tau_int=None, n=None))
    if kind == "off":
        return _exact_off(case, seed)
    sites, q = _charges(case, seed)
    parts, tg = [], []
    for ids in _groups(case):
        c = _Replay(L, ids, seed)
        c.sweep(THERM, *_mix(case))
        got = []
        for _ in range(case["n_meas"]):
            c.sweep(1, *_mix(case))
            got.append(_sample(c.phi, sites, q))
        parts.append(torch.stack(got))
        if kind == "gcv_run":
            tg.append(_global_tg(c.phi, L, sites, q, case["R"]))
    samples = torch.cat(parts, dim=1)
    if kind == "gcv_run":
        return dict(samples=samples, tg=torch.cat(tg), cv=None)
    out = dict(samples=samples, estimate=dict(mean=float(samples[:, :, 2].mean()), stderr=None, tau_int=None, n=None))
    if case.get("field"):
        out["field"] = c.phi[0]
    return out


def _exact_off(case, seed):
    L = _box(case)
    pos, q = inputs.off_lattice(L, case["n"], seed + 1)
    p, q = torch.as_tensor(pos, device="cuda"), torch.as_tensor(q, device="cuda")
    b = torch.minimum(p.floor().long(), torch.tensor(L, device="cuda") - 2)
    f = p - b
    near = (torch.cdist(p, p, compute_mode="donot_use_mm_for_euclid_dist") < case["rc"]).double().fill_diagonal_(0)
    samples, force = [], []
    for ids in _groups(case):
        c = _Replay(L, ids, seed)
        c.sweep(THERM, *_mix(case))
        got, F = [], 0.0
        for _ in range(case["n_meas"]):
            c.sweep(1, *_mix(case))
            val, grad = 0.0, 0.0
            for cx in (0, 1):
                for cy in (0, 1):
                    for cz in (0, 1):
                        w = [f[:, i] if v else 1 - f[:, i] for i, v in enumerate((cx, cy, cz))]
                        d = [1.0 if v else -1.0 for v in (cx, cy, cz)]
                        at = c.phi[:, b[:, 2] + cz, b[:, 1] + cy, b[:, 0] + cx]
                        val = val + w[0] * w[1] * w[2] * at
                        grad = grad + at[..., None] * torch.stack([d[0] * w[1] * w[2], w[0] * d[1] * w[2],
                                                                   w[0] * w[1] * d[2]], dim=1)
            t = q * val
            u = t @ near
            Q, P = t.sum(1), (t * t).sum(1) + (t * u).sum(1)
            got.append(torch.stack([Q, P, Q * Q - P], dim=1))
            F = F - 2 * (q * (Q[:, None] - t - u))[..., None] * grad
        samples.append(torch.stack(got))
        force.append(F / case["n_meas"])
    samples = torch.cat(samples, dim=1)
    return dict(samples=samples, estimate=dict(mean=float(samples[:, :, 2].mean()), stderr=None, tau_int=None, n=None),
                force=torch.cat(force).mean(0), force_stderr=None)
