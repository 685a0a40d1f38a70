"""What the speed of this framework is measured on: Monte Carlo chains of one
instance, replica batches, the serving loop, the Supplement S-I estimators and
checkpoints, each through the package's public calls.

A case is a dict of plain values; `prepare` gives what a program has in hand
before the call, `run` is one pass of it, `work` what that pass cannot do
without and `exact` its result in plain numpy where it has one that does not
depend on this package.

Every kind starts from a configuration a chain really visits: the chains, the
batch and the serving jobs are swept for a while first; the estimators read a
generated worldline configuration (so that their result can be formed without
the package) with the vertex, kink and worm densities of those chains.
"""
import math

import numpy as np

import paper_1307_0328_gb300 as P
from paper_1307_0328_gb300 import autotune, serve

ROW_FIELDS = [f for f in P.ROW_DTYPE.names]


def _chain(name, **kw):
    c = dict(kind="chain", Lx=8, Ly=8, beta=2.0, V=0.0, mu=0.0, eta=0.1, dom_x=0, dom_y=0, sub_block=0,
             exchange_every=2, legs_hint=0, dom_tau=1, vertex_window=0.0, settle=60, sweeps=16)
    c.update(kw, name=name)
    return c


def listed():
    return [
        # the 8x8 lattice at beta t = 2 that is checked against exact
        # diagonalisation: one domain, a few worms; launches and latency count
        _chain("chain_8x8_bt2", eta=0.2, sweeps=16),
        # a ragged lattice in ragged domains with an interaction and a field:
        # the 24-site edge of the replica grids with uneven domains
        _chain("chain_24x36_bt3", Lx=24, Ly=36, beta=3.0, V=1.0, mu=0.6, eta=0.2, dom_x=8, dom_y=12, sub_block=2,
               sweeps=16),
        # the benchmark's lattice (256x256, beta t = 4) with its leg hint:
        # one bin of a chain and the checkpoint that ends it
        _chain("chain_256_bt4", Lx=256, Ly=256, beta=4.0, dom_x=16, dom_y=16, sub_block=2, legs_hint=18, sweeps=64),
        # the low-temperature scaling-study shape (16x16-site domains at
        # beta t = 16) on 1/16 of its sites: the largest chain here
        _chain("chain_512_bt16", Lx=512, Ly=512, beta=16.0, dom_x=16, dom_y=16, sub_block=2, settle=90, sweeps=32),
        # the paper's superfluid point V/t = 3, mu/t = 1.2, beta t = 16 on
        # 128x128: many diagonal vertices, small domains, much boundary
        _chain("chain_128_v3_bt16", Lx=128, Ly=128, beta=16.0, V=3.0, mu=1.2, eta=0.05, dom_x=4, dom_y=4,
               sub_block=2, sweeps=16),
        # temporal domains (Step 1), as a long circle is run in slabs
        _chain("chain_128_bt8_slabs", Lx=128, Ly=128, beta=8.0, dom_x=16, dom_y=16, sub_block=2, dom_tau=4,
               sweeps=16),
        # on-the-fly vertex generation near the worms
        _chain("chain_96_bt4_window", Lx=96, Ly=96, beta=4.0, mu=0.5, eta=0.25, dom_x=16, dom_y=16, sub_block=2,
               vertex_window=0.02, sweeps=16),
        # the replica grid of uneven sizes from one captured graph; the rows of
        # every replica are what such a run keeps (the configurations stay on
        # the device)
        dict(name="batch_256_replicas", kind="batch", n=256, set=3, settle=24, graph=4, sweeps=8),
        # the serving loop with its jobs resident: one chunk of every job and
        # the rows handed back
        dict(name="serve_12_jobs", kind="serve", n=12, set=5, L_max=256, settle=24, chunk=8),
        # equal-time Green function, plaquette and listed 4-point functions
        # of the benchmark's lattice
        dict(name="equal_time_256", kind="equal_time", Lx=256, Ly=256, beta=4.0, eta=0.1, K=16, rmax=64, n=4,
             m=4096),
        # densities of b and b+, unequal-time Green function and listed
        # 3-point functions with two points on one site
        dict(name="unequal_time_128", kind="unequal_time", Lx=128, Ly=128, beta=4.0, eta=0.1, K=32, rmax=8, m=4096),
        # a checkpoint written and taken up again
        dict(name="checkpoint_256_bt4", kind="checkpoint", Lx=256, Ly=256, beta=4.0, eta=0.1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _edge(rng, beta, D, eta):
    """A domain edge whose legs, Step-3 candidates and worms fit a domain's
    shared memory by the a-priori counts."""
    best = 4
    for e in range(4, 17):
        s = e * e
        legs = 1.1 * 4.0 * beta * (D + 1.0) * s + 256.0
        cand = 2.0 * s * beta * D
        pool = 8.0 * (cand + 16.0 * math.sqrt(cand) + 128.0)
        mw = beta * eta * s
        worms = 48.0 * (mw + 16.0 * math.sqrt(mw) + 128.0) + 8.0 * s
        if 9.0 * legs + max(pool, worms) + 8192.0 + 48.0 * s <= 180e3:
            best = e
    return rng.randint(4, best)


def _lattice_edge(rng, lo, hi):
    """A lattice edge with a divisor of 2..16 to cut domains by."""
    while True:
        L = int(_log(rng, lo, hi + 1))
        if any(L % e == 0 for e in range(2, 17)):
            return L


def draw(rng):
    kind = rng.choice(["chain"] * 6 + ["batch", "serve", "equal_time", "unequal_time", "checkpoint"])
    if kind == "chain":
        V = float(rng.choice([0.0, 0.0, 1.0]))
        mu = round(rng.uniform(-1.0, 1.0), 3) if V else 0.0
        beta = round(_log(rng, 1.0, 16.0), 3)
        eta = rng.choice([0.05, 0.1, 0.2])
        corner = [0.0, -mu / 4.0, V - mu / 2.0]  # the bond energies
        D = max(corner) + 0.5 - min(corner)
        e = _edge(rng, beta, D, eta)
        e2 = e if rng.random() < 0.7 else max(2, e - rng.randint(0, e // 2))
        sites = _log(rng, 64.0, min(2.0 ** 18, 2.0 ** 21 / (beta * (D + 0.5))))
        k = max(1, int(math.sqrt(sites) / e + 0.5))
        k2 = max(1, int(sites / (k * e * e2) + 0.5))
        even = e % 2 == 0 and e2 % 2 == 0 and min(e, e2) >= 4
        opt = rng.random()
        return dict(kind="chain", Lx=e * k, Ly=e2 * k2, beta=beta, V=V, mu=mu, eta=eta, dom_x=e, dom_y=e2,
                    sub_block=2 if even else 0, exchange_every=rng.choice([1, 2, 2, 3]), legs_hint=0,
                    dom_tau=rng.randint(2, 5) if opt < 0.2 else 1,
                    vertex_window=round(_log(rng, 0.01, 0.2), 4) if opt > 0.85 else 0.0, settle=40,
                    sweeps=rng.randint(4, 24))
    if kind == "batch":
        return dict(kind="batch", n=int(_log(rng, 8, 200)), set=rng.randint(10, 10 ** 6), settle=16,
                    graph=rng.choice([0, 2, 4]), sweeps=4)
    if kind == "serve":
        return dict(kind="serve", n=rng.randint(2, 12), set=rng.randint(10, 10 ** 6), L_max=192, settle=16,
                    chunk=rng.randint(2, 8))
    beta = round(_log(rng, 0.5, 12.0), 3)
    eta = rng.choice([0.05, 0.1, 0.2])
    if kind == "equal_time":
        Lx, Ly = _lattice_edge(rng, 8, 256), _lattice_edge(rng, 8, 256)
        return dict(kind=kind, Lx=Lx, Ly=Ly, beta=beta, eta=eta, K=rng.randint(1, 20),
                    rmax=rng.randint(1, min(Lx, Ly) // 2), n=rng.randint(1, 6), m=int(_log(rng, 1, 4096)))
    if kind == "unequal_time":
        Lx, Ly = _lattice_edge(rng, 6, 128), _lattice_edge(rng, 6, 128)
        return dict(kind=kind, Lx=Lx, Ly=Ly, beta=beta, eta=eta, K=rng.randint(2, 16),
                    rmax=rng.randint(0, min(8, min(Lx, Ly) // 2)), m=int(_log(rng, 1, 4096)))
    return dict(kind=kind, Lx=_lattice_edge(rng, 8, 256), Ly=_lattice_edge(rng, 8, 256), beta=beta, eta=eta)


# --------------------------------------------------------------------------- chains
def _params(case, seed):
    return dict(Lx=case["Lx"], Ly=case["Ly"], beta=case["beta"], t=1.0, V=case["V"], mu=case["mu"], eta=case["eta"],
                dom_x=case["dom_x"], dom_y=case["dom_y"], sub_block=case["sub_block"],
                exchange_every=case["exchange_every"], legs_hint=case["legs_hint"], dom_tau=case["dom_tau"],
                vertex_window=case["vertex_window"], n_cycle=16, seed=seed + 1, init=1, init_seed=seed + 7)


def _prepare_chain(case, seed):
    # a static half-filled start, a pilot that sets N_cycle by the library's
    # rule, and the rest of the settling at that N_cycle
    sim = P.Sim(**_params(case, seed))
    pilot = max(8, case["settle"] // 2)
    sim.sweep(pilot)
    P.pmwa_set_n_cycle(sim.h, P.n_cycle(sim.params, sim.rows()[pilot // 2:]))
    sim.sweep(max(1, case["settle"] - pilot))
    sim.rows()
    return dict(kind="chain", sim=sim, sweeps=case["sweeps"], buf=_checkpoint_buffer(sim))


def _checkpoint_buffer(sim):
    """A caller-owned buffer that any configuration of the instance fits in
    (the format says how much of it is used)."""
    p = sim.params
    cap = P.pmwa_slot_capacity(**{f: getattr(p, f) for f in ("Lx", "Ly", "beta", "t", "V", "mu", "eta")})
    return np.zeros(1 + sim.N * (1 + cap), dtype=np.uint64)


def _checkpoint(st):
    rc = P.load().pmwa_export(st["sim"].h, st["buf"].ctypes.data, st["buf"].nbytes)
    if rc:
        raise P.PmwaError("pmwa_export", rc)
    return st["buf"].view(np.int64)


def _columns(rows):
    """A row table as one array per field (whole numbers as int64)."""
    return {f: rows[f].astype(np.float64) if f == "q_impr" else rows[f].astype(np.int64) for f in ROW_FIELDS}


def _run_chain(st):
    # a bin of sweeps, its measurement rows, and the checkpoint that ends it
    st["sim"].sweep(st["sweeps"])
    return dict(rows=_columns(st["sim"].rows()), configuration=_checkpoint(st))


# --------------------------------------------------------------------------- replicas
def _prepare_batch(case, seed):
    reps = autotune.replica_set(case["n"], seed=case["set"])
    for i, p in enumerate(reps):
        p.update(seed=seed * 1000003 + i, init_seed=seed * 1000003 + 500000 + i)
    batch = P.Batch(reps)
    batch.sweep(case["settle"])
    for i, p in enumerate(reps):
        batch.set_n_cycle(i, autotune.n_cycle_rule(p, batch.rows(i)[case["settle"] // 2:]))
    if case["graph"]:
        batch.graph(case["graph"])
    return dict(kind="batch", batch=batch, sweeps=case["sweeps"])


def _run_batch(st):
    b = st["batch"]
    b.sweep(st["sweeps"])
    return _columns(np.concatenate([b.rows(i) for i in range(b.n)]))


# --------------------------------------------------------------------------- serving
def _jobs(case, seed):
    jobs = serve.poisson_trace(n=case["n"], seed=case["set"], L_max=case["L_max"])
    for i, j in enumerate(jobs):
        j.params.update(seed=seed * 1000003 + i, init_seed=seed * 1000003 + 500000 + i)
        j.sweeps = 1 << 40  # resident throughout
    return jobs


def _prepare_serve(case, seed):
    srv = serve.Server(budget_bytes=64 << 30, max_jobs=case["n"], chunk=case["chunk"])
    for j in _jobs(case, seed):
        srv.submit(j)
    for _ in range(-(-case["settle"] // case["chunk"])):
        srv.step(0.0)
    return dict(kind="serve", server=srv)


def _run_serve(st):
    srv = st["server"]
    srv.step(0.0)
    return _columns(np.concatenate([j.rows.pop() for j in srv.resident]))


# --------------------------------------------------------------------------- generated configurations
_TWO59 = 1 << 59
_MASK62 = np.uint64((1 << 62) - 1)


def _configuration(case, seed):
    """Random worldlines in the checkpoint format: per site a Poisson number
    of vertex legs (about 4.1 beta, a third of them kinks) and worms (about
    0.95 beta eta) at uniform times, the state flipping at kinks and worms.
    Returns the buffer and the padded tables (keys, is_leg, count)."""
    rng = np.random.Generator(np.random.Philox(seed))
    Lx, Ly, beta, eta = case["Lx"], case["Ly"], case["beta"], case["eta"]
    N = Lx * Ly
    cap = P.pmwa_slot_capacity(Lx=Lx, Ly=Ly, beta=beta, eta=eta)
    legs, worms = 4.1 * beta, 0.95 * beta * eta
    n = np.minimum(rng.poisson(legs + worms, N), cap).astype(np.int64)
    W = max(1, int(n.max()))
    live = np.arange(W) < n[:, None]
    m = rng.integers(0, _TWO59, (N, W), dtype=np.uint64)
    m[~live] = np.uint64(_TWO59 - 1)
    m.sort(axis=1)
    worm = (rng.random((N, W)) < worms / (legs + worms)) & live
    flip = (worm | (rng.random((N, W)) < 1.0 / 3.0)) & live
    # an even number of flips round the circle: the first leg takes or loses
    # a kink (a site with worms only gets a diagonal leg for its first worm)
    odd = (flip.sum(axis=1) & 1).astype(bool)
    first = np.argmax(live & ~worm, axis=1)
    none = ~(live & ~worm).any(axis=1)
    r = np.nonzero(odd & ~none)[0]
    flip[r, first[r]] ^= True
    r = np.nonzero(odd & none)[0]
    worm[r, 0] = False
    flip[r, 0] = False
    base = rng.integers(0, 2, N)
    above = (base[:, None] + np.cumsum(flip, axis=1)) & 1
    below = above ^ flip
    x, y = np.arange(N) % Lx, np.arange(N) // Lx

    def cls(c, L):
        return np.where(c == L - 1, 2, c & 1)

    bonds = np.stack([cls(x, Lx), 3 + cls(y, Ly), cls((x - 1) % Lx, Lx), 3 + cls((y - 1) % Ly, Ly)], axis=1)
    tag = np.take_along_axis(bonds, rng.integers(0, 4, (N, W)), axis=1)
    tag = np.where(worm, 7, tag)
    second = np.where(worm, rng.integers(0, 2, (N, W)), below)  # a worm's direction, a leg's state below
    key = (m << np.uint64(5)) | (tag.astype(np.uint64) << np.uint64(2)) | (second.astype(np.uint64) << np.uint64(1)) \
        | above.astype(np.uint64)
    last = np.where(n > 0, above[np.arange(N), np.maximum(n, 1) - 1], base)
    out = np.zeros(1 + N + int(n.sum()), dtype=np.uint64)
    at = 1 + np.concatenate([[0], np.cumsum(n + 1)[:-1]])
    out[0] = N
    out[at] = n.astype(np.uint64) | (last.astype(np.uint64) << np.uint64(63))
    place = at[:, None] + 1 + np.arange(W)
    out[place[live]] = key[live]
    return out, key, live & ~worm, n


def _domain_edge(L):
    return max([e for e in range(2, 17) if L % e == 0])


def _prepare_import(case, seed):
    # (the estimators do not depend on the domains, but an instance has them)
    sim = P.Sim(Lx=case["Lx"], Ly=case["Ly"], beta=case["beta"], eta=case["eta"], n_cycle=1, init=0,
                dom_x=_domain_edge(case["Lx"]), dom_y=_domain_edge(case["Ly"]))
    sim.import_(_configuration(case, seed)[0])
    return sim


def _points(case, seed):
    rng = np.random.Generator(np.random.Philox(seed + 12345))
    N = case["Lx"] * case["Ly"]
    if case["kind"] == "equal_time":
        base = rng.integers(0, N, (case["m"], 1))
        step = np.cumsum(rng.integers(1, max(2, N // case["n"]), (case["m"], case["n"])), axis=1)
        return ((base + step) % N).astype(np.int32)  # distinct: the steps add up to less than N
    a = rng.integers(0, N, case["m"])
    b = (a + rng.integers(1, N, case["m"])) % N
    k = rng.integers(0, case["K"], (case["m"], 2))
    k[:, 1] = (k[:, 0] + 1 + k[:, 1] % (case["K"] - 1)) % case["K"]  # another slice of the same site
    k2 = rng.integers(0, case["K"], case["m"])
    comp = rng.integers(0, 2, (case["m"], 3))
    pts = np.zeros((case["m"], 3, 3), dtype=np.int32)
    pts[:, 0] = np.stack([a, k[:, 0], comp[:, 0]], axis=1)
    pts[:, 1] = np.stack([a, k[:, 1], comp[:, 1]], axis=1)
    pts[:, 2] = np.stack([b, k2, comp[:, 2]], axis=1)
    return pts


def prepare(case, seed):
    kind = case["kind"]
    if kind == "chain":
        return _prepare_chain(case, seed)
    if kind == "batch":
        return _prepare_batch(case, seed)
    if kind == "serve":
        return _prepare_serve(case, seed)
    st = dict(kind=kind, sim=_prepare_import(case, seed))
    if kind == "checkpoint":
        st["buf"] = _checkpoint_buffer(st["sim"])
    else:
        st.update(points=_points(case, seed), K=case["K"], rmax=case["rmax"])
    return st


def run(st):
    kind = st["kind"]
    if kind == "chain":
        return _run_chain(st)
    if kind == "batch":
        return _run_batch(st)
    if kind == "serve":
        return _run_serve(st)
    sim = st["sim"]
    if kind == "checkpoint":
        out = _checkpoint(st)
        sim.import_(st["buf"])
        return out
    if kind == "equal_time":
        gx, gy, plaq = P.pmwa_green(sim.h, st["K"], st["rmax"])
        return dict(rho=sim.rho_slices(st["K"]), gx=gx, gy=gy, plaq=plaq, npoint=sim.npoint(st["K"], st["points"]))
    rho, iv = sim.rho_alpha(st["K"])
    return dict(rho=rho, iv=iv, g=sim.green_tau(st["K"], st["rmax"]), npoint=sim.npoint_alpha(st["K"], st["points"]))


# --------------------------------------------------------------------------- work
def _events(sites, beta, V, mu, eta):
    """Mean events of a configuration by the a-priori counts: legs 4 beta
    (d + t/2) a site (d the mean diagonal weight), worms beta eta a site."""
    E = [V * (s & 1) * (s >> 1) - (mu / 4.0) * ((s & 1) + (s >> 1)) for s in range(4)]
    d = max(E) + 0.5 - sum(E) / 4.0
    return sites * (4.0 * beta * (d + 0.5) + beta * eta)


def work(case):
    kind = case["kind"]
    if kind == "chain":
        ev = _events(case["Lx"] * case["Ly"], case["beta"], case["V"], case["mu"], case["eta"])
        # every sweep reads and writes the 8-byte events once; the checkpoint
        # reads them and writes the buffer
        return {"bytes": 16.0 * ev * (case["sweeps"] + 1), "flops": 0.0}
    if kind in ("batch", "serve"):
        ps = autotune.replica_set(case["n"], seed=case["set"]) if kind == "batch" else \
            [j.params for j in _jobs(case, 0)]
        ev = sum(_events(p["Lx"] * p["Ly"], p["beta"], p["V"], p["mu"], p["eta"]) for p in ps)
        return {"bytes": 16.0 * ev * (case["sweeps"] if kind == "batch" else case["chunk"]), "flops": 0.0}
    N = float(case["Lx"] * case["Ly"])
    ev = _events(N, case["beta"], 0.0, 0.0, case["eta"])
    if kind == "checkpoint":
        return {"bytes": 32.0 * ev, "flops": 0.0}
    K, r, m = case["K"], case["rmax"], case["m"]
    if kind == "equal_time":
        # the events once, the densities once, the tuples and the results
        return {"bytes": 8.0 * ev + 8.0 * N * K + m * (4.0 * case["n"] + 8.0) + 16.0 * r,
                "flops": N * K * (4.0 * r + 30.0) + m * K * case["n"]}
    return {"bytes": 8.0 * ev + 20.0 * N * K + 44.0 * m + 16.0 * (r + 1) * K,
            "flops": N * K * K * (4.0 * r + 10.0) + N * K * 60.0 + m * K * 60.0}


# --------------------------------------------------------------------------- exact results
def _wpts(a, b):
    """Worm grid points strictly between time points a and b going up (b = a:
    the whole circle)."""
    hi = np.where(b > a, b, b + np.uint64(1 << 62))
    return (hi >> np.uint64(3)) - ((a + np.uint64(1)) >> np.uint64(3))


class _Slices:
    """The interval between vertex legs around each of K slices of each site."""

    def __init__(self, case, seed):
        _, key, leg, _ = _configuration(case, seed)
        self.K, self.N, self.eta = case["K"], key.shape[0], case["eta"]
        self.xw = case["beta"] * case["eta"] / 2.0 ** 59
        nl = leg.sum(axis=1)
        WL = max(1, int(nl.max()))
        order = np.argsort(~leg, axis=1, kind="stable")[:, :WL]  # the legs first, in time order
        pk = np.take_along_axis(key >> np.uint64(2), order, axis=1)
        up = np.take_along_axis((key & np.uint64(1)).astype(np.int64), order, axis=1)
        dn = np.take_along_axis(((key >> np.uint64(1)) & np.uint64(1)).astype(np.int64), order, axis=1)
        has = np.arange(WL) < nl[:, None]
        pt = np.array([k * ((1 << 62) // self.K) + (k * ((1 << 62) % self.K)) // self.K for k in range(self.K)],
                      dtype=np.uint64)
        rows = np.arange(self.N)
        self.pt = np.broadcast_to(pt, (self.N, self.K))
        self.free = nl == 0
        self.iv = np.empty((self.N, self.K), dtype=np.int32)
        self.p, self.q = np.zeros((self.N, self.K), np.int64), np.zeros((self.N, self.K), np.int64)
        self.M, self.M1 = np.empty((self.N, self.K), np.uint64), np.zeros((self.N, self.K), np.uint64)
        self.off = np.zeros((self.N, self.K), np.uint64)
        for k in range(self.K):
            lo = (has & (pk <= pt[k])).sum(axis=1) - 1
            lo = np.where(lo < 0, np.maximum(nl, 1) - 1, lo)
            hi = np.where(lo + 1 >= nl, 0, lo + 1)
            plo, phi = pk[rows, lo], pk[rows, hi]
            self.iv[:, k] = np.where(self.free, -1, order[rows, lo])
            self.p[:, k] = np.where(self.free, 0, up[rows, lo])
            self.q[:, k] = np.where(self.free, 0, dn[rows, hi])
            self.M[:, k] = np.where(self.free, np.uint64(_TWO59), _wpts(plo, phi))
            here = np.full(self.N, pt[k], dtype=np.uint64)
            self.M1[:, k] = np.where(self.free | (here == plo), np.uint64(0), _wpts(plo, here))
            self.off[:, k] = np.where(self.free, np.uint64(0), (here - plo) & _MASK62)

    def F(self, sigma, M):
        e = np.expm1(-2.0 * M.astype(np.float64) * self.xw)
        return np.where(np.asarray(sigma) != 0, -e, 2.0 + e)

    def total(self):
        s = self.q ^ self.p
        return self.eta * self.F(1 - s, self.M) / self.F(s, self.M)

    def one(self, a):
        """Density of the component a (0: b takes 1 to 0; 1: b+) at each slice."""
        num = self.F(self.q ^ a, self.M - self.M1) * self.F((1 - a) ^ self.p, self.M1)
        v = self.eta * num / (2.0 * self.F(self.q ^ self.p, self.M))
        x = 2.0 ** 59 * self.xw
        return np.where(self.free[:, None], 0.5 * self.eta * math.tanh(x), v)

    def two(self, s, k1, a1, k2, a2):
        """Joint density of a1 at slice k1 and a2 at slice k2 (k1 != k2) of the sites s."""
        one = [self.one_cache(a) for a in (0, 1)]
        v1 = np.where(a1 == 1, one[1][s, k1], one[0][s, k1])
        v2 = np.where(a2 == 1, one[1][s, k2], one[0][s, k2])
        apart = v1 * v2
        eta2 = self.eta ** 2
        swap = self.off[s, k2] < self.off[s, k1]
        kL, kU = np.where(swap, k2, k1), np.where(swap, k1, k2)
        aL, aU = np.where(swap, a2, a1), np.where(swap, a1, a2)
        Ia = self.M1[s, kL]
        Ib = np.where(self.M1[s, kU] >= self.M1[s, kL], self.M1[s, kU] - self.M1[s, kL], np.uint64(0))
        Ic = self.M[s, kL] - np.minimum(self.M1[s, kU], self.M[s, kL])
        q, p = self.q[s, kL], self.p[s, kL]
        num = self.F(q ^ aU, Ic) * self.F((1 - aU) ^ aL, Ib) * self.F((1 - aL) ^ p, Ia)
        same = eta2 * num / (4.0 * self.F(q ^ p, self.M[s, kL]))
        Jb = _wpts(self.pt[s, k1], self.pt[s, k2])
        Jc = np.uint64(_TWO59) - Jb
        ring = eta2 * self.F((1 - a2) ^ a1, Jb) * self.F((1 - a1) ^ a2, Jc) / (4.0 * (1.0 + math.exp(
            -2.0 * 2.0 ** 59 * self.xw)))
        return np.where(self.iv[s, k1] != self.iv[s, k2], apart, np.where(self.free[s], ring, same))

    def one_cache(self, a):
        if not hasattr(self, "_one"):
            self._one = [self.one(0), self.one(1)]
        return self._one[a]


def exact(case, seed):
    if case["kind"] == "equal_time":
        z = _Slices(case, seed)
        rho = z.total()
        Lx, Ly, eta, K = case["Lx"], case["Ly"], case["eta"], case["K"]
        g = rho.reshape(Ly, Lx, K)
        gx = np.array([(g * np.roll(g, -r, axis=1)).mean() for r in range(1, case["rmax"] + 1)]) / eta ** 2
        gy = np.array([(g * np.roll(g, -r, axis=0)).mean() for r in range(1, case["rmax"] + 1)]) / eta ** 2
        gxy = np.roll(g, -1, axis=1)
        plaq = float((g * gxy * np.roll(g, -1, axis=0) * np.roll(gxy, -1, axis=0)).mean()) / eta ** 4
        t = _points(case, seed)
        return dict(rho=rho, gx=gx, gy=gy, plaq=plaq, npoint=rho[t].prod(axis=1).mean(axis=1) / eta ** case["n"])
    if case["kind"] == "unequal_time":
        z = _Slices(case, seed)
        Lx, Ly, eta, K, rmax = case["Lx"], case["Ly"], case["eta"], case["K"], case["rmax"]
        b, bd = z.one_cache(0), z.one_cache(1)
        g = np.zeros((2, rmax + 1, K))
        sites, ks = np.arange(z.N)[:, None], np.arange(K)[None, :]
        for dk in range(1, K):
            g[:, 0, dk] = z.two(sites, ks, 1, (ks + dk) % K, 0).mean()
        cube, cubed = b.reshape(Ly, Lx, K), bd.reshape(Ly, Lx, K)
        for r in range(1, rmax + 1):
            for d in range(2):
                far = np.roll(cube, -r, axis=1 - d)
                for dk in range(K):
                    g[d, r, dk] = (np.roll(far, -dk, axis=2) * cubed).mean()
        t = _points(case, seed)
        acc = np.zeros(case["m"])
        for sh in range(K):
            k = (t[:, :, 1] + sh) % K
            pair = z.two(t[:, 0, 0], k[:, 0], t[:, 0, 2], k[:, 1], t[:, 1, 2])
            third = np.where(t[:, 2, 2] == 1, bd[t[:, 2, 0], k[:, 2]], b[t[:, 2, 0], k[:, 2]])
            acc += pair * third
        return dict(rho=np.stack([b, bd], axis=2), iv=None, g=g / eta ** 2, npoint=acc / K / eta ** 3)
    return None
