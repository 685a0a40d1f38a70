"""The estimators at the sizes where their kernels share lanes, blocks and rows
differently: one to sixty-four slices (a few lanes a site or tuple up to whole
warps), more tuples than fill the machine with a group of lanes each, and
lattices of few rows, of short rows and of rows longer than a block."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402

import paper_1307_0328_gb300 as P  # noqa: E402

# sums of up to 2^20 positive terms in another order: each addition rounds by
# 2^-53 of at most the sum, and orders by blocks add a few thousand times
REL = 1e-12


def _close(a, b):
    scale = max(float(np.abs(b).max()), 1e-300)
    assert np.allclose(a, b, rtol=REL, atol=REL * scale), float(np.abs(a - b).max())


@pytest.mark.parametrize("kw", [
    dict(Lx=7, Ly=5, beta=2.0, eta=0.3, V=0.5, mu=0.4, n_cycle=4, seed=29, cap_site=512),
    dict(Lx=2, Ly=3, beta=1.5, eta=0.5, n_cycle=4, seed=3, cap_site=512),
    dict(Lx=6, Ly=6, beta=0.25, t=0.0, c_off=0.1, eta=0.5, n_cycle=4, seed=5, cap_site=512),  # sites without legs
    dict(Lx=24, Ly=17, beta=3.0, eta=0.2, n_cycle=4, seed=7, cap_site=512),
], ids=["7x5", "2x3", "bare", "24x17"])
def test_unequal_time_at_every_group_of_lanes(kw):
    g, o = P.Sim(**kw), O.Oracle(**kw)
    o.sweep(8)
    g.import_(o.export())
    for K in (1, 2, 3, 4, 5, 8, 9, 13, 16, 17, 31, 32, 33, 47, 63, 64):
        for rmax in {0, 1, min(kw["Lx"], kw["Ly"]) // 2}:
            _close(g.green_tau(K, rmax), o.green_tau(K, rmax))


def test_unequal_time_of_several_sites_a_warp():
    """More sites than warps run at once (2432): 2 to 16 lanes a site, ragged."""
    kw = dict(Lx=52, Ly=49, dom_x=26, dom_y=7, beta=1.5, eta=0.3, V=0.5, mu=0.4, n_cycle=4, seed=31, cap_site=64)
    g, o = P.Sim(**kw), O.Oracle(**dict(kw, cap_site=0))
    o.sweep(6)
    g.import_(o.export())
    for K in (1, 2, 3, 4, 5, 8, 9, 13, 16):
        for rmax in (0, 2):
            _close(g.green_tau(K, rmax), o.green_tau(K, rmax))


def test_more_tuples_than_lanes():
    """Tuples evaluated all at once (few lanes each) and a hundred at a time
    (as many lanes as slices): the same operations in the same order."""
    kw = dict(Lx=32, Ly=32, beta=2.0, eta=0.3, n_cycle=4, seed=11, cap_site=20480)
    g, o = P.Sim(**kw), O.Oracle(**dict(kw, cap_site=0))
    o.sweep(8)
    g.import_(o.export())
    rng = np.random.default_rng(3)
    for K, n, m in ((1, 3, 170000), (3, 2, 90001), (8, 2, 50003), (16, 2, 170000), (32, 1, 21001), (32, 2, 85000)):
        # distinct slices where two points are on one site: sites of their own
        sites = np.stack([rng.integers(c * 1024 // n, (c + 1) * 1024 // n, m) for c in range(n)], axis=1)
        pts = np.ascontiguousarray(np.stack([sites, rng.integers(0, K, (m, n)), rng.integers(0, 2, (m, n))], -1)
                                   .astype(np.int32))
        got = g.npoint_alpha(K, pts)
        some = np.concatenate([np.arange(100), rng.integers(0, m, 100), np.arange(m - 100, m)])
        assert np.array_equal(g.npoint_alpha(K, np.ascontiguousarray(pts[some])), got[some])
        _close(got[some], o.npoint_alpha(K, np.ascontiguousarray(pts[some])))


@pytest.mark.parametrize("shape", [(2, 2), (4, 3), (5, 64), (64, 5), (700, 2), (2, 700), (1030, 4), (37, 41), (256, 16)],
                         ids=lambda s: "%dx%d" % s)
@pytest.mark.parametrize("K", [1, 3, 16])
def test_equal_time_on_lattices_of_any_shape(shape, K):
    Lx, Ly = shape
    g = P.Sim(Lx=Lx, Ly=Ly, dom_x=Lx if Lx < 64 else (Lx // 10 if Lx % 10 == 0 else Lx // 2 if Lx == 1030 else 16),
              dom_y=Ly if Ly < 64 else Ly // (10 if Ly % 10 == 0 else 4), beta=1.0, eta=0.3, seed=5, init=1, init_seed=2,
              n_cycle=4, cap_site=64)
    g.sweep(4)
    rho = g.rho_slices(K).reshape(Ly, Lx, K)
    for rmax in {0, 1, min(Lx, Ly) // 2}:
        gx, gy, plaq = P.pmwa_green(g.h, K, rmax)
        norm = Lx * Ly * K * 0.3 ** 2
        for r in range(1, rmax + 1):
            _close(np.array([gx[r - 1]]), np.array([(rho * np.roll(rho, -r, 1)).sum() / norm]))
            _close(np.array([gy[r - 1]]), np.array([(rho * np.roll(rho, -r, 0)).sum() / norm]))
        x, y = np.roll(rho, -1, 1), np.roll(rho, -1, 0)
        _close(np.array([plaq]), np.array([(rho * x * y * np.roll(x, -1, 0)).sum() / (norm * 0.3 ** 2)]))
