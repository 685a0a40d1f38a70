"""Step 5 (worm scattering) at the edges of its paths, bit for bit against the
oracle: one warp, one thread a worm and several worms a thread; groups that
fit their member table, overflow it, or have none; and configurations whose
kinks lie so close together that the 32-bit lengths of a move decide nothing
and the exact ones must."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402

import paper_1307_0328_gb300 as P  # noqa: E402

ROW_FIELDS = ("sweep", "n_v", "n_k", "n_w", "occ_lo", "occ_hi", "w_dom_min", "dom_empty")

CASES = [
    # 8x8: few worms (one warp), more than 32, more than the CTA's threads
    dict(Lx=8, Ly=8, beta=2.0, eta=0.2, n_cycle=7, seed=1),
    dict(Lx=8, Ly=8, beta=2.0, eta=0.5, sub_block=2, n_cycle=7, seed=2),
    dict(Lx=8, Ly=8, beta=2.0, t=0.5, eta=3.0, sub_block=2, n_cycle=5, seed=3),
    # one large group of 33 to 256 worms; 4x4 blocks whose groups overflow the table
    dict(Lx=9, Ly=7, beta=4.0, eta=0.4, n_cycle=6, seed=4),
    dict(Lx=16, Ly=16, beta=4.0, eta=0.22, sub_block=4, n_cycle=6, seed=5),
    # 1280 groups
    dict(Lx=16, Ly=16, beta=4.0, eta=0.3, sub_block=2, dom_tau=20, n_cycle=5, seed=6),
    # domains, an interaction, no partner table (beta t = 16)
    dict(Lx=32, Ly=16, beta=16.0, eta=0.12, dom_x=16, dom_y=16, sub_block=2, n_cycle=6, seed=7),
    dict(Lx=12, Ly=8, beta=6.0, V=3.0, mu=1.2, eta=0.2, dom_x=4, dom_y=4, sub_block=2, n_cycle=9, seed=8),
]


def squeezed(buf, shift=36):
    """The configuration with every event moved to within 2^(59 - shift) grid
    points of the middle of the circle, in the same order (shift 36: all
    times share the high 32 bits of their keys)."""
    out = buf.copy()
    n_sites, k = int(buf[0]), 1
    for _ in range(n_sites):
        n = int(buf[k]) & 0x7fffffff
        keys = buf[k + 1:k + 1 + n]
        m = (np.uint64(1) << np.uint64(58)) + (keys >> np.uint64(5 + shift))
        pk = (m << np.uint64(3)) | ((keys >> np.uint64(2)) & np.uint64(7))
        assert (np.diff(pk.astype(np.int64)) > 0).all()
        out[k + 1:k + 1 + n] = (pk << np.uint64(2)) | (keys & np.uint64(3))
        k += 1 + n
    return out


@pytest.mark.parametrize("shift", [0, 24, 36])
@pytest.mark.parametrize("kw", CASES, ids=["c%d" % i for i in range(len(CASES))])
def test_step5_bit_exact(kw, shift):
    g, o = P.Sim(**kw), O.Oracle(**kw)
    o.sweep(5)
    snap = o.export()
    if shift:
        snap = squeezed(snap, shift)
    for s in range(5, 9):
        for x in (g, o):
            x.import_(snap)
            x.sweep_index = s
            x.tile(5)
        assert np.array_equal(g.export(), o.export()), "Steps 3-5 at sweep %d" % s
        for x in (g, o):
            x.import_(snap)
            x.sweep_index = s
            x.sweep(1)
        snap = o.export()
        assert np.array_equal(g.export(), snap), "sweep %d" % s
    a, b = g.rows(), o.rows()
    for f in ROW_FIELDS:
        assert np.array_equal(a[f], b[f][-len(a):]), f


# More worms than the CTA has threads (512 of them with one domain; in a batch
# a CTA takes what its shared memory leaves room for): a thread's worms in
# turns, with sub-blocks, temporal slabs, one group (chains by leg) and a few,
# sparse and with many worms in one interval
TURNS = [
    dict(Lx=20, Ly=20, beta=6.0, eta=0.3, sub_block=2, n_cycle=5, seed=11),
    dict(Lx=20, Ly=20, beta=6.0, eta=0.3, sub_block=4, n_cycle=5, seed=12),
    dict(Lx=20, Ly=20, beta=6.0, eta=0.3, sub_block=0, n_cycle=5, seed=13),
    dict(Lx=20, Ly=20, beta=6.0, eta=0.3, sub_block=0, dom_tau=4, n_cycle=5, seed=14),
    dict(Lx=20, Ly=20, beta=6.0, eta=0.3, sub_block=2, dom_tau=3, n_cycle=5, seed=15),
    dict(Lx=8, Ly=8, beta=6.0, t=0.5, eta=2.0, sub_block=2, n_cycle=5, seed=16),
    dict(Lx=8, Ly=8, beta=6.0, t=0.5, eta=2.0, sub_block=4, n_cycle=5, seed=17),
    dict(Lx=6, Ly=6, beta=8.0, t=0.25, eta=2.5, sub_block=0, n_cycle=5, seed=18),
    dict(Lx=24, Ly=24, beta=4.0, eta=0.6, sub_block=8, n_cycle=5, seed=19),
]


@pytest.mark.parametrize("shift", [0, 24, 36])
@pytest.mark.parametrize("kw", TURNS, ids=["c%d" % i for i in range(len(TURNS))])
def test_more_worms_than_threads_bit_exact(kw, shift):
    g, o = P.Sim(**kw), O.Oracle(**kw)
    o.sweep(8)
    snap = o.export()
    if shift:
        snap = squeezed(snap, shift)
    for s in range(8, 11):
        for x in (g, o):
            x.import_(snap)
            x.sweep_index = s
            x.sweep(1)
        snap = o.export()
        assert np.array_equal(g.export(), snap), "sweep %d" % s
    a, b = g.rows(), o.rows()
    for f in ROW_FIELDS:
        assert np.array_equal(a[f], b[f][-len(a):]), f
    assert a["n_w"].min() > 512  # worms after a sweep; Step 5 neither makes nor removes any


@pytest.mark.parametrize("kw", CASES[2:6] + TURNS, ids=["c%d" % i for i in range(4 + len(TURNS))])
def test_several_domains_of_a_batch_bit_exact(kw):
    """The same in the CTA that a full machine would get, and 2x2 domains."""
    kws = [dict(kw, seed=100 + i, Lx=(1 + i % 2) * kw["Lx"], Ly=(1 + i % 2) * kw["Ly"], dom_x=kw["Lx"],
                dom_y=kw["Ly"], n_cycle=3) for i in range(2)]
    batch = P.Batch(kws)
    batch.sweep(5)
    for i, k in enumerate(kws):
        o = O.Oracle(**k)
        o.sweep(5)
        assert np.array_equal(batch.export(i), o.export()), k
