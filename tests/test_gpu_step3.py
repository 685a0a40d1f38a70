"""The sweep kernel at every CTA size and every cut of Step 3's merge, bit for
bit against the oracle: domains whose CTA has less than one up to many threads
a site (the parts of a site's circle), ragged ones that leave lanes idle, with
temporal boundaries, windows and static starts (empty lists).  Alone, a few
domains take large CTAs; in a batch each domain takes the size that its shared
memory leaves room for."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402

import paper_1307_0328_gb300 as P  # noqa: E402

DOMAINS = [(2, 2), (2, 4), (3, 3), (4, 4), (3, 7), (5, 7), (8, 12), (8, 16), (17, 15), (16, 16), (20, 18)]


@pytest.mark.parametrize("extra", [dict(), dict(dom_tau=4), dict(vertex_window=0.2)], ids=["plain", "slabs", "window"])
@pytest.mark.parametrize("dom", DOMAINS, ids=["%dx%d" % d for d in DOMAINS])
def test_step3_bit_exact(dom, extra):
    kw = dict(Lx=2 * dom[0], Ly=2 * dom[1], beta=3.0, V=0.5, mu=0.4, eta=0.3, dom_x=dom[0], dom_y=dom[1],
              n_cycle=3, seed=11, **extra)
    g, o = P.Sim(**kw), O.Oracle(**kw)
    for s in range(6):
        snap = o.export()
        for x in (g, o):
            x.import_(snap)
            x.sweep_index = s
            x.tile(3)
        assert np.array_equal(g.export(), o.export()), "Step 3 at sweep %d" % s
        for x in (g, o):
            x.import_(snap)
            x.sweep_index = s
            x.sweep(1)
        assert np.array_equal(g.export(), o.export()), "sweep %d" % s


@pytest.mark.parametrize("extra", [dict(), dict(dom_tau=4)], ids=["plain", "slabs"])
def test_cta_sizes_of_a_batch_bit_exact(extra):
    kws = [dict(Lx=2 * a, Ly=2 * b, beta=beta, V=0.5, mu=0.4, eta=0.3, dom_x=a, dom_y=b, n_cycle=3, seed=11, **extra)
           for a, b in DOMAINS for beta in (1.0, 6.0)]
    batch = P.Batch(kws)
    batch.sweep(6)
    for i, kw in enumerate(kws):
        o = O.Oracle(**kw)
        o.sweep(6)
        assert np.array_equal(batch.export(i), o.export()), kw


@pytest.mark.parametrize("L", [28, 36, 52, 72])
def test_cta_sizes_by_domain_count_bit_exact(L):
    """4x4 domains: 49, 81, 169 and 324 of them (512 threads down to 128)."""
    kw = dict(Lx=L, Ly=L, beta=2.0, V=0.5, mu=0.4, eta=0.3, dom_x=4, dom_y=4, sub_block=2, n_cycle=3, seed=12)
    g, o = P.Sim(**kw), O.Oracle(**kw)
    g.sweep(5)
    o.sweep(5)
    assert np.array_equal(g.export(), o.export())
