"""Checkpoints that are packed and checked on the device: the same bytes as
the oracle's, the same statuses as a check in buffer order, and slots too full
or too few for the packed form (which then take the host's)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from oracle import oracle as O  # noqa: E402

import paper_1307_0328_gb300 as P  # noqa: E402


@pytest.mark.parametrize("cap_site", [0, 2048])  # (8x8 and up: 2048 slots a site take the packed form)
@pytest.mark.parametrize("kw", [
    dict(Lx=2, Ly=2, beta=1.5, eta=0.5, n_cycle=4, seed=3, init=0),
    dict(Lx=19, Ly=17, beta=2.0, eta=0.3, V=0.5, mu=0.4, n_cycle=4, seed=29),
    dict(Lx=8, Ly=8, beta=4.0, eta=0.2, n_cycle=4, seed=1),
])
def test_export_and_import(kw, cap_site):
    g, o = P.Sim(**dict(kw, cap_site=cap_site)), O.Oracle(**kw)
    assert np.array_equal(g.export(), o.export())  # no events yet
    o.sweep(6)
    snap = o.export()
    g.import_(snap)
    assert np.array_equal(g.export(), snap)
    # slots with no room beside the events: the capacity is the largest count
    counts, k = [], 1
    for _ in range(int(snap[0])):
        counts.append(int(snap[k]) & 0x7fffffff)
        k += 1 + counts[-1]
    cap = max(counts)
    full = P.Sim(**dict(kw, cap_site=cap))
    full.import_(snap)
    assert np.array_equal(full.export(), snap)
    if cap > 8:
        tight = P.Sim(**dict(kw, cap_site=8 * ((cap - 1) // 8)))
        with pytest.raises(P.PmwaError) as e:
            tight.import_(snap)
        assert e.value.status == P.PMWA_ECAPACITY


@pytest.mark.parametrize("cap_site", [0, 2048])
def test_first_wrong_site_names_the_status(cap_site):
    """An invariant broken at an earlier site comes before a header that is
    wrong at a later one, and after one that is wrong earlier."""
    kw = dict(Lx=8, Ly=8, beta=2.0, eta=0.3, n_cycle=4, seed=5)
    g, o = P.Sim(**dict(kw, cap_site=cap_site)), O.Oracle(**kw)
    o.sweep(6)
    snap = o.export()
    heads, k = [], 1
    for _ in range(64):
        heads.append(k)
        k += 1 + (int(snap[k]) & 0x7fffffff)
    busy = [h for h in heads if int(snap[h]) & 0x7fffffff]

    def status(edit):
        b = snap.copy()
        edit(b)
        with pytest.raises(P.PmwaError) as e:
            g.import_(b)
        return e.value.status

    def flip(h):
        return lambda b: b.__setitem__(h + 1, b[h + 1] ^ np.uint64(1))

    def grow(h):
        return lambda b: b.__setitem__(h, np.uint64(0x7ffffff0))

    g.import_(snap)
    assert status(flip(busy[3])) == P.PMWA_EINVARIANT
    assert status(grow(busy[3])) == P.PMWA_ECAPACITY
    assert status(lambda b: (flip(busy[2])(b), grow(busy[9])(b))) == P.PMWA_EINVARIANT
    assert status(lambda b: (grow(busy[2])(b), flip(busy[9])(b))) == P.PMWA_ECAPACITY
    with pytest.raises(P.PmwaError) as e:
        g.import_(snap[:-1])
    assert e.value.status == P.PMWA_EINVAL
    assert np.array_equal(g.export(), snap)  # a refused buffer changes nothing


@pytest.mark.parametrize("full", [57342, 57344, 65536])
def test_slots_at_the_limit_of_the_packed_form(full):
    """65536 slots whose packed words, places and answer fill the scratch to its
    last word (57342 events of 4096 sites: 4097 + 4096 + 1 words beside them), do
    not fit by one event pair, or whose slots are all taken: the same bytes back,
    and an invariant broken at the last site is found."""
    kw = dict(Lx=64, Ly=64, dom_x=16, dom_y=16, beta=1.0, eta=0.3, n_cycle=4, seed=5, cap_site=16)
    n = np.full(4096, {57342: 14, 57344: 14, 65536: 16}[full], dtype=np.int64)
    if full == 57342:
        n[7] = 12
    assert n.sum() == full
    words = [np.array([4096], dtype=np.uint64)]
    for s, c in enumerate(n):
        j = np.arange(c, dtype=np.uint64)
        m = (j << np.uint64(52)) + np.uint64(977 * s + 1)
        words.append(np.array([int(c)], dtype=np.uint64))  # state 0 above the last worm
        words.append((m << np.uint64(5)) | np.uint64(28) | ((j + np.uint64(1)) & np.uint64(1)))
    buf = np.concatenate(words)
    g = P.Sim(**kw)
    g.import_(buf)
    assert np.array_equal(g.export(), buf)
    assert g.check() is None
    bad = buf.copy()
    bad[-1] ^= np.uint64(1)
    with pytest.raises(P.PmwaError) as e:
        g.import_(bad)
    assert e.value.status == P.PMWA_EINVARIANT
    assert np.array_equal(g.export(), buf)
