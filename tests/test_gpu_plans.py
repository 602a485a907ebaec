"""Parts per owner in a plan: taken where the class is searched, ignored -- by the launches, by the footprint
and by the tuner -- where it is not."""
import numpy as np
import pytest

import kcgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_1403_0734_gb300 as kc
    return kc


def plan(k, pv, slot=None, parts=1):
    return {"k": k, "per_vertex": pv, "algo": [1] * 7, "parts": [parts if i == slot else 1 for i in range(7)]}


W32, W16, W8, W4, W2 = 1, 2, 3, 4, 5


@pytest.fixture(scope="module")
def graph(kc):
    g = kcgen.random_small(420, 0.7, 3)  # owners of up to 16 words
    G = kc.orient(g.off, g.adj)
    assert 256 < G.max_dplus <= 512
    yield g, G
    G.free()


@pytest.mark.parametrize("k,slot,used", [(4, W16, False), (4, W8, False), (4, W4, False), (6, W4, False), (5, W4, True),
                                         (5, W8, True), (5, W16, True), (6, W8, True), (6, W16, True), (7, W4, True),
                                         (6, W2, True), (9, W8, False)])
def test_footprint_of_parts(kc, graph, k, slot, used):
    G = graph[1]
    bytes_ = []
    for parts in (1, 4):
        kc.set_tuning(G, plan(k, False, slot, parts))
        bytes_.append(kc.footprint(G, k))
    kc.set_tuning(G, None)
    assert (bytes_[1] > bytes_[0]) == used


@pytest.mark.parametrize("k,slot,used", [(4, W4, False), (6, W4, False), (5, W4, True), (5, W16, True)])
@pytest.mark.parametrize("pv", [False, True])
def test_launches_of_parts(kc, graph, k, slot, used, pv):
    g, G = graph
    want = oracle.count(g, k)[0] if k < 5 else None
    launches, totals = [], []
    for parts in (1, 4):
        kc.set_tuning(G, plan(k, pv, slot, parts))
        kc.count(G, k, per_vertex=pv)
        kc.set_param(kc.KC_PARAM_LAUNCH_COUNT, 0)
        totals.append(kc.count(G, k, per_vertex=pv)[0])
        launches.append(kc.get_param(kc.KC_PARAM_LAUNCH_COUNT))
    kc.set_tuning(G, None)
    totals.append(kc.count(G, k)[0])
    assert len(set(totals)) == 1 and want in (None, totals[0])
    assert (launches[1] > launches[0]) == used


@pytest.mark.parametrize("k", [5, 6])
@pytest.mark.parametrize("pv", [False, True])
def test_tuner_times_what_differs(kc, graph, k, pv):
    p = kc.tune(graph[1], k, per_vertex=pv)
    assert p["parts"][W4] in ((1,) if k == 6 else (1, 4, 16))
    # (a graph of density 0.7: totals at k = 5 are searched in the 16-word class, the others closed)
    assert p["parts"][W16] in ((1, 4, 16) if k == 5 and not pv else (1, 16))
    assert p["parts"][W8] in ((1, 4) if k == 6 else (1, 4, 16))


def test_parts_at_five_in_the_four_word_class(kc):
    # totals, estimates and owners' counts over several parts, against the oracle
    g = kcgen.random_small(150, 0.75, 4)
    G = kc.orient(g.off, g.adj)
    assert 64 < G.max_dplus <= 128
    ot, opo, _ = oracle.count(g, 5, per_owner=True)
    os_, _, ospo = oracle.estimate(g, 5, 2, 7, per_owner=True)
    for parts in (1, 2, 4, 16):
        kc.set_tuning(G, plan(5, False, W4, parts))
        t, _, po = kc.count(G, 5, per_owner=True)
        s, _, spo = kc.estimate(G, 5, 2, 7, per_owner=True)
        assert t == ot and np.array_equal(po, opo) and s == os_ and np.array_equal(spo, ospo)
        assert kc.count_static(G, 5) == ot
