"""Candidate sets closed on a compact copy of their subgraph (csrc/close.cu):
every row width of the copy (1..16 words), both sides of the flip to the
complement, against the oracle where it can enumerate the cliques, against
closed forms, and against the ordered search (KC_PARAM_COMPLEMENT = 0)."""
import itertools
from math import comb

import numpy as np
import pytest

import kcgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_1403_0734_gb300 as kc
    return kc


def counts(kc, G, k):
    t, pv, po = kc.count(G, k, per_vertex=True, per_owner=True)
    assert int(pv.sum()) == k * t and int(po.sum()) == t
    assert kc.count(G, k)[0] == t  # totals only
    return t, pv, po


@pytest.mark.parametrize("n,p,k", [(70, 0.85, 6), (140, 0.6, 6), (140, 0.3, 6), (180, 0.55, 6), (300, 0.42, 6),
                                   (150, 0.5, 7)])
def test_close_matches_oracle(kc, n, p, k):
    g = kcgen.random_small(n, p, n + k)
    G = kc.orient(g.off, g.adj)
    t, pv, po = counts(kc, G, k)
    ot, opo, opv = oracle.count(g, k, per_owner=True, per_vertex=True)
    assert t == ot and np.array_equal(pv, opv) and np.array_equal(po, opo)
    for c in (1, 2, 3):
        s, _, spo = kc.estimate(G, k, c, 5, per_owner=True)
        os_, _, ospo = oracle.estimate(g, k, c, 5, per_owner=True)
        assert s == os_ and np.array_equal(spo, ospo)


@pytest.mark.parametrize("n,p,k", [(135, 0.9, 6), (200, 0.97, 6), (260, 0.75, 6), (300, 0.9, 6), (420, 0.95, 6),
                                   (511, 0.8, 6), (280, 0.8, 7), (160, 0.93, 7)])
def test_close_matches_search(kc, n, p, k):
    g = kcgen.random_small(n, p, 7 * n + k)
    G = kc.orient(g.off, g.adj)
    got = counts(kc, G, k)
    kc.set_param(kc.KC_PARAM_COMPLEMENT, 0)
    try:
        want = counts(kc, G, k)
    finally:
        kc.set_param(kc.KC_PARAM_COMPLEMENT, 1)
    assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])


def elementary(parts, k):
    e = [1] + [0] * k
    for a in parts:
        for j in range(k, 0, -1):
            e[j] += a * e[j - 1]
    return e[k]


@pytest.mark.parametrize("parts", [(1,) * 500, (2,) * 250, (4,) * 100, (5,) * 30, (40,) * 9])
@pytest.mark.parametrize("k", [6, 7])
def test_close_closed_forms(kc, parts, k):
    # equal parts: the complement is a disjoint union of cliques (edges, triangles and 4-cliques in it)
    g = kcgen.complete_multipartite(parts, shuffle_seed=3)
    G = kc.orient(g.off, g.adj)
    t, pv, _ = counts(kc, G, k)
    q = elementary(parts, k)
    assert t == q and np.all(pv == q * k // sum(parts))


@pytest.mark.parametrize("k", [4, 5, 6])
def test_batch_of_wide_graphs(kc, k):
    # owners of every class in several graphs of one launch sequence
    graphs = [kcgen.random_small(n, p, 31 * n) for n, p in ((300, 0.5), (40, 0.9), (520, 0.35), (200, 0.6), (90, 0.8))]
    Gs = [kc.orient(g.off, g.adj) for g in graphs]
    assert kc.count_batch(Gs, k) == [kc.count(G, k)[0] for G in Gs]
    assert kc.count(Gs[4], k)[0] == oracle.count(graphs[4], k)[0]
