"""Owners with few edges or none among their elements: random graphs with next to no triangles, and the
same with a few cliques planted, against the oracle."""
import numpy as np
import pytest

import kcgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_1403_0734_gb300 as kc
    return kc


def sparse(n, m, cliques, size, seed):
    rng = np.random.default_rng(seed)
    edges = [rng.integers(n, size=(m, 2))]
    iu, ju = np.triu_indices(size, 1)
    for _ in range(cliques):
        c = rng.choice(n, size, replace=False)
        edges.append(np.stack([c[iu], c[ju]], axis=1))
    return kcgen.from_edges(n, np.concatenate(edges), f"sparse_{n}_{m}")


def check(kc, g, k):
    G = kc.orient(g.off, g.adj)
    t, pv, po = kc.count(G, k, per_vertex=True, per_owner=True)
    ot, opo, opv = oracle.count(g, k, per_owner=True, per_vertex=True)
    assert t == ot and np.array_equal(pv, opv) and np.array_equal(po, opo)
    assert kc.count(G, k)[0] == t and kc.count_batch([G, G], k) == [t, t] and kc.count_static(G, k) == t
    s, _, spo = kc.estimate(G, k, 2, 5, per_owner=True)
    os_, _, ospo = oracle.estimate(g, k, 2, 5, per_owner=True)
    assert s == os_ and np.array_equal(spo, ospo)
    s, _, spo = kc.estimate_pairs(G, k, 0.7, 5, per_owner=True)
    os_, _, ospo = oracle.estimate_pairs(g, k, 0.7, 5, per_owner=True)
    assert s == os_ and np.array_equal(spo, ospo)


@pytest.mark.parametrize("n,per,cliques,size", [(20000, 45, 0, 0), (20000, 45, 60, 8), (3000, 40, 5, 12)])
@pytest.mark.parametrize("k", [3, 4, 5, 6, 7])
def test_sparse_two_word_owners(kc, n, per, cliques, size, k):
    check(kc, sparse(n, n * per, cliques, size, n + cliques), k)


@pytest.mark.parametrize("n,per,cliques,size", [(30000, 2, 0, 0), (30000, 3, 400, 6), (40000, 4, 100, 20), (30000, 7, 0, 0),
                                                (9000, 3, 50, 6)])
def test_sparse_one_word_owners(kc, n, per, cliques, size):
    # both sides of the rule at k = 3: on average 2.7..7 elements, more and fewer than 16384 owners
    g = sparse(n, n * per, cliques, size, n + per)
    check(kc, g, 3)
    G = kc.orient(g.off, g.adj)
    t, pv, po = kc.count(G, 3, per_vertex=True, per_owner=True)
    parts = [kc.count_part(G, 3, p, 3, per_vertex=True, per_owner=True) for p in range(3)]
    assert sum(p[0] for p in parts) == t
    assert np.array_equal(sum(p[1] for p in parts), pv) and np.array_equal(sum(p[2] for p in parts), po)
    got = np.sort(kc.list_cliques(G, 3), axis=1)
    want = np.sort(oracle.list_cliques(g, 3), axis=1)
    assert np.array_equal(got[np.lexsort(got.T)], want[np.lexsort(want.T)])


@pytest.mark.parametrize("p", [0.05, 0.4, 0.89, 0.91, 0.99])
@pytest.mark.parametrize("k", [4, 5, 6])
def test_pairs_in_wide_owners(kc, p, k):
    # owners of 16 words, both sides of the rule at k = 5 (p = 0.9)
    g = kcgen.from_edges(1100, np.random.default_rng(2).integers(1100, size=(200000, 2)), "wide")
    G = kc.orient(g.off, g.adj)
    assert 256 < G.max_dplus <= 512
    s, _, spo = kc.estimate_pairs(G, k, p, 5, per_owner=True)
    os_, _, ospo = oracle.estimate_pairs(g, k, p, 5, per_owner=True)
    assert s == os_ and np.array_equal(spo, ospo)


@pytest.mark.parametrize("n,m", [(1100, 200000), (3000, 600000), (24000, 7200000)])
def test_pairs_over_parts(kc, n, m):
    # some 150, 1000 and 11000 owners of 16 words: searched over 16, 4 parts and one
    g = kcgen.from_edges(n, np.random.default_rng(3).integers(n, size=(m, 2)), "wide")
    G = kc.orient(g.off, g.adj)
    d = np.diff(kc.export(G)["off_plus"])
    owners = int(((d > 256) & (d <= 512)).sum())
    assert (owners >= 600) + (owners >= 8192) == [1100, 3000, 24000].index(n)
    s, _, spo = kc.estimate_pairs(G, 5, 0.5, 5, per_owner=True)
    os_, _, ospo = oracle.estimate_pairs(g, 5, 0.5, 5, per_owner=True)
    assert s == os_ and np.array_equal(spo, ospo)


@pytest.mark.parametrize("n,p,k", [(520, 0.5, 5), (560, 0.75, 5), (420, 0.9, 5), (700, 0.4, 6), (440, 0.62, 6)])
def test_closed_or_searched_by_density(kc, n, p, k):
    """Owners of 8 and 16 words of a dense graph, and of the same graph among 20,000 vertices without edges: whether
    their sets are closed or searched depends on the density of the whole."""
    g = kcgen.random_small(n, p, 5)
    G = kc.orient(g.off, g.adj)
    assert 128 < G.max_dplus <= 512
    off = np.concatenate([g.off, np.full(20000 - n, g.off[-1])])
    H = kc.orient(off, g.adj)
    t, pv, po = kc.count(G, k, per_vertex=True, per_owner=True)
    tt, ppv, ppo = kc.count(H, k, per_vertex=True, per_owner=True)
    assert t == tt and np.array_equal(pv, ppv[:n]) and np.array_equal(po, ppo[:n])
    for X in (G, H):
        x, _, xo = kc.count(X, k, per_owner=True)
        assert x == t and np.array_equal(xo[:n], po) and kc.count_batch([X, X], k) == [t, t]
    for c in (2, 5):
        a, b = kc.estimate(G, k, c, 3, per_owner=True), kc.estimate(H, k, c, 3, per_owner=True)
        assert a[0] == b[0] and np.array_equal(a[2], b[2][:n])
    for q in (0.5, 0.7, 0.85, 0.95):
        a, b = kc.estimate_pairs(G, k, q, 3, per_owner=True), kc.estimate_pairs(H, k, q, 3, per_owner=True)
        assert a[0] == b[0] and np.array_equal(a[2], b[2][:n])


@pytest.mark.parametrize("ps", [(0.5, 0.6), (0.5, 0.95), (0.02, 0.6), (0.3,)])
def test_batches_by_density(kc, ps):
    # 16-word owners in graphs of middling density, in one denser, beside a sparse graph, and none at all
    graphs = [kcgen.random_small(560, p, 7) for p in ps]
    Gs = [kc.orient(g.off, g.adj) for g in graphs]
    for k in (5, 6):
        assert kc.count_batch(Gs, k) == [kc.count(G, k, per_vertex=True)[0] for G in Gs]
