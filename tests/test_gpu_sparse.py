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
