"""The ordered search's complement count with saturated non-degree bytes, on the paths that still run it."""
from math import comb

import numpy as np
import pytest

import kcgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kc():
    import paper_1403_0734_gb300 as kc
    return kc


@pytest.fixture(scope="module")
def split_core(kc):
    """K_500 on S + T (200 and 300 vertices), a vertex a adjacent to S only, pendants so that by degree S < T < a.  A
    first-level set of an owner in S is S above it, T and a, with edges between all but a and T: 300 non-edges
    among some 125,000 pairs (closed through the complement), all of them at a, whose byte stops at 255."""
    S, T, a = np.arange(200), np.arange(200, 500), 500
    iu, ju = np.triu_indices(500, 1)
    edges = [np.stack([iu, ju], axis=1), np.stack([np.full(200, a), S], axis=1),
             np.stack([np.repeat(T, 5), 501 + np.arange(1500)], axis=1),
             np.stack([np.full(400, a), 2001 + np.arange(400)], axis=1)]
    g = kcgen.from_edges(2401, np.concatenate(edges), "k500_split_core")
    G = kc.orient(g.off, g.adj)
    assert 257 <= G.max_dplus <= 512
    yield G
    G.free()


@pytest.mark.parametrize("k,pv", [(5, True), (6, False), (6, True)])
def test_saturated_non_degrees_in_the_unsplit_search(kc, split_core, k, pv):
    G, total = split_core, comb(500, k) + comb(200, k - 1)
    kc.set_tuning(G, {"k": k, "per_vertex": pv, "algo": [kc.KC_ALGO_DFS] * 7, "parts": [1] * 7})
    try:
        t, mem, _ = kc.count(G, k, per_vertex=pv)
    finally:
        kc.set_tuning(G, None)
    assert t == total
    if pv:
        assert int(mem[500]) == comb(200, k - 1) and np.all(mem[:200] == comb(499, k - 1) + comb(199, k - 2))
        assert np.all(mem[200:500] == comb(499, k - 1)) and np.all(mem[501:] == 0)


@pytest.mark.parametrize("k", [5, 6])
def test_saturated_non_degrees_without_allocation(kc, split_core, k):
    assert kc.count_static(split_core, k) == comb(500, k) + comb(200, k - 1)
