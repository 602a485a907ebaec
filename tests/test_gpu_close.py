"""Candidate sets closed on a compact copy of their subgraph (csrc/close.cu):
every row width of the copy (1..16 words), both sides of the flip to the
complement, against the oracle where it can enumerate the cliques, against
closed forms, and against the ordered search (KC_PARAM_COMPLEMENT = 0)."""
# Sets are closed at k = 5 and 6; the cases at k = 7 run the ordered search over the same graphs.
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


@pytest.mark.parametrize("d", [31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1000, 1024])
@pytest.mark.parametrize("k", [3, 4, 5])
def test_class_edges(kc, d, k):
    # K_{d+1}: its first owner has d elements; then d elements of three colours and an apex
    G = kc.orient(*_csr(kcgen.complete(d + 1)))
    t, pv, _ = counts(kc, G, k)
    assert t == comb(d + 1, k) and np.all(pv == comb(d, k - 1))
    parts = (1,) + (d // 3, d // 3, d - 2 * (d // 3))
    G = kc.orient(*_csr(kcgen.complete_multipartite(parts, shuffle_seed=d)))
    assert counts(kc, G, k)[0] == elementary(parts, k)


def _csr(g):
    return g.off, g.adj


@pytest.mark.parametrize("name", ["sbm", "chung_lu", "dense"])
@pytest.mark.parametrize("k", [3, 4, 5, 6])
def test_rows_from_lists_and_core(kc, name, k):
    # rows read from sorted lists, from the bitmap of the last ranks, and from both within one owner
    g = {"sbm": lambda: kcgen.sbm(2000, 50, 0.5, 50000, 4), "chung_lu": lambda: kcgen.chung_lu(3000, 40000, 2.1, 400.0, 5),
         "dense": lambda: kcgen.random_small(120, 0.5, 6)}[name]()
    G = kc.orient(*_csr(g))
    t, pv, po = counts(kc, G, k)
    ot, opo, opv = oracle.count(g, k, per_owner=True, per_vertex=True)
    assert t == ot and np.array_equal(pv, opv) and np.array_equal(po, opo)
    assert kc.count_batch([G, G], k) == [t, t]
    for c in (1, 3):
        s, _, spo = kc.estimate(G, k, c, 5, per_owner=True)
        os_, _, ospo = oracle.estimate(g, k, c, 5, per_owner=True)
        assert s == os_ and np.array_equal(spo, ospo)
    if k <= 4:
        rows = np.sort(kc.list_cliques(G, k), axis=1)
        want = np.sort(oracle.list_cliques(g, k), axis=1)
        assert np.array_equal(rows[np.lexsort(rows.T)], want[np.lexsort(want.T)])


@pytest.mark.parametrize("k", [3, 4, 5])
def test_listing_order_and_alignment(kc, k):
    # owners of 1..8 words; the same rows in the same places of a buffer that starts off a 16-byte boundary
    import torch
    g = kcgen.random_small(300, 0.45, 8)
    G = kc.orient(*_csr(g))
    want = oracle.list_cliques(g, k)
    buf = torch.empty((len(want) + 1) * k + 1, dtype=torch.int32, device="cuda")
    got = []
    for start in (0, 1):
        buf.fill_(-1)
        part = buf[start:]
        assert kc.list_runs(G, k, lambda a: False, cap=len(want), device_buffer=part) == len(want)
        rows = part[: len(want) * k].view(len(want), k).cpu().numpy()
        assert int((part[len(want) * k :] == -1).all()) and (start == 0 or int(buf[0]) == -1)
        got.append(rows.copy())
    assert np.array_equal(got[0], got[1])
    a, b = np.sort(got[0], axis=1), np.sort(want, axis=1)
    assert np.array_equal(a[np.lexsort(a.T)], b[np.lexsort(b.T)])


@pytest.mark.parametrize("pairs", [40, 65])
def test_work_counter_counts_edges(kc, pairs):
    # K_{2,2,...,2}: every candidate set's complement is a matching, edges without triangles.  Owners of more than
    # 64 elements alone: less the work of the same graph's last 66 vertices.
    def work(n):
        G = kc.orient(*_csr(kcgen.complete_multipartite((2,) * n)))
        kc.set_param(kc.KC_PARAM_WORK_COUNT, 1)
        try:
            t = kc.count(G, 6)[0]
            return t, kc.get_param(kc.KC_PARAM_WORK_COUNT)
        finally:
            kc.set_param(kc.KC_PARAM_WORK_COUNT, 0)

    want = 0
    for half in range(33, pairs):          # two owners each, of 2 half elements
        for c in range(4, 2 * half, 2):    # two sets each: rows squeezed, all rows met by each, the matching's edges
            wc = 1 if c <= 32 else 4
            want += 4 * (c * ((2 * half + 31) // 32 + c * wc) + c // 2 * wc)
    (t, w), (_, last) = work(pairs), work(33)
    assert t == comb(pairs, 6) * 64 and w - last == want


def apex_over(parts):
    """A vertex adjacent to all of a complete multipartite graph whose vertices have one pendant for each vertex of
    their part: by degree the apex comes before them, so it is an owner of exactly sum(parts) elements."""
    d = sum(parts)
    label = np.repeat(np.arange(len(parts)), parts)
    iu, ju = np.triu_indices(d, 1)
    cross = label[iu] != label[ju]
    size = np.array(parts)[label]
    at = np.repeat(np.arange(d), size)
    edges = [np.stack([iu[cross], ju[cross]], axis=1), np.stack([np.full(d, d), np.arange(d)], axis=1),
             np.stack([at, d + 1 + np.arange(len(at))], axis=1)]
    return kcgen.from_edges(d + 1 + len(at), np.concatenate(edges), f"apex_{d}"), label


@pytest.mark.parametrize("k,d", [(k, d) for k in (5, 6) for d in (31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512)]
                         + [(5, 513), (4, 64), (4, 65), (4, 512), (4, 513)])
def test_class_edges_multipartite(kc, k, d):
    # eight unequal parts: cliques of every k, and complements that are cliques of different sizes
    cut = [d * i * (i + 1) // 72 for i in range(9)]
    parts = tuple(b - a for a, b in zip(cut, cut[1:]) if b > a)
    assert sum(parts) == d and len(set(parts)) >= 5
    g, label = apex_over(parts)
    G = kc.orient(*_csr(g))
    assert G.max_dplus == d
    t, pv, po = counts(kc, G, k)
    assert t == elementary((1,) + parts, k) > 0 and int(po[d]) == elementary(parts, k - 1)
    for i, p in enumerate(parts):
        rest = (1,) + parts[:i] + parts[i + 1:]
        assert np.all(pv[:d][label == i] == elementary(rest, k - 1))
    assert int(pv[d]) == elementary(parts, k - 1) and np.all(pv[d + 1:] == 0)


@pytest.mark.parametrize("n,p", [(900, 0.4), (520, 0.55), (500, 0.7), (420, 0.9)])
def test_close_matches_search_at_five(kc, n, p):
    # 16-word owners at k = 5, their sets on both sides of half density
    g = kcgen.random_small(n, p, 3 * n)
    G = kc.orient(g.off, g.adj)
    assert 257 <= G.max_dplus <= 512
    got = counts(kc, G, 5)
    kc.set_param(kc.KC_PARAM_COMPLEMENT, 0)
    try:
        want = counts(kc, G, 5)
    finally:
        kc.set_param(kc.KC_PARAM_COMPLEMENT, 1)
    assert got[0] == want[0] and np.array_equal(got[1], want[1]) and np.array_equal(got[2], want[2])


@pytest.mark.parametrize("maxw", [1, 2, 4])
@pytest.mark.parametrize("k", [3, 4, 5])
def test_listing_on_narrow_global_tiles(kc, maxw, k):
    # owners of 2..8 words forced onto global tiles
    g = kcgen.random_small(260, 0.35, 8)
    G = kc.orient(*_csr(g))
    want = oracle.list_cliques(g, k)
    kc.set_param(kc.KC_PARAM_SMEM_MAX_WORDS, maxw)
    try:
        got = kc.list_cliques(G, k)
    finally:
        kc.set_param(kc.KC_PARAM_SMEM_MAX_WORDS, 32)
    a, b = np.sort(got, axis=1), np.sort(want, axis=1)
    assert np.array_equal(a[np.lexsort(a.T)], b[np.lexsort(b.T)])
