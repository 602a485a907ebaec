"""The orientation's core bitmap (csrc/orient.cu): its bits are set by the kernels that write the rows, so
it costs no launch of its own, whatever kernel writes a row (at most 32, 512, more entries)."""
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


@pytest.mark.parametrize("name", ["er", "chung_lu", "sparse", "complete"])
def test_core_needs_no_launch(kc, name):
    g = {"er": lambda: kcgen.random_small(300, 0.07, 1), "chung_lu": lambda: kcgen.chung_lu(20000, 200000, 2.1, 2000.0, 1),
         "sparse": lambda: kcgen.chung_lu(30000, 60000, 2.5, 50.0, 2), "complete": lambda: kcgen.complete(1100)}[name]()
    kc.orient(g.off, g.adj).free()
    kc.set_param(kc.KC_PARAM_LAUNCH_COUNT, 0)
    G = kc.orient(g.off, g.adj)
    bits = min(g.n - 1, 2 * g.m).bit_length()
    # degrees, rank, two gathers, offsets, three row kernels, queue; a sort pass for each byte of a degree
    assert kc.get_param(kc.KC_PARAM_LAUNCH_COUNT) == 9 + (bits + 7) // 8
    for k in (3, 4):
        t, pv, po = kc.count(G, k, per_vertex=True, per_owner=True)
        if name == "complete":
            assert t == comb(g.n, k) and np.all(pv == comb(g.n - 1, k - 1))
        else:
            ot, opo, opv = oracle.count(g, k, per_owner=True, per_vertex=True)
            assert t == ot and np.array_equal(pv, opv) and np.array_equal(po, opo)
