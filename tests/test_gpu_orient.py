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


def circulant(n, r):
    """Vertex i adjacent to i +- 1..r modulo n; n C(r, k - 1) k-cliques for n > 3 r, all on arcs of r + 1."""
    d = np.concatenate([np.arange(-r, 0), np.arange(1, r + 1)])
    adj = np.sort((np.arange(n)[:, None] + d) % n, axis=1).astype(np.int32)
    return np.arange(n + 1, dtype=np.int64) * 2 * r, adj.reshape(-1)


@pytest.mark.parametrize("n,r", [(10, 2), (100, 3), (300, 40), (5000, 7), (20000, 2)])
def test_core_declined_and_its_size(kc, n, r):
    off, adj = circulant(n, r)
    m = n * r
    A, B = kc.orient(off, adj), kc.orient(off, adj, core=False)
    # T: rounded up to 128 from the least of n, 16384 and sqrt(32 m), but 128 at least
    T = max(128, -(-min(n, 16384, int((32 * m) ** 0.5)) // 128) * 128)
    assert 0 < A.device_bytes - B.device_bytes <= min(n, T) * T // 8 + 255
    a, b = kc.export(A), kc.export(B)
    assert all(np.array_equal(a[x], b[x]) for x in a)
    for k in (2, 3, 4, 5, 6):
        x, y = kc.count(A, k, per_vertex=True, per_owner=True), kc.count(B, k, per_vertex=True, per_owner=True)
        assert x[0] == y[0] and np.array_equal(x[1], y[1]) and np.array_equal(x[2], y[2])
        if n > 3 * r:
            assert x[0] == n * comb(r, k - 1)
        assert kc.count_batch([A, B], k) == [x[0], x[0]]
        s, t = kc.estimate(A, k, 2, 9, per_owner=True), kc.estimate(B, k, 2, 9, per_owner=True)
        assert s[0] == t[0] and np.array_equal(s[2], t[2])


LITTLE_MEMORY = """
import ctypes, sys
import numpy as np, torch
sys.path.insert(0, "tests")
import paper_1403_0734_gb300 as kc
from test_gpu_orient import circulant
off, adj = circulant(16384, 512)  # lists and bitmap of 32 MiB each, scratch of 64
lo, la = (torch.from_numpy(x).cuda() for x in circulant(2000, 40))
G = kc.orient(lo, la); kc.count(G, 3); G.free()  # kernels loaded
off, adj = torch.from_numpy(off).cuda(), torch.from_numpy(adj).cuda()
torch.cuda.synchronize()
fill = [torch.empty(torch.cuda.mem_get_info()[0] - (1 << 30), dtype=torch.uint8, device="cuda")]
while True:
    try:
        fill.append(torch.empty(16 << 20, dtype=torch.uint8, device="cuda"))
    except torch.OutOfMemoryError:
        break
seen = []
while len(fill) > 1:
    try:
        G = kc.orient(off, adj)
    except kc.KcError:
        seen.append("none")
    else:
        assert kc.count(G, 3)[0] == 16384 * 512 * 511 // 2
        seen.append("core" if G.device_bytes > 4 * 16384 * 512 + (32 << 20) else "lists")
        G.free()
        if seen[-1] == "core":
            break
    fill.pop()
    torch.cuda.empty_cache()
print("steps", ",".join(seen))
"""


def test_no_memory_for_the_core(kc):
    """As memory is given back in steps of 16 MiB, the graph is refused, then fits without its bitmap, then with it."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", LITTLE_MEMORY], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    steps = r.stdout.split("steps ")[1].strip().split(",")
    order = [s for i, s in enumerate(steps) if i == 0 or steps[i - 1] != s]
    assert order == ["none", "lists", "core"], steps
