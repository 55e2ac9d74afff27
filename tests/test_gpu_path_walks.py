"""Paths through bit-parallel vertices, whose last step goes to a vertex that is known:
a root or a member of its set, of the pair's own graph in a batch index, at both
ends of long neighbour lists."""
import numpy as np
import pytest

from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from . import brute, graphs
from .gpu_util import dev_u32, gpu_build
from .paths_util import adjacency_sets, check_path

pytestmark = pytest.mark.gpu


def check(P, g, D):
    adj = adjacency_sets(g)
    s, u = np.meshgrid(np.arange(g.n), np.arange(g.n), indexing="ij")
    s, u = s.ravel().astype(np.uint32), u.ravel().astype(np.uint32)
    if len(s) > 40_000:
        at = np.sort(np.argsort(gg.uniform(7, len(s)))[:40_000])
        s, u = s[at], u[at]
    for a, b, p in zip(s.tolist(), u.tolist(), P.paths(dev_u32(s), dev_u32(u))):
        check_path(p.tolist(), a, b, D, adj)


@pytest.mark.parametrize("t", [1, 3, 64])
@pytest.mark.parametrize("make", [lambda: graphs.complete(200), lambda: graphs.star(300), lambda: gg.ba(400, 40, 1),
                                  lambda: gg.ws(500, 60, 0.1, 2), lambda: graphs.grid(3, 90)],
                         ids=["complete", "star", "ba", "ws", "grid"])
def test_every_end(make, t, tmp_path):
    g = make()
    D = brute.apsp(g.offsets, g.cols)
    ix = gpu_build(g, t)
    ix.save(tmp_path / "i")
    for index in (ix, pll.Index.load(tmp_path / "i")):
        with pll.Paths(index, dev_u32(g.offsets), dev_u32(g.cols)) as P:
            check(P, g, D)


@pytest.mark.parametrize("t", [2, 16])
def test_each_graph_of_a_batch_has_its_own_roots(t):
    parts = [graphs.complete(60), gg.ba(90, 20, 1), graphs.star(50), gg.ws(80, 20, 0.2, 3), graphs.path(12)]
    off, col, start = gg.union(parts)
    g = graphs.disjoint(*parts)
    assert np.array_equal(g.cols, col)
    ix = pll.Index.build_batch(dev_u32(off), dev_u32(col), start, t=t)
    with pll.Paths(ix, dev_u32(off), dev_u32(col)) as P:
        check(P, g, brute.apsp(g.offsets, g.cols))


def test_a_file_with_wrong_graph_ids(tmp_path):
    """The graph ids of a batch index's file are taken as they are: paths through roots are refused, as
    for a graph that is not the index's, and distances inside a graph stay."""
    parts = [graphs.complete(60), gg.ba(90, 20, 1)]
    off, col, start = gg.union(parts)
    t, n = 16, 150
    ix = pll.Index.build_batch(dev_u32(off), dev_u32(col), start, t=t)
    path = tmp_path / "i"
    ix.save(path)
    data = bytearray(path.read_bytes())
    at = len(data) - 4 * ix.label_entries() - 8 * (n + 1) - 4 * n
    ids = np.frombuffer(bytes(data[at:at + 4 * n]), np.uint32)
    assert sorted(np.bincount(ids).tolist()) == [60, 90]
    data[at:at + 4 * n] = (ids + 1_000_000).tobytes()
    path.write_bytes(bytes(data))
    wrong = pll.Index.load(path)
    s, u = dev_u32(np.arange(59, dtype=np.uint32)), dev_u32(np.arange(1, 60, dtype=np.uint32))
    assert bool((wrong.query(s, u) == 1).all())
    with pll.Paths(wrong, dev_u32(off), dev_u32(col)) as P:
        with pytest.raises(pll.PLLError) as e:
            P.query(s, u)
    assert e.value.code == pll.PLL_E_INVAL
