"""The pruned stage's sweeps at the sizes where their paths change, against the
oracle's labels: row widths (t around 16, 32, 48), levels at which the distance
test changes its rows (5 to nibbles, 60 to clamped bytes, then bytes), neighbour
lists around the slice length, lists cut at every batch's first rank, labels
longer than a root's table, and depths next to the 8-bit limit."""
import numpy as np
import pytest

import oracle
from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from . import graphs
from .gpu_util import dev_u32, first_label_diff, gpu_build, same_labels

pytestmark = pytest.mark.gpu


def hubs(degrees, seed):
    """One hub of each given degree over a shared set of leaves, plus random edges among them."""
    n = len(degrees) + max(degrees) + 40
    e, leaf0 = [], len(degrees)
    for h, d in enumerate(degrees):
        e += [(h, leaf0 + (7 * h + i) % (n - leaf0)) for i in range(d)]
    x = gg.below(seed, 4 * n, n).astype(np.int64).reshape(-1, 2)
    e = np.concatenate([np.asarray(e, dtype=np.int64), x])
    return gg.from_edges(n, e[:, 0], e[:, 1], f"hubs{degrees}")


def check(g, t, **kw):
    ref = oracle.Index(g.offsets, g.cols, t)
    ix = gpu_build(g, t, **kw)
    La, Lb = ix.labels(), ref.labels()
    assert same_labels(La, Lb), first_label_diff(La, Lb, g.n)


@pytest.mark.parametrize("t", [0, 1, 15, 17, 31, 32, 33, 48, 49, 63])
@pytest.mark.parametrize("root_batch", [0, 3, 64])
def test_row_widths_and_slice_lengths(t, root_batch):
    check(hubs([63, 64, 65, 127, 128, 129, 192, 193, 257, 700], 5), t, root_batch=root_batch)


@pytest.mark.parametrize("t", [0, 2, 33])
@pytest.mark.parametrize("make", [lambda: graphs.grid(4, 9), lambda: graphs.grid(3, 70), lambda: graphs.grid(2, 130),
                                  lambda: graphs.path(250), lambda: graphs.cycle(505)],
                         ids=["grid4x9", "grid3x70", "grid2x130", "path250", "cycle505"])
@pytest.mark.parametrize("root_batch", [1, 40, 0])
def test_levels_across_the_row_kinds(make, t, root_batch):
    check(make(), t, root_batch=root_batch)


@pytest.mark.parametrize("t", [0, 1])
@pytest.mark.parametrize("n", [300, 520])
def test_a_depth_of_255_is_still_a_range_error(n, t):
    g = graphs.path(n) if n == 300 else graphs.cycle(n)
    with pytest.raises(pll.PLLError) as e:
        gpu_build(g, t)
    assert e.value.code == pll.PLL_E_RANGE


def test_labels_longer_than_a_roots_table():
    """No bit-parallel labels on a random-order high-diameter graph: labels of
    over a thousand entries, past the largest reach table's share of four bytes
    an entry."""
    g = gg.ws(4000, 8, 0.5, 9)
    order = np.argsort(gg.uniform(3, g.n)).astype(np.uint32)
    ref = oracle.Index(g.offsets, g.cols, 0, order=order).labels()
    assert np.diff(ref.offsets.astype(np.int64)).max() > 600
    for root_batch in (0, 100):
        ix = gpu_build(g, 0, order=order, root_batch=root_batch)
        assert same_labels(ix.labels(), ref), first_label_diff(ix.labels(), ref, g.n)


def two_way_ladder(n):
    """A directed path of n vertices with arcs back from everywhere to the first few: deep forward
    BFSs whose vertices reach low ranks at every level."""
    arcs = [(i, i + 1) for i in range(n - 1)] + [(i, j) for i in range(5, n) for j in range(0, 4)]
    return gg.digraph(n, arcs, f"ladder{n}")


@pytest.mark.parametrize("n", [240, 250, 254])
@pytest.mark.parametrize("root_batch", [0, 1, 30])
def test_directed_depths_next_to_the_limit(n, root_batch):
    """Arcs to finished hubs at every depth: the cut lists must give the labels of whole ones, and
    a depth of 255 must be an error only where whole lists make it one."""
    from .gpu_util import dev_u32
    d = two_way_ladder(n)
    ref = oracle.DirectedIndex(d.offsets, d.cols)
    ix = pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols), root_batch=root_batch)
    assert same_labels(ix.labels_in(), ref.labels_in()) and same_labels(ix.labels_out(), ref.labels_out())


@pytest.mark.parametrize("n", [2, 256, 257, 65536, 65537])
def test_rank_space_lists_at_the_sort_widths(n):
    """The lists come from a radix sort over as many bits as a rank has: one, two and three passes."""
    g = graphs.path(2) if n == 2 else gg.ba(n, 2, n)
    check(g, 16)
    d = gg.oriented(g, 3, both=0.3)
    ix, ref = pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols)), oracle.DirectedIndex(d.offsets, d.cols)
    for a, b in ((ix.labels_in(), ref.labels_in()), (ix.labels_out(), ref.labels_out())):
        assert same_labels(a, b), first_label_diff(a, b, d.n)


@pytest.mark.parametrize("name,make,t", [("ba", lambda: gg.ba(20000, 6, 7), 0), ("ws", lambda: gg.ws(12000, 6, 0.02, 2), 0),
                                         ("ws8", lambda: gg.ws(12000, 6, 0.05, 2), 8)])
@pytest.mark.parametrize("root_batch", [0, 500])
def test_stores_that_outgrow_their_near_copy(name, make, t, root_batch):
    """Two to three million entries, at distances on both sides of the last distance class."""
    check(make(), t, root_batch=root_batch)


def test_directed_stores_that_outgrow_their_near_copy():
    d = gg.oriented(gg.ba(20000, 6, 7), 3, both=0.3)
    ref = oracle.DirectedIndex(d.offsets, d.cols)
    ix = pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols), root_batch=1000)
    for a, b in ((ix.labels_in(), ref.labels_in()), (ix.labels_out(), ref.labels_out())):
        assert same_labels(a, b), first_label_diff(a, b, d.n)
