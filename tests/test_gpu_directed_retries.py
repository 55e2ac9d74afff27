"""The directed build where a batch runs again: buffers that overflow, roots without
a table, label pools that move, and a depth of 255 that only the cut lists show."""
import numpy as np
import pytest

import oracle
from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from .gpu_util import dev_u32, first_label_diff, same_labels

pytestmark = pytest.mark.gpu


def check(d, order=None, **kw):
    ref = oracle.DirectedIndex(d.offsets, d.cols, order=order)
    ix = pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols), order=None if order is None else dev_u32(order), **kw)
    for a, b in ((ix.labels_in(), ref.labels_in()), (ix.labels_out(), ref.labels_out())):
        assert same_labels(a, b), first_label_diff(a, b, d.n)
    s, t = gg.pairs(d.n, 20_000, 5)
    assert np.array_equal(ix.query(dev_u32(s), dev_u32(t)).cpu().numpy(), ref.query_batch(s, t))


@pytest.mark.parametrize("caps", [(256, 64, 256, 64), (256, 0, 0, 0), (0, 64, 0, 0), (0, 0, 256, 0), (0, 0, 0, 64)])
@pytest.mark.parametrize("make,root_batch", [
    (lambda: gg.oriented(gg.ba(3000, 4, 1), 3, both=0.3), 0),
    (lambda: gg.oriented(gg.rmat(11, 16, seed=3), 5, both=0.5), 0),
    (lambda: gg.oriented(gg.rmat(11, 16, seed=3), 5, both=0.5), 500),
    (lambda: gg.oriented(gg.ws(1500, 6, 0.1, 5), 7, both=1.0), 0),
], ids=["ba", "rmat", "rmat500", "ws"])
def test_small_capacities(make, root_batch, caps):
    """The first 64 roots alone leave more than 64 tuples, and their candidates, labels and tables more
    than 256, 256 and 64 entries: every one of these limits is passed."""
    lib = pll.load()
    lib.pll_test_capacities(*caps)
    try:
        check(make(), root_batch=root_batch)
    finally:
        lib.pll_test_capacities(0, 0, 0, 0)


def chain_with_a_sink(n):
    """64 sinks of the lowest ranks and a chain of n vertices with arcs to the first of them from its
    first vertex and its last. Batch after batch the sinks' ranks are cut off the lists, so the BFS
    of the chain's start first meets the sink at level n, far past its distance of 1."""
    arcs = [(64 + i, 64 + i + 1) for i in range(n - 1)] + [(64, 0), (64 + n - 1, 0)]
    return gg.digraph(64 + n, arcs, f"sink{n}"), np.arange(64 + n, dtype=np.uint32)


@pytest.mark.parametrize("n", [254, 255])
@pytest.mark.parametrize("root_batch", [0, 64, 100])
def test_a_depth_of_255_that_only_the_cut_lists_show(n, root_batch):
    """With 255 vertices the chain's end is at depth 254 and its arc leads to depth 255, where whole
    lists have met the sink long before: the batch runs again over them and succeeds."""
    check(*chain_with_a_sink(n), root_batch=root_batch)


def test_a_depth_of_255_over_whole_lists_is_an_error():
    d, order = chain_with_a_sink(256)
    with pytest.raises(pll.PLLError) as e:
        pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols), order=dev_u32(order))
    assert e.value.code == pll.PLL_E_RANGE
