"""Memory that a build can do without: every allocation of a build is made to fail
in turn. Those that only save time must not fail the build, and whatever the
build then goes without, its labels are the same."""
import gc

import numpy as np
import pytest

import oracle
from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from . import graphs
from .gpu_util import dev_u32, same_labels

pytestmark = pytest.mark.gpu

OK, NOMEM = pll.PLL_OK, pll.PLL_E_NOMEM


def allocations(build):
    """How many allocations the build makes: with a countdown of just that many it succeeds, and the
    next call's first one fails."""
    lib, empty = pll.load(), gg.from_edges(1, [], [])
    for k in range(400):
        lib.pll_test_fail_alloc(k)
        try:
            build().close()
        except pll.PLLError:
            continue
        try:
            undirected(empty, 0)[0]().close()
        except pll.PLLError:
            return k
        finally:
            lib.pll_test_fail_alloc(-1)
    pytest.fail("the build never completed")


def outcomes(build, labels):
    """The status of the build with its k-th allocation failing, for each of them."""
    lib = pll.load()
    ix = build()
    want = labels(ix)
    ix.close()
    gc.collect()
    base, codes = lib.pll_test_live_allocs(), []
    for k in range(allocations(build)):
        lib.pll_test_fail_alloc(k)
        try:
            ix = build()
        except pll.PLLError as e:
            codes.append(e.code)
        else:
            codes.append(OK)
            lib.pll_test_fail_alloc(-1)
            assert all(same_labels(a, b) for a, b in zip(labels(ix), want)), k
            ix.close()
        finally:
            lib.pll_test_fail_alloc(-1)
        assert lib.pll_test_live_allocs() == base, k
    assert set(codes) == {OK, NOMEM} and codes.count(NOMEM) > 10
    return codes


def undirected(g, t, **kw):
    off, col = dev_u32(g.offsets), dev_u32(g.cols)
    return lambda: pll.Index.build(off, col, t=t, **kw), lambda ix: [ix.labels()]


def directed(g, **kw):
    off, col = dev_u32(g.offsets), dev_u32(g.cols)
    return lambda: pll.DirectedIndex(off, col, **kw), lambda ix: [ix.labels_in(), ix.labels_out()]


@pytest.mark.parametrize("make", [lambda: undirected(gg.ba(20000, 6, 7), 0), lambda: undirected(gg.ba(20000, 6, 7), 0, root_batch=500),
                                  lambda: directed(gg.oriented(gg.ba(20000, 6, 7), 3, both=0.3))],
                         ids=["default", "batches-of-500", "directed"])
def test_a_store_without_its_near_copy(make):
    """Over 2M entries: the near copy is rebuilt several times, and each of its allocations may fail."""
    codes = outcomes(*make())
    assert codes.count(OK) >= 3


def test_buffers_grown_ahead_of_demand():
    """Every root of the first batch labels every vertex (3.84M tuples, all but 120,000 dropped again);
    the tuple buffers are grown for the second, which would have fitted."""
    codes = outcomes(*undirected(graphs.star(60000), 0))
    assert codes.count(OK) >= 4  # the tuples, sorted, their marks, the sort's space


@pytest.mark.parametrize("make,after", [(lambda: undirected(gg.ba(20000, 6, 7), 0), 1),
                                        (lambda: directed(gg.oriented(gg.ba(20000, 6, 7), 3, both=0.3)), 0)],
                         ids=["undirected", "directed"])
def test_the_near_copy_makes_room_for_what_the_build_needs(make, after):
    """The index's label arrays (and the sizes of their compaction) are the build's last allocations but
    `after`: one of them failing costs the near copy, not the build."""
    codes = outcomes(*make())
    assert codes[len(codes) - after - 3:len(codes) - after] == [OK, OK, OK]


def test_a_small_graph_needs_little_scratch():
    """2000 vertices: the least candidate, tuple and label buffers are 0.55 GB, and nothing else that a
    build holds has a fixed size of more than a few MB."""
    g = gg.ba(2000, 3, 1)
    with_roots = undirected(g, 16)[0]()
    assert 0 < with_roots.stats()["scratch_peak_bytes"] < 0.8e9
    with_roots.close()


@pytest.mark.parametrize("root_batch", [8, 13])
def test_an_older_near_copy_beside_a_store_that_moved(root_batch):
    """Label pools that start small (a batch of few roots asks for little more) move to larger ones
    between rebuilds of the near copy, which then covers the labels as they were."""
    lib, g = pll.load(), gg.ba(20000, 6, 7)
    d = gg.oriented(g, 3, both=0.3)
    lib.pll_test_capacities(0, 0, 1 << 18, 0)
    try:
        ix = undirected(g, 0, root_batch=root_batch)[0]()
        dix = directed(d, root_batch=root_batch)[0]()
    finally:
        lib.pll_test_capacities(0, 0, 0, 0)
    assert ix.stats()["pool_regrows"] > 1
    assert same_labels(ix.labels(), oracle.Index(g.offsets, g.cols, 0).labels())
    ref = oracle.DirectedIndex(d.offsets, d.cols)
    assert same_labels(dix.labels_in(), ref.labels_in()) and same_labels(dix.labels_out(), ref.labels_out())
