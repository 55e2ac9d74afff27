"""Distance queries where the query kernel changes its way, against the oracle:
ends that nothing reaches, labels longer than the reading of near entries covers,
more near entries than fit (few bit-parallel roots leave a loose bound), pairs
whose distance one end's label holds directly, and every launch size class."""
import numpy as np
import pytest

import oracle
from paper_1304_4661_gb300 import graphgen as gg

from . import graphs
from .gpu_util import gpu_build, gpu_query

pytestmark = pytest.mark.gpu


def cases():
    lone = graphs.disjoint(gg.rmat(11, 4, seed=3), graphs.path(2), graphs.star(4), graphs.complete(1),
                           graphs.complete(1), gg.ba(300, 2, 1))
    return [(lone, 0), (lone, 1), (lone, 64),
            (gg.ws(4000, 6, 0.1, 5), 1), (gg.ws(4000, 6, 0.1, 5), 16),  # labels of hundreds of entries
            (gg.rmat(13, 16, seed=2), 1), (gg.rmat(13, 16, seed=2), 4), (gg.rmat(13, 16, seed=2), 64),
            (graphs.star(3000), 1), (graphs.grid(40, 40), 2), (graphs.path(250), 33)]


@pytest.mark.parametrize("i", range(len(cases())))
def test_distances(i):
    g, t = cases()[i]
    ix, ref = gpu_build(g, t), oracle.Index(g.offsets, g.cols, t)
    for q, seed in ((1, 1), (1217, 2), (4864, 3), (4865, 4), (20_000, 5), (300_001, 6)):
        s, u = gg.pairs(g.n, q, seed)
        got = gpu_query(ix, s, u)
        want = ref.query_batch(s, u)
        assert np.array_equal(got, want), (q, np.flatnonzero(got != want)[:5])
    # every pair of neighbours, both ways round
    rows = np.repeat(np.arange(g.n, dtype=np.uint32), np.diff(g.offsets.astype(np.int64)))
    assert (gpu_query(ix, rows, g.cols) == 1).all() and (gpu_query(ix, g.cols, rows) == 1).all()


def test_long_labels_of_an_arbitrary_order():
    g = gg.ws(3000, 8, 0.3, 9)
    order = np.argsort(gg.uniform(3, g.n)).astype(np.uint32)
    for t in (0, 1, 8):
        ix, ref = gpu_build(g, t, order=order), oracle.Index(g.offsets, g.cols, t, order=order)
        s, u = gg.pairs(g.n, 100_000, 7)
        assert np.array_equal(gpu_query(ix, s, u), ref.query_batch(s, u))
