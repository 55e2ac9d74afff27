"""Errors among the pairs of a call: counted exactly by the asynchronous call in
every launch size class, and cheap for the synchronous ones, whose kernels add to
host memory."""
import time

import numpy as np
import pytest

import oracle
from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from . import graphs
from .gpu_util import dev_u32, gpu_build
from .test_oracle_pins import centroid_order

pytestmark = pytest.mark.gpu


def mixed(n, q, seed):
    """Pairs of a path of n vertices, some with an id out of range: (s, t, bad, too far)."""
    s, t = gg.pairs(n, q, seed)
    s, t = s.astype(np.int64), t.astype(np.int64)
    bad = np.arange(q) % 7 == 3
    s[bad & (np.arange(q) % 2 == 0)] += n
    t[bad & (np.arange(q) % 2 == 1)] = 0xffffffff
    return s.astype(np.uint32), t.astype(np.uint32), bad, ~bad & (np.abs(s - t) >= 255)


@pytest.mark.parametrize("q", [1, 5, 1217, 4864, 4865, 9727, 100_003, 400_001])
@pytest.mark.parametrize("t", [0, 1])
def test_counts(q, t):
    import torch
    g = graphs.path(400)
    ix = gpu_build(g, t, order=centroid_order(g), root_batch=1)
    s, u, bad, far = mixed(g.n, q, q)
    out = torch.empty(q, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        ix.query_async(dev_u32(s), dev_u32(u), out)
        got = out.cpu().numpy()
        assert ix.query_errors() == int(bad.sum() + far.sum())
        assert (got[bad | far] == 255).all()
        ok = ~bad & ~far
        assert np.array_equal(got[ok], np.abs(s[ok].astype(np.int64) - u[ok].astype(np.int64)))

    def status(a, b):
        try:
            ix.query(dev_u32(a), dev_u32(b))
        except pll.PLLError as e:
            return e.code
        return pll.PLL_OK
    for keep, want in ((~bad & ~far, pll.PLL_OK), (~bad, pll.PLL_E_RANGE if far.any() else pll.PLL_OK),
                       (bad | True, pll.PLL_E_INVAL if bad.any() else None)):
        if want is not None and keep.any():
            assert status(s[keep], u[keep]) == want
    assert ix.query_errors() == 0  # the synchronous calls count for themselves


@pytest.mark.parametrize("kind", ["query", "dquery", "paths"])
def test_many_errors_are_cheap(kind):
    """4M pairs, every id out of range, against pairs of a vertex with itself: neither looks at a label.
    With a system-wide addition for each pair 20 to 230 times as slow, a few times with one a warp."""
    import torch
    g = gg.ba(2000, 3, 1)
    off, col = dev_u32(g.offsets), dev_u32(g.cols)
    ix = gpu_build(g, 16)
    same = torch.randint(g.n, (4_000_000,), device="cuda", dtype=torch.int32)
    paths = pll.Paths(ix, off, col)
    room = torch.arange(len(same) + 1, device="cuda")
    call = {"query": lambda x: ix.query(x, x), "dquery": lambda x: directed.query(x, x),
            "paths": lambda x: paths.query(x, x, room, len(same))}[kind]
    directed = pll.DirectedIndex(off, col)

    def least(x, code):
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0, got = time.perf_counter(), pll.PLL_OK
            try:
                call(x)
            except pll.PLLError as e:
                got = e.code
            best = min(best, time.perf_counter() - t0)
            assert got == code
        return best
    assert least(same + g.n, pll.PLL_E_INVAL) < 10 * least(same, pll.PLL_OK)


def test_directed_counts():
    d = gg.oriented(gg.ba(2000, 3, 1), 3, both=0.3)
    ix, ref = pll.DirectedIndex(dev_u32(d.offsets), dev_u32(d.cols)), oracle.DirectedIndex(d.offsets, d.cols)
    s, t = gg.pairs(d.n, 50_001, 4)
    assert np.array_equal(ix.query(dev_u32(s), dev_u32(t)).cpu().numpy(), ref.query_batch(s, t))
    for at in (0, 31, 50_000):
        x = s.copy()
        x[at] = d.n
        with pytest.raises(pll.PLLError) as e:
            ix.query(dev_u32(x), dev_u32(t))
        assert e.value.code == pll.PLL_E_INVAL
