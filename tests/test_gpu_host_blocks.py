"""The pinned words in which synchronous calls learn their status: a call that
ends early leaves nothing behind that a later call could take for its own, threads
that come and go leave no pinned memory, and calls of many threads at once keep
their statuses apart."""
import gc
import subprocess
import sys
import threading
from pathlib import Path

import numpy as np
import pytest

from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from .gpu_util import dev_u32, gpu_build

pytestmark = pytest.mark.gpu
ROOT = Path(__file__).resolve().parents[1]


def test_an_early_end_leaves_no_status_to_the_next_call():
    """A path-offset call whose scratch cannot be had returns while its pairs (every id out of range)
    are still being answered; a good query on another stream must not see their errors."""
    import torch
    g = gg.ba(2000, 3, 1)
    ix = gpu_build(g, 16)
    paths = pll.Paths(ix, dev_u32(g.offsets), dev_u32(g.cols))
    q = 20_000_000
    bad = torch.full((q,), g.n + 7, dtype=torch.int32, device="cuda")
    one = dev_u32(np.array([5], np.uint32))
    other = torch.cuda.Stream()
    lib = pll.load()
    torch.cuda.synchronize()
    codes = []
    for k in range(4):
        lib.pll_test_fail_alloc(k)
        try:
            with pytest.raises(pll.PLLError) as e:
                paths.offsets(bad, bad)
        finally:
            lib.pll_test_fail_alloc(-1)
        codes.append(e.value.code)
        assert int(ix.query(one, one, stream=other).cpu()[0]) == 0, k  # raises on a status of another call
        torch.cuda.synchronize()
    assert pll.PLL_E_NOMEM in codes and codes[-1] == pll.PLL_E_INVAL


THREADS = """
import sys, threading
import numpy as np, torch
from paper_1304_4661_gb300 import graphgen as gg, pll

def resident_kb():
    with open("/proc/self/status") as f:
        return next(int(line.split()[1]) for line in f if line.startswith("VmRSS:"))

net = pll.MLP(64)
net.set_params(gg.mlp_init(3))
want, _ = net.grad(torch.ones(64, 8, device="cuda"), torch.zeros(64, device="cuda"))
got, lib = np.empty_like(want), pll.load()

def run(count):
    for _ in range(count):
        th = threading.Thread(target=lib.pll_mlp_read_grad, args=(net._h, got.ctypes.data, None, None))
        th.start()
        th.join()

run(50)  # thread stacks and the allocator's arenas
before = resident_kb()
run(2000)
assert np.array_equal(got, want)
print(resident_kb() - before)
"""


def test_threads_leave_no_pinned_memory():
    """2000 threads, one after another, each read a gradient (a copy of 19 KB to pinned memory): 38 MB
    if each left its buffer behind. In a process of its own, where nothing else comes or goes."""
    r = subprocess.run([sys.executable, "-c", THREADS], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert int(r.stdout) < 10 << 10


def test_many_threads_keep_their_statuses_apart():
    """More threads at once than blocks are kept; every third one asks for an id out of range."""
    import torch
    g = gg.ba(500, 3, 2)
    ix = gpu_build(g, 8)
    lib = pll.load()
    gc.collect()  # indices of earlier tests must not be freed mid-count
    live = lib.pll_test_live_allocs()
    good, bad = dev_u32(np.arange(500, dtype=np.uint32)), dev_u32(np.full(500, 500, np.uint32))
    wrong, gate = [], threading.Barrier(100)

    def work(i):
        stream, out = torch.cuda.Stream(), torch.empty(500, dtype=torch.uint8, device="cuda")
        gate.wait()
        for _ in range(20):
            code = pll.PLL_OK
            try:
                ix.query(bad if i % 3 == 0 else good, good, out=out, stream=stream)
            except pll.PLLError as e:
                code = e.code
            if code != (pll.PLL_E_INVAL if i % 3 == 0 else pll.PLL_OK):
                wrong.append((i, code))
    threads = [threading.Thread(target=work, args=(i,)) for i in range(100)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not wrong
    assert lib.pll_test_live_allocs() == live
    pll.release_cached()
    assert int(ix.query(good[:1], good[:1]).cpu()[0]) == 0


def test_calls_without_a_block_of_host_memory():
    """The first allocation of each call, its block, fails: the status comes back from device words."""
    g = gg.ba(3000, 3, 4)
    ix = gpu_build(g, 16)
    off, col = dev_u32(g.offsets), dev_u32(g.cols)
    paths, dix = pll.Paths(ix, off, col), pll.DirectedIndex(off, col)
    net = pll.MLP(64)
    net.set_params(gg.mlp_init(3))
    x, t = dev_u32(np.ones((64, 8))).float(), dev_u32(np.zeros(64)).float()
    s, d = (dev_u32(a) for a in gg.pairs(g.n, 5000, 9))
    bad = dev_u32(np.full(5000, g.n, np.uint32))
    room = paths.offsets(s, d)[0]
    lib = pll.load()

    def without(call, *args):
        lib.pll_test_fail_alloc(0)
        try:
            r = call(*args)
        except pll.PLLError as e:
            return e.code
        finally:
            lib.pll_test_fail_alloc(-1)
        r = r if isinstance(r, tuple) else (r,)
        return [a.cpu().numpy().tolist() if hasattr(a, "cpu") else np.asarray(a).tolist() for a in r]

    for call, good, wrong in ((ix.query, (s, d), (bad, d)), (dix.query, (s, d), (s, bad)),
                              (paths.offsets, (s, d), (bad, d)), (paths.query, (s, d, room), (s, bad, room)),
                              (net.grad, (x, t), None)):
        want = call(*good)
        want = want if isinstance(want, tuple) else (want,)
        want = [a.cpu().numpy().tolist() if hasattr(a, "cpu") else np.asarray(a).tolist() for a in want]
        for _ in range(2):
            if wrong:
                assert without(call, *wrong) == pll.PLL_E_INVAL
            assert without(call, *good) == want
