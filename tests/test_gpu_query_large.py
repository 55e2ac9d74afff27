"""Distance queries on indices whose labels are past twice the L2, where only near
label entries are read: against plain breadth-first searches, over every launch
size class, with weak bounds (few roots) and strong ones, and with more near
entries than are kept."""
import numpy as np
import pytest

from paper_1304_4661_gb300 import graphgen as gg

from .gpu_util import dev_u32, gpu_build

pytestmark = pytest.mark.gpu


def distances(src, col, n, root):
    """Distances from root over the arcs (src, col): level by level, 255 if unreachable."""
    import torch
    d = torch.full((n,), 255, dtype=torch.uint8, device="cuda")
    d[root] = 0
    front = torch.zeros(n, dtype=torch.bool, device="cuda")
    front[root] = True
    for level in range(1, 255):
        seen = torch.zeros(n, dtype=torch.bool, device="cuda")
        seen[col[front[src]]] = True
        front = seen & (d == 255)
        if not bool(front.any()):
            break
        d[front] = level
    return d


@pytest.mark.parametrize("make,t", [(lambda: gg.rmat(20, 16, seed=5), 64), (lambda: gg.rmat(19, 16, seed=6), 1),
                                    (lambda: gg.ba(300_001, 4, 3), 16)], ids=["rmat20", "rmat19-one-root", "ba"])
def test_against_searches(make, t):
    import torch
    g = make()
    ix = gpu_build(g, t)
    assert 4 * ix.label_entries() > 2 * torch.cuda.get_device_properties(0).L2_cache_size
    deg = np.diff(g.offsets.astype(np.int64))
    src = torch.repeat_interleave(torch.arange(g.n, device="cuda"), torch.from_numpy(deg).cuda())
    col = dev_u32(g.cols).long()
    by_degree = np.argsort(deg, kind="stable")
    roots = [int(by_degree[-1]), int(by_degree[-1000]), int(by_degree[np.searchsorted(deg[by_degree], 1)]), int(by_degree[0]), g.n // 3, g.n - 1]
    rng = torch.Generator(device="cuda").manual_seed(1)
    for i, r in enumerate(roots):
        want = distances(src, col, g.n, r)
        v = torch.randperm(g.n, generator=rng, device="cuda").to(torch.int32)
        s = torch.full_like(v, r)
        for q in (g.n, 4865, 30_001, 150_001):
            a, b = (s[:q], v[:q]) if i % 2 else (v[:q], s[:q])
            got = ix.query(a.contiguous(), b.contiguous())
            assert torch.equal(got, want[v[:q].long()]), (r, q)
