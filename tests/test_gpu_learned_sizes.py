"""The learned order's kernels at the sizes where their paths change, against the
oracle: lists around the length that gets a block of its own in the core-number
steps, chains that take many steps, rows around a block's tile and the switch to
two rows a thread, unaligned inputs, and minibatches around the gradient's tile.

Tolerances as in test_gpu_learned.py: scores within 1e-5 of their scale, gradients
within 1e-4 of the largest entry plus 1e-4 relative; core numbers are exact."""
import numpy as np
import pytest

from oracle import learned as OL
from paper_1304_4661_gb300 import graphgen as gg
from paper_1304_4661_gb300 import pll

from . import graphs
from .gpu_util import dev_u32
from .test_gpu_learned import random_params

pytestmark = pytest.mark.gpu


def wheel_of_stars(degrees):
    """Hubs of the given degrees over shared leaves, the hubs a clique, the leaves a cycle."""
    k, leaves = len(degrees), max(degrees) + 3
    e = [(i, j) for i in range(k) for j in range(i)]
    e += [(h, k + (31 * h + i) % leaves) for h, d in enumerate(degrees) for i in range(d)]
    e += [(k + i, k + (i + 1) % leaves) for i in range(leaves)]
    e = np.asarray(e)
    return gg.from_edges(k + leaves, e[:, 0], e[:, 1], f"stars{degrees}")


@pytest.mark.parametrize("g", [
    graphs.star(511), graphs.star(513), graphs.complete(540), graphs.path(200), graphs.grid(2, 150),
    wheel_of_stars([500, 511, 512, 513, 700, 1500]), wheel_of_stars([40] * 30 + [2000] * 5),
    gg.ba(3000, 40, 3), graphs.disjoint(graphs.complete(600), graphs.path(70), graphs.star(900)),
], ids=lambda g: f"{g.name}-{g.n}")
def test_core_numbers(g):
    _, core, _ = pll.features(dev_u32(g.offsets), dev_u32(g.cols), 0, raw=True)
    _, _, ref, _ = OL.raw_features(g.offsets, g.cols, 0)
    assert np.array_equal(core.cpu().numpy().astype(np.int64), ref)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 255, 1000, 152 * 3 * 256 - 1, 152 * 3 * 256, 152 * 3 * 256 + 1, 300_007])
@pytest.mark.parametrize("shift", [0, 1])
def test_scores(n, shift):
    import torch
    p = random_params(7)
    mlp = pll.MLP(max_batch=1)
    mlp.set_params(p)
    X = np.random.default_rng(n).standard_normal((n, 8)).astype(np.float32)
    flat = torch.zeros(8 * n + 4, dtype=torch.float32, device="cuda")
    x = flat[shift:shift + 8 * n].view(n, 8)  # shift 1: rows not on 16 bytes
    x.copy_(torch.from_numpy(X))
    y = mlp.forward(x).cpu().numpy()
    yr, _ = OL.forward(p, X)
    assert np.max(np.abs(y - yr)) <= 1e-5 * max(1.0, np.abs(yr).max())


@pytest.mark.parametrize("batch", [1, 63, 64, 65, 511, 512, 513, 4000])
@pytest.mark.parametrize("shift", [0, 1])
def test_gradients(batch, shift):
    import torch
    p = random_params(9)
    rng = np.random.default_rng(batch)
    X = rng.standard_normal((4096, 8)).astype(np.float32)
    T = rng.standard_normal(4096).astype(np.float32)
    idx = rng.integers(0, 4096, batch).astype(np.int32)
    mlp = pll.MLP(max_batch=batch)
    mlp.set_params(p)
    flat = torch.zeros(X.size + 4, dtype=torch.float32, device="cuda")
    x = flat[shift:shift + X.size].view(-1, 8)
    x.copy_(torch.from_numpy(X))
    got, loss = mlp.grad(x, torch.from_numpy(T).cuda(), idx=torch.from_numpy(idx).cuda())
    ref_loss, ref = OL.loss_grad(p, X[idx].astype(np.float64), T[idx].astype(np.float64))
    assert np.all(np.abs(got - ref) <= 1e-4 * np.abs(ref).max() + 1e-4 * np.abs(ref))
    assert abs(loss - ref_loss) <= 1e-4 * max(1.0, ref_loss)
    again, _ = mlp.grad(x, torch.from_numpy(T).cuda(), idx=torch.from_numpy(idx).cuda())
    assert np.array_equal(got, again)
