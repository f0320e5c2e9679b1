"""Training batches of more tiles than the launch has blocks: the memory of the
per-block partials does not grow with the batch, and a batch that repeats its
samples has the loss and gradient of the samples once.

Tolerance: both sides are chains of FP32 sums over the same products, the long
one with three or four tiles more per block and up to 608 blocks, below
(240 + 159 + 608) 2^-24 = 6e-5 of the sums of magnitudes; 1e-4 as at the block
edges (tests/test_gpu_train_tiles.py).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import inputs as inp  # noqa: E402
from paper_1509_02615_gb300 import learned, rbffd  # noqa: E402

R, SNAP = 2, 3


@pytest.fixture(scope="module")
def network():
    nodes = inp.density_current_nodes(800.0)
    rng = np.random.default_rng(4)
    S = torch.as_tensor(rng.standard_normal((R, SNAP, nodes.n_all, 4)), dtype=torch.float32, device="cuda")
    T = torch.as_tensor(rng.standard_normal((R, SNAP - 1, nodes.n_prog, 4)), dtype=torch.float32, device="cuda")
    coarse = rbffd.ns_problem(nodes, precision=32, threads_per_node=2)
    mlp = rbffd.Mlp(coarse)
    params = learned.init_params(4 * 37, seed=3)
    mlp.set_params(params + (0.05 * np.random.default_rng(8).standard_normal(params.shape)).astype(np.float32))
    mlp.set_scales(np.array([2.0, 1.5, 0.5, 3.0, 1.1, 0.9, 0.7, 1.3, 4.0, 3.0, 6.0, 2.0], np.float32))
    yield nodes, coarse, mlp, S, T
    mlp.close()
    coarse.close()


def _samples(nodes, batch, seed):
    rng = np.random.default_rng(seed)
    return torch.as_tensor(np.stack([rng.integers(0, R * (SNAP - 1), batch), rng.integers(0, nodes.n_prog, batch)], 1),
                           dtype=torch.int64, device="cuda").contiguous()


@pytest.mark.parametrize("batch,times", [(589, 32), (589, 33), (500, 100)])   # 608 tiles, a few more, three each
def test_repeated_samples(network, batch, times):
    nodes, _, mlp, S, T = network
    once = _samples(nodes, batch, batch)
    L, ref = mlp.grad(S, T, R, SNAP, once)
    loss, g = mlp.grad(S, T, R, SNAP, once.repeat(times, 1).contiguous())
    assert abs(loss - L) <= 1e-4 * L
    assert np.linalg.norm(g - ref) <= 1e-4 * np.linalg.norm(ref)


def test_partials_do_not_grow_with_the_batch(network):
    nodes, coarse, _, S, T = network
    samples = _samples(nodes, 300_000, 1)
    mlp = rbffd.Mlp(coarse)
    mlp.set_params(learned.init_params(4 * 37, seed=3))
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    loss, g = mlp.grad(S, T, R, SNAP, samples)
    used = free - torch.cuda.mem_get_info()[0]
    print(f"300,000 samples: {used / 2 ** 20:.0f} MiB")
    assert np.isfinite(loss) and used < 100 * 2 ** 20
    mlp.close()
