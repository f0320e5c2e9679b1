"""The training kernel at the edges of its tiles: batches around one, two and
many blocks of 31 samples, the narrowest and the widest input layer, a single
sample.  Loss and gradient against the oracle in FP64 on the same FP32 states
and BF16 weights, and training bit for bit repeatable.

Tolerance: the gradient is a chain of FP32 sums of at most n_in + 64 + 64 + 31
products per block and one term per block after it, so its rounding is below
(240 + 159 + blocks) 2^-24 = 2.6e-5 of the sums of magnitudes; 1e-4 leaves a
factor of four for cancellation in those sums and tanhf.
"""
import numpy as np
import pytest

from oracle import mlp as omlp
from oracle import stencils as ost

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import inputs as inp  # noqa: E402
from paper_1509_02615_gb300 import learned, rbffd  # noqa: E402

R, SNAP = 2, 3


@pytest.fixture(scope="module")
def data():
    nodes = inp.density_current_nodes(800.0)
    rng = np.random.default_rng(4)
    S = rng.standard_normal((R, SNAP, nodes.n_all, 4)).astype(np.float32)
    T = rng.standard_normal((R, SNAP - 1, nodes.n_prog, 4)).astype(np.float32)
    return nodes, S, T


def _network(nodes, n, l):
    coarse = rbffd.ns_problem(nodes, precision=32, n=n, l=l, threads_per_node=2)
    mlp = rbffd.Mlp(coarse)
    n_in = 4 * (n - 1) + 4
    params = learned.init_params(n_in, seed=3)
    params += (0.05 * np.random.default_rng(8).standard_normal(params.shape)).astype(np.float32)
    mlp.set_params(params)
    scales = np.array([2.0, 1.5, 0.5, 3.0, 1.1, 0.9, 0.7, 1.3, 4.0, 3.0, 6.0, 2.0], np.float32)
    mlp.set_scales(scales)
    return coarse, mlp, n_in, params, scales


@pytest.mark.parametrize("n,l", [(15, 2), (37, 4), (60, 5)])
@pytest.mark.parametrize("batch", [1, 30, 31, 32, 62, 63, 500])
def test_gradient_at_block_edges(data, n, l, batch):
    nodes, S, T = data
    coarse, mlp, n_in, params, scales = _network(nodes, n, l)
    rng = np.random.default_rng(batch)
    ks, ii = rng.integers(0, R * (SNAP - 1), batch), rng.integers(0, nodes.n_prog, batch)
    samples = torch.as_tensor(np.stack([ks, ii], 1), dtype=torch.int64, device="cuda").contiguous()
    loss, g = mlp.grad(torch.as_tensor(S, device="cuda"), torch.as_tensor(T, device="cuda"), R, SNAP, samples)
    w = omlp.bf16_round(params)
    for o, cnt in ((n_in * 64, 64), (n_in * 64 + 64 + 4096, 64), (len(params) - 4, 4)):
        w[o:o + cnt] = params[o:o + cnt]
    idx = ost.knn(nodes.x, nodes.z, np.arange(nodes.n_prog), n, nodes.period_x)
    sc = scales.astype(np.float64)
    X, Y = np.zeros((batch, n_in)), np.zeros((batch, 4))
    for b in range(batch):
        U = S[ks[b] // (SNAP - 1), ks[b] % (SNAP - 1)].astype(np.float64).T
        X[b] = omlp.features(U, idx, np.array([ii[b]]), sc[:4], sc[8:])[0]
        Y[b] = T.reshape(-1, nodes.n_prog, 4)[ks[b], ii[b]] / sc[4:8]
    L, ref = omlp.loss_and_grad(X, Y, w, n_in, 64)
    err = np.linalg.norm(g - ref) / np.linalg.norm(ref)
    print(f"n={n} batch={batch}: loss {loss:.7g} {L:.7g}, gradient off by {err:.2e}")
    assert abs(loss - L) <= 1e-4 * L
    assert err < 1e-4
    assert np.all(g[-4:] == 0.0)   # f(x) - f(0) does not depend on the output bias
    mlp.close()
    coarse.close()


def test_training_repeats_bit_for_bit(data):
    nodes, S, T = data
    St, Tt = torch.as_tensor(S, device="cuda"), torch.as_tensor(T, device="cuda")
    out = []
    for _ in range(2):
        coarse, mlp, _, params, _ = _network(nodes, 37, 4)
        loss = mlp.train(St, Tt, R, SNAP, 20, batch=333, seed=5)
        out.append((loss, mlp.params()))
        assert not np.array_equal(mlp.params(), params)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert np.all(out[0][1][-4:] == params[-4:])
