"""Stencil search (rbf_build_stencils, rbf_build_stencils_static) against the
brute-force oracle where its ranking can go wrong: odd and even candidate
counts, more than 192 candidates (several ranking groups), exact ties, equal
high words of unequal distances, windows that grow or wrap, one row or column
of cells, and centres whose candidates exceed the ranked kernel's space and
fall to the general kernel.  Indices are whole numbers: they are equal."""
import numpy as np
import pytest

from oracle import stencils

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import rbffd  # noqa: E402


def _static(x, z, n_centers, n, period):
    X, Z = (torch.as_tensor(v, dtype=torch.float64, device="cuda") for v in (x, z))
    idx = torch.empty((n_centers, n), dtype=torch.int32, device="cuda")
    rbffd._check(rbffd.lib().rbf_build_stencils_static(rbffd._ptr(X), rbffd._ptr(Z), X.numel(), n_centers, n, period,
                                                       rbffd._ptr(idx), rbffd._stream()))
    return idx.cpu().numpy()


def _points(kind, seed=3):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        return rng.uniform(0, 3, 3001), rng.uniform(0, 1, 3001), 0.0
    if kind == "periodic":
        return rng.uniform(0, 3, 2048), rng.uniform(0, 1, 2048), 3.0
    if kind == "lattice":            # exact ties in every stencil
        X, Z = np.meshgrid(np.arange(53) * 0.25, np.arange(41) * 0.25)
        return X.ravel(), Z.ravel(), 0.0
    if kind == "near-ties":          # distances that differ only in their low words
        X, Z = np.meshgrid(np.arange(45.0), np.arange(37.0))
        e = 1e-9 * rng.uniform(-1, 1, (2, X.size))
        return X.ravel() + e[0], Z.ravel() + e[1], 0.0
    if kind == "line":
        return rng.uniform(0, 1, 700), np.zeros(700), 0.0
    if kind == "column":
        return np.zeros(700), rng.uniform(0, 1, 700), 0.0
    # a dense cluster in a sparse field: hundreds of candidates in a small window
    x = np.concatenate([rng.uniform(0, 1, 2000), 0.5 + 0.012 * rng.standard_normal(900)])
    z = np.concatenate([rng.uniform(0, 1, 2000), 0.5 + 0.012 * rng.standard_normal(900)])
    return x, z, 0.0


@pytest.mark.parametrize("kind", ["uniform", "periodic", "lattice", "near-ties", "line", "column", "cluster"])
@pytest.mark.parametrize("n", [1, 2, 21, 37, 56, 75, 128])
def test_search_equals_brute_force(kind, n):
    x, z, period = _points(kind)
    count = x.size - 7
    ref = stencils.knn(x, z, np.arange(count), n, period)
    got = rbffd.build_stencils(torch.as_tensor(x), torch.as_tensor(z), count, n, period).cpu().numpy()
    assert np.array_equal(got, ref)
    assert np.array_equal(_static(x, z, count, n, period), ref)


def test_fewest_nodes():
    rng = np.random.default_rng(5)
    for n in (1, 5, 33):
        x, z = rng.uniform(0, 1, n), rng.uniform(0, 1, n)
        got = rbffd.build_stencils(torch.as_tensor(x), torch.as_tensor(z), n, n).cpu().numpy()
        assert np.array_equal(got, stencils.knn(x, z, np.arange(n), n))
