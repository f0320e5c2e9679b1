"""The FP64 stencil sums on the integer units (csrc/fixdot.cuh) where a
stencil's products lie far apart: values that exceed their neighbours 8 to a
million times, among them the node's own value where its weight vanishes;
negative zeros and values at the lower end of the range; infinities; sums whose
products are all alike (the accumulators' range), up to 128 of them.  Against
sums in long double (113 bits on aarch64) of the problem's own weights.

Tolerance.  Every product keeps its bits down to 2^-58 of the sum's largest
product and loses at most 2^-55 of it with the two low halves, so a sum of n
slots is off by less than n 2^-54 max |w f| and one rounding; with the shared
roundings of the epilogue every tendency is compared at
2^-53 (n max |w f| + 8 sum |w f|), summed over its terms: no part of it depends
on a value that a weight does not bring in.  Relative to sum |w f|, the root
mean square over the nodes that read a spike is no larger than that of plain
FP64 sums in slot order.  Results are the same bits for every number of lanes.
"""
import numpy as np
import pytest

from paper_1509_02615_gb300 import inputs as inp
from test_gpu_fixed_point import CASES, LD, _smooth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import rbffd  # noqa: E402


def _rows(pb, mu):
    W = {}
    for op in ("dx", "dz", "lap", "hv"):
        W[op], idx = pb.weights(op)
    g = float(pb.params.gamma_c * pb.params.spacing ** 5)
    return {"x": W["dx"], "z": W["dz"], "d": (LD(g) * W["hv"].astype(LD) + (mu * W["lap"]).astype(LD)).astype(np.float64),
            "h": g * W["hv"]}, idx


def _tendencies(rows, idx, nodes, U, T):
    """Tendencies [4, n_prog] with sums in precision T in slot order; n max |w f| + 8 sum |w f|; sum |w f|."""
    P, n = nodes.n_prog, idx.shape[1]

    def dot(w, f):
        s, a, m = np.zeros(P, T), np.zeros(P), np.zeros(P)
        for k in range(n):
            s = s + w[:, k].astype(T) * U[f, idx[:, k]].astype(T)
            p = np.abs(w[:, k] * U[f, idx[:, k]])
            a, m = a + p, np.maximum(m, p)
        return s, n * m + 8 * a, a

    D = {(o, f): dot(rows["h" if o == "d" and f == 3 else o], f) for f in range(4) for o in "xzd"}
    u, w, th, p = (U[f, :P].astype(T) for f in range(4))
    cpth = T(inp.CP) * (T(inp.THETA_BAR) + th)
    pib = (1.0 - inp.G * nodes.z[:P] / (inp.CP * inp.THETA_BAR)).astype(T) + p
    one = np.ones(P, T)
    coef = [{("x", 0): -u, ("z", 0): -w, ("x", 3): -cpth, ("d", 0): one},
            {("x", 1): -u, ("z", 1): -w, ("z", 3): -cpth, ("d", 1): one},
            {("x", 2): -u, ("z", 2): -w, ("d", 2): one},
            {("x", 3): -u, ("z", 3): -w, ("x", 0): -T(inp.RD / inp.CV) * pib, ("z", 1): -T(inp.RD / inp.CV) * pib,
             ("d", 3): one}]
    extra = [0 * u, T(inp.G / inp.THETA_BAR) * th, 0 * u, -w * T(-inp.G / (inp.CP * inp.THETA_BAR))]
    K = np.stack([sum(c * D[key][0] for key, c in cf.items()) + e for cf, e in zip(coef, extra)])
    M, A = (np.stack([sum(np.abs(c).astype(float) * D[key][q] for key, c in cf.items()) + 8 * np.abs(e).astype(float)
                      for cf, e in zip(coef, extra)]) for q in (1, 2))
    K[1][(nodes.kind == 1) | (nodes.kind == 2)] = 0
    K[0][(nodes.kind == 3) | (nodes.kind == 4)] = 0
    return K, M, A


def _rhs(pb, U):
    t = rbffd.state_tensor(U, 64)
    got = rbffd.fields(pb.rhs(0.0, t))
    return got, rbffd.fields(t)   # with the ghosts the call filled


@pytest.mark.parametrize("case,k,lanes", [("hex37", 8.0, 1), ("hex37", 64.0, 2), ("hex37", 1e6, 1), ("walls31", 1e3, 4),
                                          ("walls31", 1e6, 1), ("bubble56", 64.0, 1), ("bubble56", 1e6, 8)])
def test_spikes_cost_their_neighbours_nothing(case, k, lanes):
    nodes, prm = CASES[case]()
    pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
    rng = np.random.default_rng(5)
    U = _smooth(nodes, rng)
    at = rng.choice(nodes.n_prog, nodes.n_prog // 40, replace=False)
    U[:, at] *= k
    got, Uf = _rhs(pb, U)
    rows, idx = _rows(pb, prm["mu"])
    ref, M, A = _tendencies(rows, idx, nodes, Uf, LD)
    plain, _, _ = _tendencies(rows, idx, nodes, Uf, np.float64)
    e, b = np.abs(got.astype(LD) - ref).astype(float), np.abs(plain.astype(LD) - ref).astype(float)
    print(f"{case} k={k:g}: error / bound up to {(e / (2.0 ** -53 * M + 1e-300)).max():.3f}")
    assert np.all(e <= 2.0 ** -53 * M)
    near = np.isin(idx, at).any(1) & (A > 0).all(0)
    for f in range(4):
        x, y = (float(np.sqrt(np.mean((v[f, near] / A[f, near]) ** 2))) for v in (e, b))
        print(f"   field {f}: relative to sum |w f| {x:.2e}, plain FP64 {y:.2e}")
        assert x <= y
    pb.close()


@pytest.mark.parametrize("lanes", [1, 4])
def test_low_end_and_negative_zeros(lanes):
    nodes, prm = CASES["hex37"]()
    pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
    rng = np.random.default_rng(6)
    U = _smooth(nodes, rng)
    U[0] = -0.0
    U[1] = -np.abs(U[1]) * 10.0 ** rng.uniform(-320, -280, nodes.n_all)   # through the subnormal numbers to zero
    U[2] = np.where(rng.random(nodes.n_all) < 0.5, -0.0, U[2] * 10.0 ** rng.uniform(-60, 0, nodes.n_all))
    got, Uf = _rhs(pb, U)
    rows, idx = _rows(pb, prm["mu"])
    ref, M, _ = _tendencies(rows, idx, nodes, Uf, LD)
    e = np.abs(got.astype(LD) - ref).astype(float)
    # below the normal range every product rounds at 2^-1074, times the largest coefficient (c_p theta)
    assert np.all(e <= 2.0 ** -53 * M + 4e5 * 37 * 2.0 ** -1074)
    pb.close()


@pytest.mark.parametrize("scale", [1e-283, 1e-290, 1e-300, 1e-308, 1e-320])
def test_whole_fields_at_the_low_end(scale):
    nodes, prm = CASES["walls31"]()
    rng = np.random.default_rng(10)
    U = _smooth(nodes, rng)
    U[1:] *= scale * 10.0 ** rng.uniform(-6, 2, (3, nodes.n_all))   # u stays in the ordinary range
    U[1:][rng.random((3, nodes.n_all)) < 0.2] = 0.0
    out = []
    for lanes in (1, 2):
        pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
        got, Uf = _rhs(pb, U)
        rows, idx = _rows(pb, prm["mu"])
        ref, M, _ = _tendencies(rows, idx, nodes, Uf, LD)
        e = np.abs(got.astype(LD) - ref).astype(float)
        assert np.all(e <= 2.0 ** -53 * M + 4e5 * 31 * 2.0 ** -1074)
        out.append(got)
        pb.close()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("lanes", [1, 2])
def test_infinite_value_gives_what_fp64_gives(lanes):
    nodes, prm = inp.density_current_nodes(400.0), dict(n=37, l=4, mu=75.0)
    pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
    U = _smooth(nodes, np.random.default_rng(7))
    P = nodes.n_prog
    at = int(np.argmin(np.abs(nodes.z[:P] - 3200.0) + np.abs(nodes.x[:P])))   # its readers are off the walls
    U[2, at] = np.inf
    got, Uf = _rhs(pb, U)
    rows, idx = _rows(pb, prm["mu"])
    reads = (idx == at).any(1)
    reads[at] = False   # a slot that pads a row holds the node's own value with weight 0: NaN there
    with np.errstate(invalid="ignore"):
        plain, _, _ = _tendencies(rows, idx, nodes, Uf, np.float64)
    a, b = got[2, reads], plain[2, reads]
    assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isposinf(a), np.isposinf(b))
    assert np.array_equal(np.isneginf(a), np.isneginf(b)) and not np.isfinite(a).any() and np.isinf(a).any()
    pb.close()


@pytest.mark.parametrize("n,l,sign", [(37, 4, 1.0), (75, 5, -1.0), (128, 6, 1.0)])
def test_products_all_alike(n, l, sign):
    nodes = inp.density_current_nodes(300.0)
    pb = rbffd.ns_problem(nodes, precision=64, n=n, l=l, mu=75.0, threads_per_node=1)
    rows, idx = _rows(pb, 75.0)
    P = nodes.n_prog
    full = np.flatnonzero((idx < P).all(1))   # off the walls: no ghosts among the neighbours
    i = int(full[np.argmin(np.abs(nodes.x[full]))])
    U = _smooth(nodes, np.random.default_rng(8))
    for f, o in ((0, "x"), (1, "z"), (2, "d"), (3, "h")):   # a sum of equal products of full mantissas in each field
        w = rows[o][i]
        m, e = np.frexp(w)
        U[f, idx[i]] = np.where(w == 0, 0.0, sign * np.sign(w) * np.ldexp(1 - 2.0 ** -53, -e) * {0: 8.0, 1: 4.0, 2: 1.0, 3: 1e-4}[f])
    U[2] *= 1.0 / np.abs(U[2]).max()
    got, Uf = _rhs(pb, U)
    ref, M, _ = _tendencies(rows, idx, nodes, Uf, LD)
    e = np.abs(got.astype(LD) - ref).astype(float)
    assert np.all(e <= 2.0 ** -53 * M)
    pb.close()


@pytest.mark.parametrize("case", ["hex37", "bubble56"])
def test_lanes_do_not_change_a_bit(case):
    nodes, prm = CASES[case]()
    rng = np.random.default_rng(9)
    U = _smooth(nodes, rng) * 10.0 ** rng.uniform(-12, 0, (4, nodes.n_all))
    out = []
    for lanes in (1, 2, 4, 8):
        pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
        out.append(pb.rhs(0.0, rbffd.state_tensor(U, 64)).clone())
        pb.close()
    assert all(torch.equal(v, out[0]) for v in out[1:])
