"""The fixed-point stencil sums of the FP64 right-hand side (csrc/fixdot.cuh)
against sums in long double (113 bits on aarch64), formed from the problem's
own FP64 weights and the state it filled, over states that exercise the
exponent handling: a developed flow, a compact bubble at rest (exact zeros),
values over eight decades in one stencil, one spike, values near the smallest
and the largest exponents, and non-finite values.

Tolerance.  Weights and values are cut below 2^-55 of the row's and the
stencil's largest and the product of the low halves (below 2^-55 of the
largest product) is dropped, so a sum over n slots is off by at most
3 n 2^-55 max|w| max|f|, plus one rounding; the plain FP64 sum is off by up to
n 2^-53 sum |w f|.  Every field's tendency is compared at
2^-53 (n max|w| max|f| + 8 sum |w f|) summed over its terms, and over the whole
state the fixed-point error is no larger than that of plain FP64 sums in slot
order.  (The spike, a million times its neighbours, is held to the first bound
alone: where a stencil gives it no weight, the others lose bits to it.)
"""
import numpy as np
import pytest

from paper_1509_02615_gb300 import configs
from paper_1509_02615_gb300 import inputs as inp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import rbffd  # noqa: E402

LD = np.longdouble
CASES = {"hex37": lambda: (inp.density_current_nodes(800.0), dict(n=37, l=4, mu=75.0)),
         "walls31": lambda: (inp.rising_bubble_nodes(500.0, "cart"), dict(n=31, l=3, mu=10.0)),
         "bubble56": lambda: (configs.bubble(h=800.0).nodes, dict(configs.BUBBLE_METHOD))}


def _smooth(nodes, rng):
    x = 2 * np.pi * (nodes.x - nodes.x.min()) / (nodes.x.max() - nodes.x.min())
    z = np.pi * nodes.z / nodes.z.max()
    return np.stack([a * np.cos(k * x + p) * np.cos(m * z) for a, k, m, p in
                     zip((8.0, 4.0, 1.5, 1.5e-4), rng.integers(1, 4, 4), rng.integers(1, 3, 4), rng.uniform(0, 6, 4))])


def _state(kind, nodes):
    rng = np.random.default_rng(11)
    if kind == "flow":
        return _smooth(nodes, rng)
    if kind == "rest":
        U = np.zeros((4, nodes.n_all))
        U[2] = np.where(np.hypot(nodes.x - nodes.x.mean(), nodes.z - 3000.0) < 2000.0, -15.0, 0.0)
        return U
    if kind == "decades":
        return rng.choice([-1.0, 1.0], (4, nodes.n_all)) * 10.0 ** rng.uniform(-8, 0, (4, nodes.n_all))
    if kind == "spike":
        U = _smooth(nodes, rng)
        U[:, nodes.n_prog // 2] *= 1e6
        return U
    scale = {"tiny": 1e-250, "large": 1e60}[kind]
    return scale * rng.uniform(-1, 1, (4, nodes.n_all))


def _reference(pb, nodes, U, mu, T):
    """Tendencies [4, n_prog] in precision T (sums in slot order) and, per entry, the tolerance's magnitude."""
    W = {}
    for op in ("dx", "dz", "lap", "hv"):
        W[op], idx = pb.weights(op)
    g = float(pb.params.gamma_c * pb.params.spacing ** 5)
    diss = (LD(g) * W["hv"].astype(LD) + (mu * W["lap"]).astype(LD)).astype(np.float64)   # as packed: two roundings
    hv = g * W["hv"]
    P = nodes.n_prog

    def dot(w, f):
        s, a = np.zeros(P, T), np.zeros(P)
        for k in range(idx.shape[1]):
            s = s + w[:, k].astype(T) * U[f, idx[:, k]].astype(T)
            a += np.abs(w[:, k] * U[f, idx[:, k]])
        return s, idx.shape[1] * np.abs(w).max(1) * np.abs(U[f, idx]).max(1) + 8 * a

    D = {(o, f): dot(w, f) for f in range(4) for o, w in (("x", W["dx"]), ("z", W["dz"]), ("d", hv if f == 3 else diss))}
    u, w, th, p = (U[f, :P].astype(T) for f in range(4))
    z = nodes.z[:P]
    cpth = T(inp.CP) * (T(inp.THETA_BAR) + th)
    pib = (1.0 - inp.G * z / (inp.CP * inp.THETA_BAR)).astype(T) + p
    coef = [{("x", 0): -u, ("z", 0): -w, ("x", 3): -cpth, ("d", 0): T(1)},
            {("x", 1): -u, ("z", 1): -w, ("z", 3): -cpth, ("d", 1): T(1)},
            {("x", 2): -u, ("z", 2): -w, ("d", 2): T(1)},
            {("x", 3): -u, ("z", 3): -w, ("x", 0): -T(inp.RD / inp.CV) * pib, ("z", 1): -T(inp.RD / inp.CV) * pib, ("d", 3): T(1)}]
    extra = [T(0), T(inp.G / inp.THETA_BAR) * th, T(0), -w * T(-inp.G / (inp.CP * inp.THETA_BAR))]
    K = np.stack([sum(c * D[key][0] for key, c in cf.items()) + e for cf, e in zip(coef, extra)])
    M = np.stack([sum(np.abs(c).astype(float) * D[key][1] for key, c in cf.items()) + 8 * np.abs(np.asarray(e, float))
                  for cf, e in zip(coef, extra)])
    kind = nodes.kind
    K[1][(kind == 1) | (kind == 2)] = 0
    K[0][(kind == 3) | (kind == 4)] = 0
    return K, M


@pytest.mark.parametrize("case,state,lanes", [
    ("hex37", "flow", 1), ("hex37", "flow", 2), ("hex37", "rest", 1), ("hex37", "decades", 4), ("hex37", "spike", 1),
    ("walls31", "flow", 8), ("walls31", "decades", 1), ("walls31", "tiny", 2), ("bubble56", "flow", 1),
    ("bubble56", "decades", 2), ("bubble56", "spike", 4), ("bubble56", "rest", 8), ("bubble56", "large", 1)])
def test_sums_are_no_less_exact_than_plain_fp64(case, state, lanes):
    nodes, prm = CASES[case]()
    pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=lanes, **prm)
    U = rbffd.state_tensor(_state(state, nodes), 64)
    got = rbffd.fields(pb.rhs(0.0, U))
    Uf = rbffd.fields(U)   # ghosts as the call filled them
    with np.errstate(over="ignore", invalid="ignore"):
        ref, mag = _reference(pb, nodes, Uf, prm["mu"], LD)
        plain, _ = _reference(pb, nodes, Uf, prm["mu"], np.float64)
    fine = np.isfinite(ref.astype(float)) & np.isfinite(plain)
    e = np.abs(got.astype(LD) - ref).astype(float)
    assert np.all(e[fine] <= (2.0 ** -53 * mag)[fine])
    for f in range(4):
        a, b, n = (float(np.sqrt(np.mean(v[fine[f]] ** 2))) for v in (e[f].astype(LD), plain[f].astype(LD) - ref[f], ref[f]))
        print(f"{case} {state} G={lanes} field {f}: fixed point {a / max(n, 1e-300):.2e}, plain FP64 {b / max(n, 1e-300):.2e}")
        assert state == "spike" or a <= b * 1.05 + 1e-300   # 5%: the shared roundings of the epilogue are in both
    pb.close()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_values_stay_in_their_stencils(bad):
    nodes, prm = inp.density_current_nodes(400.0), dict(n=37, l=4, mu=75.0)   # mid-height stencils off the walls
    pb = rbffd.ns_problem(nodes, precision=64, threads_per_node=1, **prm)
    U0 = _state("flow", nodes)
    clean = pb.rhs(0.0, rbffd.state_tensor(U0, 64)).cpu().numpy()
    _, idx = pb.weights("dx")
    at = int(np.argmin(np.abs(nodes.z[:nodes.n_prog] - 3200.0) + np.abs(nodes.x[:nodes.n_prog])))
    U0[0, at] = bad
    got = pb.rhs(0.0, rbffd.state_tensor(U0, 64)).cpu().numpy()
    reads = (idx == at).any(1)
    assert not np.isfinite(got[reads, 0]).any()        # every tendency of u there
    assert np.array_equal(got[~reads], clean[~reads])
    pb.close()
