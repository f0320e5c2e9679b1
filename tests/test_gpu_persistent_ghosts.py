"""The persistent mode's ghost solve and plans where they can go wrong.

* FP32 ghost values straight from the records: against graph replay on walls
  on all sides (three boundary classes, corners), wide stencils, odd numbers of
  ghosts per CTA, and few or many threads per pair of ghosts; FP64 (ghost,
  field) items alike.  FP32 tolerance: rounding of the same sums in another
  order, below 1e-5 of each field after 10 steps (the graph mode itself is
  bounded at 1e-5 against FP64 there); FP64 1e-12.
* Helper threads (a CTA with far fewer nodes than threads) change nothing but
  the order of the ghost sums.
* Plans of several problems that share a kernel: a later plan with less shared
  memory does not disturb an earlier one.
"""
import numpy as np
import pytest

from paper_1509_02615_gb300 import configs
from paper_1509_02615_gb300 import inputs as inp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import rbffd  # noqa: E402


def _case(name):
    if name == "box":
        wl = configs.rising_bubble(500.0, "cart")
        return wl.nodes, dict(wl.params), wl.U0, wl.dt
    if name == "box_hex":
        wl = configs.rising_bubble(330.0, "hex")
        return wl.nodes, dict(wl.params), wl.U0, wl.dt
    if name == "bubble56":
        wl = configs.bubble(h=700.0, seed=1, t_end=10.0)
        return wl.nodes, dict(wl.params), wl.U0, wl.dt
    nodes = inp.density_current_nodes(800.0 if name == "current75" else 430.0)
    prm = dict(n=75, l=5, mu=75.0) if name == "current75" else dict(n=37, l=4, mu=75.0)
    return nodes, prm, inp.density_current_state(nodes), nodes.h / 400.0


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("case,lanes,ctas", [
    ("box", 1, 5), ("box", 2, 19), ("box", 4, 40), ("box_hex", 1, 7), ("box_hex", 4, 100), ("bubble56", 1, 3),
    ("bubble56", 2, 17), ("current75", 1, 10), ("current75", 4, 60), ("current37", 1, 31), ("current37", 2, 152)])
def test_persistent_ghosts_equal_graph(case, lanes, ctas, precision):
    nodes, prm, U0, dt = _case(case)
    U0 = U0 + 0.1 * np.cos(np.arange(U0.size)).reshape(U0.shape) * np.array([1.0, 0.0, 1.0, 1e-4])[:, None]
    pb = rbffd.ns_problem(nodes, precision=precision, threads_per_node=1, **prm)
    P = nodes.n_prog
    A = rbffd.state_tensor(U0, precision)
    B = A.clone()
    pb.set_run_mode("graph")
    pb.run(0.0, dt, 10, A)
    pb.set_run_mode("persistent", lanes, ctas)
    pb.run(0.0, dt, 10, B)
    pb.sync()
    a, b = A[:P].double(), B[:P].double()
    errs = [float(torch.linalg.vector_norm(a[:, f] - b[:, f]) / torch.linalg.vector_norm(a[:, f])) for f in range(4)]
    print(f"{case} FP{precision} lanes {lanes} CTAs {ctas}: persistent against graph {['%.1e' % e for e in errs]}")
    assert max(errs) < (1e-5 if precision == 32 else 1e-12)
    pb.close()


@pytest.mark.parametrize("precision", [32, 64])
def test_plans_sharing_a_kernel_do_not_disturb_each_other(precision):
    big, small = inp.density_current_nodes(300.0), inp.density_current_nodes(800.0)
    pbs, states = [], []
    for nodes, ctas in ((big, 20), (small, 40)):
        pb = rbffd.ns_problem(nodes, precision=precision, threads_per_node=1)
        pb.set_run_mode("persistent", 1, ctas)
        pbs.append(pb)
        states.append(rbffd.state_tensor(inp.density_current_state(nodes), precision))
    for _ in range(2):
        for pb, U, nodes in zip(pbs, states, (big, small)):
            pb.run(0.0, nodes.h / 400.0, 3, U)
            pb.sync()
            assert bool(torch.isfinite(U).all())
    for pb in pbs:
        pb.close()
