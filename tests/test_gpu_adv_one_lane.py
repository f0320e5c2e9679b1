"""Advection where the packed pairs of slots and the register-resident forms
change: problems that fill the register file (one lane per node in FP32),
stencils past the register variants, odd slot counts, and the two sources of
the velocity time factors (the call's own time, the graph's device time).

Every comparison is bit for bit: the forms share lanes, slot order, time
factors and updates.
"""
import pytest

from paper_1509_02615_gb300 import configs
from paper_1509_02615_gb300 import inputs as inp

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1509_02615_gb300 import rbffd  # noqa: E402


@pytest.mark.parametrize("flow", ["vortex", "deformational"])
@pytest.mark.parametrize("precision", [32, 64])
def test_large_problem_run_equals_graph(flow, precision):
    wl = configs.vortex(0.005, "hex") if flow == "vortex" else configs.advection(201)
    pb = rbffd.advection_problem(wl.nodes, precision=precision, **wl.params)
    lanes = pb.info()["threads_per_node"]
    A = rbffd.state_tensor(wl.U0, precision)
    B = A.clone()
    pb.run(0.3 * wl.dt, wl.dt, 21, A)
    pb.sync()
    print(flow, precision, "run mode", pb.info()["run_mode"], "lanes", lanes)
    pb.set_run_mode("graph")
    assert pb.info()["threads_per_node"] == lanes
    pb.run(0.3 * wl.dt, wl.dt, 21, B)
    pb.sync()
    assert torch.equal(A, B) and not torch.equal(A, rbffd.state_tensor(wl.U0, precision))
    pb.close()


@pytest.mark.parametrize("precision", [32, 64])
@pytest.mark.parametrize("n,l", [(21, 3), (37, 4), (40, 4), (45, 4), (56, 5)])
def test_run_equals_single_steps(n, l, precision):
    wl = configs.advection(40)
    prm = dict(wl.params, n=n, l=l)
    pb = rbffd.advection_problem(wl.nodes, precision=precision, **prm)
    pb.set_run_mode("graph")
    dt, t0 = 0.25 * wl.dt, 0.4
    A = rbffd.state_tensor(wl.U0, precision)
    B = A.clone()
    pb.run(t0, dt, 3, A)
    for k in range(3):
        # the device time of a replay is t0 + dt + ... in order
        pb.rk4_step(t0 if k == 0 else t0 + dt if k == 1 else (t0 + dt) + dt, dt, B)
    pb.sync()
    assert torch.equal(A, B)
    pb.close()
