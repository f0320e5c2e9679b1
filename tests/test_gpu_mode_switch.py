"""Run modes of one problem in turn on one state: a graph captured before a
persistent plan is built still reads live buffers afterwards, so a replay on
the same state, step and step count equals the first one bit for bit.  Another
problem is created in between, so that memory given back would be overwritten.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1509_02615_gb300 import inputs as inp  # noqa: E402
from paper_1509_02615_gb300 import rbffd  # noqa: E402


@pytest.mark.parametrize("precision", [64, 32])
@pytest.mark.parametrize("storage", ["per-node", "lattice"])
def test_graph_persistent_graph(precision, storage):
    nodes = inp.density_current_nodes(400.0)
    pb = rbffd.ns_problem(nodes, precision=precision, threads_per_node=2, storage=storage)
    U0 = rbffd.state_tensor(inp.perturbed_density_current(nodes, 5), precision)
    U = U0.clone()

    def run():
        U.copy_(U0)
        pb.run(0.0, 1.0, 20, U)
        pb.sync()
        return U.clone()

    pb.set_run_mode("graph")
    first = run()
    for lanes in (1, 4):
        pb.set_run_mode("persistent", lanes=lanes)
        other = rbffd.ns_problem(nodes, precision=precision, mu=10.0, threads_per_node=1)
        assert torch.isfinite(run()).all()
        pb.set_run_mode("graph")
        assert torch.equal(run(), first)
        other.close()
    pb.close()
