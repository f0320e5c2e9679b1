"""The register-filling FP32 forms of the persistent advection kernel, asked for
where nothing else fits, so that they are the ones that run.

In the vortex flow (two velocity parts) two lanes per node hold up to 320 nodes
per SM and one lane up to 384, both with 16-bit indices; 52,000 to 58,000 nodes
on 152 SMs therefore run with one lane, 46,516 with two when asked, and past
65,536 nodes no form fits.  Runs equal graph replay with the same lanes bit for
bit.
"""
import pytest

from paper_1509_02615_gb300 import configs

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1509_02615_gb300 import rbffd  # noqa: E402


def _against_graph(pb, wl, lanes):
    i = pb.info()
    assert i["run_mode"] == 2 and i["persist_lanes"] == lanes and i["threads_per_node"] == lanes
    A = rbffd.state_tensor(wl.U0, 32)
    B = A.clone()
    pb.run(0.3 * wl.dt, wl.dt, 11, A)
    pb.sync()
    pb.set_run_mode("graph")
    assert pb.info()["threads_per_node"] == lanes
    pb.run(0.3 * wl.dt, wl.dt, 11, B)
    pb.sync()
    assert torch.equal(A, B) and not torch.equal(A, rbffd.state_tensor(wl.U0, 32))


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_one_lane():
    wl = configs.vortex(0.00465, "hex")
    if not 320 * _sms() < wl.nodes.n_prog <= 384 * _sms():
        pytest.skip("sized for 152 SMs")
    pb = rbffd.advection_problem(wl.nodes, precision=32, **wl.params)
    pb.set_run_mode("persistent")
    _against_graph(pb, wl, 1)
    pb.close()


def test_two_lanes():
    wl = configs.vortex(0.005, "hex")
    if wl.nodes.n_prog > 320 * _sms():
        pytest.skip("sized for 152 SMs")
    pb = rbffd.advection_problem(wl.nodes, precision=32, **wl.params)
    pb.set_run_mode("persistent", lanes=2)
    _against_graph(pb, wl, 2)
    pb.close()


def test_more_nodes_than_16_bit_indices():
    wl = configs.vortex(0.00415, "hex")
    assert wl.nodes.n_prog > 65536
    pb = rbffd.advection_problem(wl.nodes, precision=32, **wl.params)
    assert pb.info()["run_mode"] == 1
    with pytest.raises(rbffd.RBFError) as e:
        pb.set_run_mode("persistent")
    assert e.value.code == rbffd.RBF_E_ARG
    pb.close()
