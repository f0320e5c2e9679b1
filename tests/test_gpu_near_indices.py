"""The FP32 stage kernels that take their operands through a ring in shared
memory and their neighbour indices in 16 bits (csrc/stream32.cuh): nodes whose
neighbours all lie within 32,767 places of the node order, nodes with farther
ones (ghosts), and both in one warp, over whole and partial rounds of the ring.

Tolerance.  Sums over n slots in FP32 of rounded weights are off by at most
(n + 2) 2^-24 sum |w (f_j - f_i)| <= (n + 2) 2^-23 n max|w| max|f| (a wrong
neighbour is off by some max|w| max|f|, a thousand times that), the reference being the FP64 sum over the problem's FP64 weights and the state,
ghosts included, that the FP32 call left.  A member of an ensemble does the
arithmetic of the same problem stepped alone, whose 4-lane kernel holds up to 48
slots in registers and reads 32-bit indices: these are equal in every bit.
"""
import numpy as np
import pytest

from paper_1509_02615_gb300 import inputs as inp

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

from paper_1509_02615_gb300 import rbffd  # noqa: E402
from test_gpu_fixed_point import _reference, _smooth  # noqa: E402


@pytest.mark.parametrize("h,layout,n,l,lanes", [
    (800.0, "hex", 37, 4, 1), (100.0, "hex", 37, 4, 1), (100.0, "hex", 37, 4, 2), (100.0, "cart", 31, 3, 1),
    (100.0, "scattered", 56, 5, 4), (400.0, "hex", 13, 2, 1), (100.0, "hex", 9, 1, 1)])
def test_rhs_with_near_and_far_neighbours(h, layout, n, l, lanes):
    nodes = (inp.poisson_disk_nodes(-25600.0, 25600.0, 0.0, 6400.0, h, seed=3, periodic_x=True)
             if layout == "scattered" else inp.density_current_nodes(h, layout))
    pb = rbffd.ns_problem(nodes, precision=32, n=n, l=l, mu=75.0, threads_per_node=lanes)
    U = rbffd.state_tensor(_smooth(nodes, np.random.default_rng(5)), 32)
    got = rbffd.fields(pb.rhs(0.0, U))
    ref, mag = _reference(pb, nodes, rbffd.fields(U), 75.0, np.float64)
    e, tol = np.abs(got - ref), (n + 2) * 2.0 ** -23 * mag
    print(f"h={h:g} {layout} n={n} lanes={lanes}: error / bound up to {(e / (tol + 1e-300)).max():.4f}")
    assert np.all(e <= tol)
    pb.close()


@pytest.mark.parametrize("lanes", [1, 2, 4])
def test_ensemble_members_equal_the_problem_alone(lanes):
    mem = [inp.density_current_member(h, lay, n, l, seed=3 + i, t_end=2 * 0.4)
           for i, (h, lay, n, l) in enumerate([(100.0, "hex", 37, 4), (800.0, "cart", 31, 3), (400.0, "scattered", 56, 5)])]
    ens = rbffd.ensemble_problem(mem, precision=32, threads_per_node=lanes)
    U = ens.state()
    ens.run(2, U)
    ens.sync()
    for r, m in enumerate(mem):
        pb = rbffd.ns_problem(m.nodes, precision=32, n=m.n, l=m.l, gamma_c=m.gamma_c, threads_per_node=lanes)
        V = rbffd.state_tensor(m.U0, 32)
        pb.run(0.0, m.dt, min(2, m.n_steps), V)
        pb.sync()
        assert torch.equal(U[ens.rec0[r]:ens.rec0[r] + m.nodes.n_prog], V[:m.nodes.n_prog]), r
        pb.close()
