"""Corrected runs whose network leaves the ghost data little shared memory: wide
stencils and many nodes per CTA.  With ghost data in their smallest form the run
takes place in one launch and agrees with the stand-alone kernels to 1e-5
relative l2 per field after 10 steps (FP32 sums in another order, the bound of
tests/test_gpu_learned_fused.py for 40 steps), and so does the plain run of the
same plan.  Where nothing makes room, the stand-alone kernels run instead.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1509_02615_gb300 import inputs as inp  # noqa: E402
from paper_1509_02615_gb300 import learned  # noqa: E402
from paper_1509_02615_gb300 import rbffd  # noqa: E402

SCALES = np.array([2.0, 1.5, 0.5, 2e-4, 0.1, 0.05, 0.02, 1e-5, 4.0, 3.0, 6.0, 1e-3], np.float32)
ALPHA = (0.5, 0.5, 1.0, 0.25)


def _rel(a, b):
    return max(float((a[:, f] - b[:, f]).norm() / b[:, f].norm()) for f in range(4))


def _problem(h, n, l):
    nodes = inp.density_current_nodes(h)
    pb = rbffd.ns_problem(nodes, precision=32, n=n, l=l, threads_per_node=1)
    mlp = rbffd.Mlp(pb)
    mlp.set_params(learned.init_params(4 * n, seed=7))
    mlp.set_scales(SCALES)
    return nodes, pb, mlp, rbffd.state_tensor(inp.perturbed_density_current(nodes, 3), 32)


def _check(nodes, pb, mlp, U0, label):
    out = {}
    for mode in ("planned", "graph"):
        if mode == "graph":
            pb.set_run_mode("graph")
        A, B = U0.clone(), U0.clone()
        assert mlp.run(0.0, nodes.h / 400.0, 10, A, alpha=ALPHA) == 0
        pb.run(0.0, nodes.h / 400.0, 10, B)
        pb.sync()
        out[mode] = [v[:pb.n_prog].double() for v in (A, B)]
    errs = [_rel(a, b) for a, b in zip(out["planned"], out["graph"])]
    effect = _rel(*out["graph"])
    print(f"{label}: corrected {errs[0]:.1e}, plain {errs[1]:.1e}, effect of the correction {effect:.1e}")
    assert max(errs) < 1e-5
    assert effect > 10 * max(errs)
    return errs[0]


@pytest.mark.parametrize("h,n,l,lanes,ctas", [(141.0, 45, 4, 1, 152), (141.0, 45, 4, 1, 76), (200.0, 45, 4, 1, 38),
                                              (200.0, 56, 5, 1, 152), (400.0, 56, 5, 1, 38), (300.0, 37, 4, 1, 19)])
def test_explicit_plan(h, n, l, lanes, ctas):
    nodes, pb, mlp, U0 = _problem(h, n, l)
    pb.set_run_mode("persistent", lanes, ctas)
    assert pb.info()["persist_ctas"] == ctas
    assert _check(nodes, pb, mlp, U0, f"h={h:g} n={n} {ctas} CTAs") > 0.0   # equal bits: the stand-alone kernels ran
    mlp.close()
    pb.close()


def test_tuned_plan():
    nodes, pb, mlp, U0 = _problem(141.0, 45, 4)
    lanes, ctas = mlp.tune_run()
    assert pb.info()["run_mode"] == 2
    _check(nodes, pb, mlp, U0, f"tuned {lanes} lanes, {ctas} CTAs")
    mlp.close()
    pb.close()


def test_no_room_at_all():
    nodes, pb, mlp, U0 = _problem(124.0, 56, 5)   # some 160 nodes per CTA: lists and network exceed shared memory
    pb.set_run_mode("persistent", 1, 152)
    assert _check(nodes, pb, mlp, U0, "no room") == 0.0
    mlp.close()
    pb.close()
