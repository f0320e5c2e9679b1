"""Stencil searches of different sizes from several threads at once, each on a
stream of its own: every search needs its own amount of shared memory, and none
may change what another one's launch is allowed.  Results equal those of the
same searches one after the other.
"""
import threading

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1509_02615_gb300 import rbffd  # noqa: E402


def test_searches_of_several_threads():
    g = torch.Generator(device="cuda").manual_seed(3)
    x, z = (torch.rand(2000, generator=g, device="cuda", dtype=torch.float64) for _ in range(2))
    sizes = (128, 7, 37, 91)
    want = {n: rbffd.build_stencils(x, z, 2000, n) for n in sizes}
    torch.cuda.synchronize()
    bad = []

    def work(n):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(300):
                    if not torch.equal(rbffd.build_stencils(x, z, 2000, n), want[n]):
                        bad.append((n, "another result"))
                        return
        except rbffd.RBFError as e:
            bad.append((n, str(e)))

    threads = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
