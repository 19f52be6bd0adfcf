"""GPU: fixed-point products of handles with operators of different sizes (other block
shapes and shared memory), called from several threads on streams of their own."""
import threading

import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def test_handles_of_different_sizes_in_threads():
    from paper_2410_14786_gb300 import BDDC
    jobs = []
    for size, nsub in ((5, 6), (8, 3), (10, 2), (7, 6)):
        p = synth.make_problem(3, size * nsub, nsub, "lognormal", k=141)
        g = BDDC.from_problem(p, precision="fp64")
        r = torch.from_numpy(synth.uniform(142, g.n_nodes)).cuda()
        jobs.append((g, r, g.apply(r)))
    torch.cuda.synchronize()
    bad = []

    def work(g, r, want):
        try:
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                out = [g.apply(r) for _ in range(60)]
            s.synchronize()
            bad.extend(not torch.equal(z, want) for z in out if not torch.equal(z, want))
        except Exception as e:   # (a launch that another thread's setting made fail)
            bad.append(repr(e))
    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad[:3]
