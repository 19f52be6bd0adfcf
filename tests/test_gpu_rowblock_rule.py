"""GPU: when the several-column sweeps are row-blocked: the interior forest of the
sparse local solver always, whatever the coarse threshold (set by hand or by the
autotuner); the coarse factor from 2 columns on, large ones from 4."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def test_interior_forest_ignores_the_coarse_threshold():
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(2, 60, 1, "lognormal", k=111)   # one subdomain: an apply is two interior solves
    h = BDDC.from_problem(p, nrhs_max=3, local_solver="sparse")
    r = torch.from_numpy(synth.uniform(112, h.n_nodes * 3).reshape(h.n_nodes, 3)).cuda()
    z = h.apply(r)
    t = h.get_tuning()
    h.set_tuning(dict(t, coarse_rowblock_min_nrhs=65))
    assert torch.equal(h.apply(r), z)   # (one row and column per warp sums in another order)


def test_autotuned_sparse_local_handle():
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(2, 96, 4, "one", k=113)
    h = BDDC.from_problem(p, nrhs_max=2, local_solver="sparse")
    r = torch.from_numpy(synth.uniform(114, h.n_nodes * 2).reshape(h.n_nodes, 2)).cuda()

    def interior_us():
        v = sorted(h.profile_apply(r, reps=9)["interior_op"] for _ in range(5))
        return v[2]
    before = interior_us()
    h.autotune()
    assert interior_us() <= 1.5 * before


@pytest.mark.parametrize("ne,nsub,least", [(32, 8, 2), (48, 12, 4)])
def test_coarse_default(ne, nsub, least):
    from paper_2410_14786_gb300 import BDDC
    h = BDDC.from_problem(synth.make_problem(3, ne, nsub, "one", k=115), precision="fp32", nrhs_max=4)
    assert (h.info()["coarse_factor_entries"] > 5_000_000) == (least == 4)
    assert h.get_tuning()["coarse_rowblock_min_nrhs"] == least
