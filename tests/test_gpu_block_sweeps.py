"""GPU: the row-blocked sweeps on the float64 matrix instruction (several
columns) against the one-column sweeps, column by column: the coarse factor on
one and several levels, and the interior forest of the sparse local solver, with
column counts off the blocks of 8."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# both sides sum at most 2000 float64 products per row, over at most 12 levels, in
# another order: 12 * sqrt(2000) * 2^-53 = 6e-14 for typical terms, times the
# condition of the factors' rows (below 100 on these problems)
BOUND = 6e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


@pytest.mark.parametrize("nrhs", [2, 7, 8, 9, 33])
@pytest.mark.parametrize("case", ["one_level", "levels", "forest"])
def test_columns_match_the_one_column_sweeps(case, nrhs):
    from paper_2410_14786_gb300 import BDDC
    p = {"one_level": synth.make_problem(3, 16, 4, "lognormal", k=81),
         "levels": synth.make_problem(3, 48, 8, "lognormal", k=82),
         "forest": synth.make_problem(2, 120, 3, "lognormal", k=83)}[case]
    kw = dict(precision="fp64", local_solver="sparse" if case == "forest" else "dense")
    g = BDDC.from_problem(p, nrhs_max=nrhs, **kw)
    one = BDDC.from_problem(p, nrhs_max=1, **kw)
    r = torch.from_numpy(synth.uniform(84, g.n_nodes * nrhs).reshape(g.n_nodes, nrhs)).cuda()
    z = g.apply(r)
    uc = g.coarse_vectors(nrhs)[1]
    for k in {0, nrhs // 2, nrhs - 1}:
        zk = one.apply(r[:, k].contiguous())
        uk = one.coarse_vectors(1)[1][:, 0]
        assert float((uc[:, k] - uk).abs().max() / uk.abs().max()) < BOUND, k
        assert float((z[:, k] - zk).abs().max() / zk.abs().max()) < BOUND, k
