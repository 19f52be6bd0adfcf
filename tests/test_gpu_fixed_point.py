"""GPU: the float64 local operators in block fixed point (lower triangles of
32 x 32 tiles) against the float64 operators in full (full_operators=True),
through the C ABI, at operator sizes around the tile edges, few and many
subdomains (one or several blocks per operator) and every column blocking;
operands with infinities and NaN."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# (dim, elements, subdomains per direction): interiors of 1, 16, 25, 36, 961
# and 64, 343 rows, interfaces from 3 to 386 rows
SHAPES = [(2, 4, 2), (2, 15, 3), (2, 24, 4), (2, 14, 2), (2, 64, 2), (3, 10, 2), (3, 24, 3)]
# both sides round their products to float64 accuracy (2^-53 of the absolute
# sum per product, sums of at most 961 terms) in a chain of three local
# operators, the coarse solve and the couplings: 3 * 961 * 2^-53 = 3e-13, times
# the cancellation between v1, v2 and v3 (below 10 on these problems)
BOUND = 3e-12


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


@pytest.mark.parametrize("nrhs", [1, 2, 3, 8, 9])
@pytest.mark.parametrize("shape", SHAPES)
def test_matches_the_float64_operators(shape, nrhs):
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(*shape, "lognormal", k=61)
    g = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs)
    f = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs, full_operators=True)
    assert g.info()["symmetric_operators"] == 1 and f.info()["symmetric_operators"] == 0
    r = synth.uniform(62, g.n_nodes * nrhs).reshape(g.n_nodes, nrhs)
    r *= 10.0 ** np.linspace(-200, 200, nrhs)[None, :] if nrhs > 1 else 1.0   # every column has its own scale
    r = torch.from_numpy(r if nrhs > 1 else r[:, 0].copy()).cuda()
    zg, zf = g.apply(r), f.apply(r)
    err = (zg - zf).abs().amax(0) / zf.abs().amax(0)
    assert float(err.max()) < BOUND, err
    # the first column alone, on the handle set up for several
    r0 = r[:, 0].contiguous() if nrhs > 1 else r
    assert float((g.apply(r0) - f.apply(r0)).abs().max() / f.apply(r0).abs().max()) < BOUND
    zero = torch.zeros_like(r)
    assert bool((g.apply(zero) == 0).all())


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_operands(bad):
    """One non-finite entry spoils its own column only, as in float64."""
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(3, 16, 2, "lognormal", k=63)
    g = BDDC.from_problem(p, precision="fp64", nrhs_max=3)
    f = BDDC.from_problem(p, precision="fp64", nrhs_max=3, full_operators=True)
    r = torch.from_numpy(synth.uniform(64, g.n_nodes * 3).reshape(g.n_nodes, 3)).cuda()
    z = g.apply(r)
    r2 = r.clone()
    node = 3 + 17 * (3 + 17 * 3)   # an interior node of the first subdomain
    r2[node, 1] = bad
    zg, zf = g.apply(r2), f.apply(r2)
    assert torch.equal(zg[:, 0], z[:, 0]) and torch.equal(zg[:, 2], z[:, 2])
    assert torch.equal(torch.isfinite(zg), torch.isfinite(zf))
    assert torch.equal(torch.isnan(zg), torch.isnan(zf))
