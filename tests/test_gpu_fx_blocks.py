"""GPU: the block shapes of the fixed-point products: 4, 6 and 12 warps, one to three
blocks per SM (few units against more than there are SMs), 1 to 8 columns, operators
of 1 to 11 tile rows, against the operators in full."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


# (dim, elements per subdomain, subdomains per direction): 216 or 256 operators (more
# than SMs) of 64, 125, 216 and 343 rows in 3D, and a few of the same
@pytest.mark.parametrize("nrhs", [1, 2, 3, 8])
@pytest.mark.parametrize("size,nsub", [(5, 6), (6, 6), (7, 6), (8, 6), (6, 3), (8, 2)])
def test_every_block_shape(size, nsub, nrhs):
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(3, size * nsub, nsub, "lognormal", k=131)
    g = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs)
    f = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs, full_operators=True)
    assert g.info()["symmetric_operators"] == 1
    u = synth.uniform(132, g.n_nodes * nrhs).reshape(g.n_nodes, nrhs)
    r = torch.from_numpy(u if nrhs > 1 else u[:, 0].copy()).cuda()
    zg, zf = g.apply(r).reshape(-1, nrhs), f.apply(r).reshape(-1, nrhs)
    # three products of at most 386 terms in a chain, 10 for the cancellation between their sums
    assert float(((zg - zf).abs().amax(0) / zf.abs().amax(0)).max()) < 3 * 386 * 2.0 ** -53 * 10
    assert torch.equal(g.apply(r).reshape(-1, nrhs), zg)
