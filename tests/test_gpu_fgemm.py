"""GPU: the blocked float32 product for blocks of right-hand sides (from 5
columns on) against the streamed GEMV, which runs single columns of the same
operators: every column of a block against the oracle-tested single-column
path, with row tiles, operator columns and right-hand sides off the tile sizes
(32 to 128 rows, 128 operator columns, 8 to 32 right-hand sides)."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# float32 products and sums over at most 1500 terms on both sides, in another
# order: sqrt(1500) 2^-24 = 2.3e-6 for a typical entry of one product, three
# products in a chain
BOUND = 1e-5


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


@pytest.mark.parametrize("nrhs", [5, 8, 9, 16, 17, 33, 64])
@pytest.mark.parametrize("cells,ne", [(3, 14), (30, 28)])
def test_blocks_match_single_columns(cells, ne, nrhs):
    from paper_2410_14786_gb300 import BDDC
    sub, n_sub, cell = synth.voronoi_partition(ne, cells, 4100 + ne)
    sigma = synth.layer_sigma(ne, cell)
    g = BDDC(3, ne, sigma, sub, n_sub, precision="fp32", nrhs_max=nrhs)
    one = BDDC(3, ne, sigma, sub, n_sub, precision="fp32", nrhs_max=nrhs)
    r = torch.from_numpy(synth.uniform(71, g.n_nodes * nrhs).reshape(g.n_nodes, nrhs)).cuda()
    z = g.apply(r)
    for k in {0, 3, nrhs // 2, nrhs - 1}:
        zk = one.apply(r[:, k].contiguous())
        assert float((z[:, k] - zk).abs().max() / zk.abs().max()) < BOUND, k
    # the columns are independent: the same block in another order
    perm = torch.arange(nrhs - 1, -1, -1, device="cuda")
    zp = g.apply(r[:, perm].contiguous())
    assert torch.allclose(zp[:, perm], z, rtol=0, atol=1e-12 * float(z.abs().max()))
