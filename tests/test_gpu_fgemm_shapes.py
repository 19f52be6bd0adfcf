"""GPU: every shape of the blocked float32 product (row tiles of 32, 64 and 128
rows; 1, 2 and 4 column blocks) bit for bit against the streamed GEMV, which sums
in the same order and takes blocks of 4 columns. x0 = P_I b (a solve of 0
iterations) is one product with every A_II^-1; the packing of the operand is one
launch more."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


@pytest.fixture(scope="module", params=["many rows", "few rows"])
def handle(request):
    from paper_2410_14786_gb300 import BDDC
    if request.param == "many rows":   # 512 operators of 343 rows: 1536 tiles of 128 rows, more than two per SM
        p = synth.make_problem(3, 64, 8, "lognormal", k=123)
        h = BDDC.from_problem(p, precision="fp32", nrhs_max=33)
    else:                              # 12 operators of about 500 to 2100 rows: about 110 tiles of 128 rows
        sub, n_sub, cell = synth.voronoi_partition(24, 12, 4124)
        h = BDDC(3, 24, synth.layer_sigma(24, cell), sub, n_sub, precision="fp32", nrhs_max=33)
    yield h
    h.close()


def _product(h, b):
    n0 = h.info()["kernel_launches"]
    x = h.pcg_solve(b, maxit=0)[0].reshape(h.n_nodes, -1)
    return x, h.info()["kernel_launches"] - n0


@pytest.mark.parametrize("nrhs", [5, 8, 9, 16, 17, 33])
def test_same_values_as_the_streamed_gemv(handle, nrhs):
    h = handle
    b = torch.from_numpy(synth.uniform(124, h.n_nodes * nrhs).reshape(h.n_nodes, nrhs)).cuda()
    x, launches = _product(h, b)
    for k in range(0, nrhs - nrhs % 4, 4):
        y, launches4 = _product(h, b[:, k:k + 4].contiguous())
        assert launches == launches4 + 1
        assert torch.equal(x[:, k:k + 4], y), k
