"""GPU: load vector and element gradient over the whole range of float64: inputs
scaled by powers of two give the same results scaled alike, up to the largest
finite values (no sum overflows that its result does not)."""
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def _values(h, seed, nrhs):
    u = synth.uniform(seed, h.n_nodes * nrhs).reshape(h.n_nodes, nrhs)
    return torch.from_numpy(u if nrhs > 1 else u[:, 0].copy()).cuda()


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("dim,ne,nsub", [(3, 10, 2), (2, 18, 2)])
def test_load_vector(dim, ne, nsub, nrhs):
    from paper_2410_14786_gb300 import BDDC
    h = BDDC.from_problem(synth.make_problem(dim, ne, nsub, "one", k=105), nrhs_max=nrhs)
    for f in (_values(h, 106, nrhs), torch.ones_like(_values(h, 106, nrhs))):
        b = h.rhs(f)
        for k in (-900, 900, 1016, 1020, 1023):
            got = h.rhs(f * 2.0 ** k)
            assert bool(torch.isfinite(got).all()), k
            assert torch.equal(got, b * 2.0 ** k), k
