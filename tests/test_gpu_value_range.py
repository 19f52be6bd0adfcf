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


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("dim,ne,nsub", [(3, 10, 2), (2, 18, 2)])
def test_element_gradient(dim, ne, nsub, nrhs):
    from paper_2410_14786_gb300 import BDDC
    h = BDDC.from_problem(synth.make_problem(dim, ne, nsub, "one", k=107), nrhs_max=nrhs)
    # differences of u exceed 2^1024 when scaled, K_ref u (4 / 3 of u at most) does not
    u, lam = 1.45 * _values(h, 108, nrhs), _values(h, 109, nrhs)
    g = h.elem_grad(u, lam)
    # 16 roundings of sums of at most 4^dim products and columns, h / 3 or 2 / 3 the largest weight
    bound = 1.45 * 16 * 2.0 ** -53 * 4 ** dim * nrhs * (1.0 / ne if dim == 3 else 2.0)
    for ku, kl in ((1023, 0 if dim == 3 else -30), (1023, -1000), (-1000, 1023), (1022, -3), (1010, 10), (700, 300), (500, 520), (-500, -400), (0, 0)):
        got = h.elem_grad(u * 2.0 ** ku, lam * 2.0 ** kl)
        assert bool(torch.isfinite(got).all()), (ku, kl)
        back = got * 2.0 ** (-(ku + kl) // 2) * 2.0 ** (-(ku + kl) - (-(ku + kl) // 2))
        assert float((back - g).abs().max()) <= bound, (ku, kl)
