"""GPU: the element term of the adjoint gradient, every element relative to its own
sum |K_ab| |u_a| |lambda_b|, against extended precision: smooth and random fields,
and fields whose peaks meet along edges, where K_ref has no weight in 3D."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def _exact(dim, ne, u, lam):
    """(g, sum of magnitudes) per element, summed over the columns."""
    h = np.longdouble(1) / ne
    K = {2: [np.longdouble(4) / 6, -np.longdouble(1) / 6, -np.longdouble(2) / 6],
         3: [h / 3, np.longdouble(0), -h / 12, -h / 12]}[dim]
    n1 = ne + 1
    free = np.zeros((n1,) * dim, dtype=bool)
    free[(slice(1, -1),) * dim] = True
    grid = [np.where(free.reshape(-1, 1), v, 0).astype(np.longdouble).reshape((n1,) * dim + (-1,)) for v in (u, lam)]

    def corner(v, a):
        return v[tuple(slice((a >> (dim - 1 - ax)) & 1, ne + ((a >> (dim - 1 - ax)) & 1)) for ax in range(dim))]
    g = size = 0
    for a in range(1 << dim):
        for b in range(1 << dim):
            p = K[bin(a ^ b).count("1")] * corner(grid[0], b) * corner(grid[1], a)
            g, size = g - p, size + abs(p)
    return g.sum(-1).reshape(-1), size.sum(-1).reshape(-1)


@pytest.mark.parametrize("nrhs", [1, 3])
@pytest.mark.parametrize("kind", ["smooth", "random", "edge peaks", "spread"])
@pytest.mark.parametrize("dim,ne,nsub", [(3, 12, 2), (3, 9, 3), (2, 20, 2)])
def test_every_element(dim, ne, nsub, kind, nrhs):
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(dim, ne, nsub, "one", k=101)
    h = BDDC.from_problem(p, nrhs_max=nrhs)
    n1 = ne + 1
    idx = np.arange(n1 ** dim)
    x = idx % n1
    rnd = synth.uniform(102, 2 * idx.size * nrhs).reshape(2, idx.size, nrhs)
    v = 1.0 + 0.1 * rnd if kind == "smooth" else rnd.copy()
    if kind == "edge peaks":   # u large at every third x, lambda one edge further
        for f in range(2):
            v[f] *= np.where(x % 3 == f, 1.0, 1e-8)[:, None]
    if kind == "spread":
        v *= 10.0 ** synth.uniform(103, v.size, -7.0, 0.0).reshape(v.shape)
    u, lam = (torch.from_numpy(q if nrhs > 1 else q[:, 0].copy()).cuda() for q in v)
    g = h.elem_grad(u, lam).cpu().numpy()
    want, size = _exact(dim, ne, v[0], v[1])
    # float64: 8 products of 8 in a chain, and the sum over the columns
    bound = (8 + 8 + nrhs) * 2.0 ** -53
    live = size > 0
    assert (g[~live] == 0).all()
    err = np.abs(g - want)[live] / size[live]
    assert err.max() <= bound, float(err.max())
