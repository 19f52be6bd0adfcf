"""GPU: the rows of the fixed-point float64 operators against the operators in
full (full_operators=True), each relative to its own sum |a_ij| |x_j|: operands
with one entry, on one side of a weakly conducting slab, or spread over many
decades, conductivities with jumps inside a subdomain, and the largest operators.
x0 = P_I b (a solve of 0 iterations) is one product with every A_II^-1."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def _problem(dim, ne, nsub, field):
    p = synth.make_problem(dim, ne, nsub, "lognormal" if field == "lognormal" else "one", k=91)
    e = np.arange(ne ** dim)
    s = ne // nsub
    last = e // ne ** (dim - 1) % s   # place along the last axis within the subdomain
    if field == "slab":
        p.elem_sigma = np.where(last == s // 2, 1e-6, 1.0)
    if field == "decades":
        p.elem_sigma = 10.0 ** synth.uniform(92, ne ** dim, -3.0, 3.0)
    return p


def _operand(kind, dim, ne, nsub, nrhs):
    n1, s = ne + 1, ne // nsub
    n = n1 ** dim
    u = synth.uniform(93, n * nrhs).reshape(n, nrhs)
    idx = np.arange(n)
    place = np.stack([idx // n1 ** k % n1 % s for k in range(dim)])   # within the subdomain
    if kind == "one":
        u *= (place == 1 + np.arange(dim)[:, None] % (s - 1)).all(0)[:, None]
    if kind == "side":
        u *= (place[-1] < s // 2)[:, None]
    if kind == "spread":
        u *= 10.0 ** synth.uniform(94, n * nrhs, -9.0, 0.0).reshape(n, nrhs)
    return u


@pytest.mark.parametrize("nrhs", [1, 3, 8])
@pytest.mark.parametrize("kind", ["dense", "one", "side", "spread"])
@pytest.mark.parametrize("dim,ne,nsub,field", [(3, 16, 2, "lognormal"), (3, 16, 2, "slab"), (3, 14, 2, "decades"),
                                               (2, 24, 2, "slab"), (3, 24, 4, "lognormal")])
def test_rows_against_the_full_operators(dim, ne, nsub, field, kind, nrhs):
    from oracle.bddc_oracle import Oracle
    from paper_2410_14786_gb300 import BDDC
    p = _problem(dim, ne, nsub, field)
    b = _operand(kind, dim, ne, nsub, nrhs)
    bd = torch.from_numpy(b if nrhs > 1 else b[:, 0].copy()).cuda()
    x = {}
    for full in (False, True):
        h = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs, full_operators=full)
        assert h.info()["symmetric_operators"] == (0 if full else 1)
        x[full] = h.pcg_solve(bd, maxit=0)[0].cpu().numpy().reshape(-1, nrhs)
    o = Oracle(p.dim, p.ne, p.elem_sigma, p.elem_subdomain, p.n_sub)
    # both sides: a float64 sum of n products in 16 parts or more, or no worse,
    # and the two triangles of the inverse averaged or not (its own rounding)
    for i in range(p.n_sub):
        I = o.interior[i]
        A = np.linalg.inv(o.Ai[i][np.ix_(I, I)])
        rows = np.asarray(o.free)[o.R[i][I]]
        size = np.abs(A) @ np.abs(b[rows])
        bound = 4 * (I.size / 16 + 5) * 2.0 ** -53
        err = np.abs(x[False][rows] - x[True][rows])
        assert (err <= bound * size).all(), (i, float((err / np.maximum(size, 1e-300)).max()), bound)


@pytest.mark.parametrize("size", [57, 62, 65])
def test_largest_operators(size):
    """3136 and 3721 rows: 12 and 8 warps, a column at a time; 4096 rows: beyond the fixed-point form (interiors)."""
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(2, 2 * size, 2, "lognormal", k=95)
    g = BDDC.from_problem(p, precision="fp64", nrhs_max=2)
    f = BDDC.from_problem(p, precision="fp64", nrhs_max=2, full_operators=True)
    r = torch.from_numpy(synth.uniform(96, g.n_nodes * 2).reshape(g.n_nodes, 2)).cuda()
    for v in (r, r[:, 0].contiguous()):
        zg, zf = g.apply(v), f.apply(v)
        # three products of at most 4096 terms in a chain, 10 for the cancellation between their sums
        assert float((zg - zf).abs().max() / zf.abs().max()) < 3 * 4096 * 2.0 ** -53 * 10
