"""GPU: which families of float64 operators run in block fixed point: large ones
and few ones; many small operators stay with the streamed GEMV, one family or both."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


# (dim, elements, subdomains per direction, columns): interiors and interfaces of
# about 25 and 23, 27 and 76, 225 and 55, 343 and 290 rows
@pytest.mark.parametrize("dim,ne,nsub,nrhs,families", [(2, 72, 12, 1, 0), (2, 72, 12, 8, 0), (3, 24, 6, 1, 1),
                                                       (3, 24, 6, 8, 1), (2, 96, 6, 1, 1), (3, 32, 4, 1, 2)])
def test_families(dim, ne, nsub, nrhs, families):
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(dim, ne, nsub, "lognormal", k=97)
    g = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs)
    f = BDDC.from_problem(p, precision="fp64", nrhs_max=nrhs, full_operators=True)
    assert g.info()["symmetric_operators"] == (1 if families else 0)
    # a family in full has the same bytes on both handles
    same = [g.info()[k] == f.info()[k] for k in ("interior_op_bytes", "interface_op_bytes")]
    assert 2 - sum(same) == families
    u = synth.uniform(98, g.n_nodes * nrhs).reshape(g.n_nodes, nrhs)
    r = torch.from_numpy(u if nrhs > 1 else u[:, 0].copy()).cuda()
    zg, zf = g.apply(r), f.apply(r)
    if not families:
        assert torch.equal(zg, zf)
    # three products of at most 343 terms in a chain, 10 for the cancellation between their sums
    assert float((zg - zf).abs().max() / zf.abs().max()) < 3 * 343 * 2.0 ** -53 * 10
    t = g.autotune()
    assert np.isfinite(g.apply(r).cpu().numpy()).all() and t["gemv_rows_interior"] in (64, 128, 256)
