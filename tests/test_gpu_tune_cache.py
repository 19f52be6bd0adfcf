"""GPU: a tune cache written for other kernels is measured again, not applied."""
import json

import pytest

import synth

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2410_14786_gb300 import build
    build.build()


def test_entries_of_other_kernels(tmp_path):
    from paper_2410_14786_gb300 import BDDC
    p = synth.make_problem(3, 16, 4, "one", k=121)
    path = tmp_path / "tune.json"
    a = BDDC.from_problem(p, nrhs_max=2, tune_cache=str(path))
    assert not a.tuned_from_cache
    (key, entry), = json.loads(path.read_text()).items()
    # without a revision, and with another one
    old = key[key.index("dim"):]
    stale = dict(entry, coarse_rowblock_min_nrhs=65, gemv_rows_interior=256)
    path.write_text(json.dumps({old: stale, "kernels1|" + old: stale}))
    b = BDDC.from_problem(p, nrhs_max=2, tune_cache=str(path))
    assert not b.tuned_from_cache
    table = json.loads(path.read_text())
    assert set(table) == {old, "kernels1|" + old, key} and table[key] == b.get_tuning()
    assert BDDC.from_problem(p, nrhs_max=2, tune_cache=str(path)).tuned_from_cache
