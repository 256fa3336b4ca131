"""The work split of the bulk kernel as a handle reports and keeps it."""
import pytest

from paper_2604_11959_gb300 import inputs

from _gpu_helpers import FIELDS, make_geometry, refs_for, to_device

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_11959_gb300 import eb as _eb
    _eb.load(build_if_missing=True)
    return _eb


def small(eb, precision):
    w = inputs.Workload("split", 32, 32, 16, 1, terrain="woa", hmax=0.1)
    refs = refs_for(w.nz, w.Lz)
    return w, refs, make_geometry(eb, w, w.heights(), precision, refs)


def test_reported_tile_rows_are_those_in_use(eb):
    """A small FP64 domain runs 16 x 8 tiles and says so; rows the caller sets
    stay set, with any height of the slabs."""
    w, refs, g = small(eb, "f64")
    U = to_device(w.state("sheltered", seed=3), "f64", refs)
    assert g.info()["tile_rows"] == 8
    want = eb.step(g, U, w.dt(), 2)
    eb.set_slab_levels(g, 4)
    assert g.info()["tile_rows"] == 16
    eb.set_slab_levels(g, 0)
    assert g.info()["tile_rows"] == 8
    eb.set_tile_rows(g, 16)
    for split in (0, 4, 0):
        eb.set_slab_levels(g, split)
        assert g.info()["tile_rows"] == 16
        got = eb.step(g, U, w.dt(), 2)
        for f in FIELDS:
            assert torch.equal(got[f], want[f]), (split, f)
    g.close()
    _, _, m = small(eb, "mixed")
    for rows in (16, 14):
        eb.set_tile_rows(m, rows)
        assert m.info()["tile_rows"] == rows
    m.close()
