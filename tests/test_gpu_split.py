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


def test_an_ensemble_leaves_its_members_splits_alone(eb):
    """A handle keeps its own split (16 x 8 tiles on a small FP64 domain)
    through a rejected ensemble, a member's life in one and its end; the
    ensemble's steps are the handle's bit for bit."""
    w, refs, g = small(eb, "f64")
    _, _, other = small(eb, "mixed")
    U = to_device(w.state("sheltered", seed=3), "f64", refs)
    want = eb.step(g, U, w.dt(), 2)
    for members in ([g, other], [g, g]):
        with pytest.raises(eb.EbError):
            eb.Ensemble(members)
        assert g.info()["tile_rows"] == 8
    _, _, h = small(eb, "f64")
    for schedule in ("persistent", "branches"):
        ens = eb.Ensemble([g, h])
        ens.set_schedule(schedule)
        for q in range(2):
            ens.set_state(q, U)
        ens.step([w.dt()] * 2, 2)
        assert g.info()["tile_rows"] == 8
        for q in range(2):
            got = ens.get_state(q)
            for f in FIELDS:
                assert torch.equal(got[f], want[f]), (schedule, q, f)
        ens.close()
    assert g.info()["tile_rows"] == 8
    got = eb.step(g, U, w.dt(), 2)
    for f in FIELDS:
        assert torch.equal(got[f], want[f]), f


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_captured_steps_outlive_an_ensemble(eb, precision):
    """A graph of a handle's step replays right while the handle is a member
    of an ensemble, and after: creating one frees nothing the graph reads."""
    w, refs, g = small(eb, precision)
    U = to_device(w.state("sheltered", seed=3), precision, refs)
    out = g.empty_state()
    want = {f: t.clone() for f, t in eb.step(g, U, w.dt(), out=out).items()}
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        eb.step(g, U, w.dt(), out=out)

    def replay():
        for f in FIELDS:
            out[f].zero_()
        graph.replay()
        torch.cuda.synchronize()
        for f in FIELDS:
            assert torch.equal(out[f], want[f]), f

    replay()
    ens = eb.Ensemble([g])
    replay()
    ens.set_state(0, U)
    ens.step([w.dt()], 1)
    replay()
    ens.close()
    replay()


@pytest.mark.parametrize("n", [(400, 400, 128), (320, 200, 30)])
def test_the_automatic_split_is_no_slow_one(eb, n):
    """An untuned mixed step of a hill takes no longer than the best of a few
    explicit slab heights but for 15 %: about the spread of the heights near the
    best one, and half of what a split whose last wave is nearly empty, or whose
    pieces are mostly prologue, loses."""
    w = inputs.Workload("split", *n, 1, terrain="gaussian", hmax=0.12)
    refs = w.references("sheltered")
    g = make_geometry(eb, w, w.heights(), "mixed", refs)
    U = to_device(w.state("sheltered", seed=3), "mixed", refs)
    out = g.empty_state()

    def time():
        best = float("inf")
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            eb.step(g, U, w.dt(), out=out)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    time()
    auto = time()
    explicit = {}
    for levels in (16, 32, 43, 64):
        eb.set_slab_levels(g, levels)
        explicit[levels] = time()
    assert auto <= 1.15 * min(explicit.values()), (auto, explicit)
    g.close()
