"""The projection's operator kernel walks column groups one after another over
a plane: grids whose planes end within a block, with odd rows (one column per
thread), rows shorter than a warp and several slabs, against the oracle."""
import numpy as np
import pytest

from paper_2604_11959_gb300 import inputs

from _gpu_helpers import make_geometry, refs_for

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-9, "mixed": 2e-6}   # the solves' 1e-12 and float rounding, as in the other projection tests


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_11959_gb300 import eb as _eb
    _eb.load(build_if_missing=True)
    return _eb


@pytest.mark.parametrize("n", [(4, 4, 4), (5, 7, 6), (17, 5, 9), (45, 37, 20), (130, 14, 6), (62, 33, 41)])
@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_ragged_projections_match_oracle(eb, oracle, n, precision):
    from oracle import eb_project as proj
    w = inputs.Workload("ragged", *n, 1, terrain="grf", seed=3, hmax=0.15)
    h = w.heights()
    dom = oracle.Domain(w.nx, w.ny, w.nz, w.Lx, w.Ly, w.Lz, h)
    G = oracle.geometry(dom)
    rng = np.random.default_rng(4)
    dtype = torch.float64 if precision == "f64" else torch.float32
    dev = {}
    for g, f in ((1, "rhou"), (2, "rhov"), (3, "rhow")):
        a = 1.0 + 0.5 * rng.standard_normal(dom.shape(g))
        a[G[g]["alpha"] == 0] = 0.0
        if g == 3:
            a[0] = a[-1] = 0.0
        dev[f] = torch.from_numpy(a).to(device="cuda", dtype=dtype)
    host = {f: dev[f].double().cpu().numpy() for f in dev}
    dt = 0.5 * w.Lx / w.nx
    geo = make_geometry(eb, w, h, precision, refs_for(w.nz, w.Lz))
    U = geo.empty_state()
    U["rho"].zero_()
    U["rhotheta"].zero_()
    for f in dev:
        U[f].copy_(dev[f])
    it, res = eb.project(geo, U, dt, rtol=1e-12, maxit=5000)
    assert res <= 1e-12, (it, res)
    want = proj.project(dom, G, host["rhou"], host["rhov"], host["rhow"], dt, rtol=1e-12)[:3]
    scale = max(np.abs(x).max() for x in want)
    for f, x in zip(("rhou", "rhov", "rhow"), want):
        assert np.abs(U[f].double().cpu().numpy() - x).max() <= TOL[precision] * scale, f
    geo.close()
