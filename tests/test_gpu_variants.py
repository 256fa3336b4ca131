"""Kernel variants that a dispatch chooses by size: each must give the same
results as the general path at the sizes where it can go wrong (tile edges,
remainders, the smallest grids)."""
import numpy as np
import pytest

from paper_2604_11959_gb300 import amr, inputs

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


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("n", [(4, 4, 4), (16, 8, 12), (17, 9, 13), (31, 17, 20), (33, 15, 9), (64, 48, 40)])
def test_automatic_split_steps_like_whole_columns(eb, precision, n):
    """The automatic split of the bulk kernel (16 x 8 tiles and short slabs on
    small FP64 domains) only changes who computes what: bit for bit the steps
    of whole columns of 32 x 16 tiles."""
    nx, ny, nz = n
    w = inputs.Workload("split", nx, ny, nz, 1, terrain="gaussian", hmax=0.1)
    refs = refs_for(nz, w.Lz)
    g = make_geometry(eb, w, w.heights(), precision, refs)
    U = to_device(w.state("sheltered", seed=3), precision, refs)
    auto = eb.step(g, U, w.dt(), 2, 3)
    eb.set_slab_levels(g, nz)
    whole = eb.step(g, U, w.dt(), 2, 3)
    for f in FIELDS:
        assert torch.equal(auto[f], whole[f]), (precision, n, f)
    eb.sync_status(g)


@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_covered_values_come_from_the_first_state(eb, precision):
    """Covered CVs and the w walls of the result are Un's, whatever the
    scratch states of several steps and stages hold."""
    w = inputs.Workload("static", 20, 18, 16, 1, terrain="grf", seed=2, hmax=0.2)
    refs = refs_for(w.nz, w.Lz)
    g = make_geometry(eb, w, w.heights(), precision, refs)
    U = to_device(w.state("sheltered", seed=1), precision, refs)
    wall = U["rhow"]
    wall[0], wall[-1] = 0.25, -0.5
    for nsteps, stages in ((1, 1), (3, 1), (1, 3), (2, 3)):
        V = eb.step(g, U, w.dt(), nsteps, stages)
        for f in FIELDS:
            cov = g.export(eb.FIELD_GRID[f], "alpha") <= 0
            assert torch.equal(V[f][cov], U[f][cov]), (f, nsteps, stages)
        assert torch.equal(V["rhow"][0], wall[0]) and torch.equal(V["rhow"][-1], wall[-1])


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("stages", [1, 3])
def test_steps_of_a_window_whose_ends_do_not_meet(eb, precision, stages):
    """The terrain jumps from the last column of the window to the first, so
    stencils across that seam read covered CVs: two steps in one call (scratch
    state between them) are bit for bit two calls (full states between them)."""
    w = inputs.Workload("seam", 24, 20, 16, 1, terrain="grf", seed=4, hmax=0.12)
    refs = refs_for(w.nz, w.Lz)
    h = w.heights() + np.linspace(0.0, 0.2, w.nx + 1)[None, :]
    U = to_device(w.state("uniform", pert=1e-2, seed=5), precision, refs)
    for nsteps in (2, 4):
        once = make_geometry(eb, w, h, precision, refs)
        got = eb.step(once, U, w.dt(), nsteps, stages)
        each = make_geometry(eb, w, h, precision, refs)
        want = U
        for _ in range(nsteps):
            want = eb.step(each, want, w.dt(), 1, stages)
        for f in FIELDS:
            assert torch.allclose(got[f], want[f], rtol=0.0, atol=0.0, equal_nan=True), (f, nsteps)


def test_patch_steps_beside_its_seam(eb):
    """Faces open on one side of a patch's seam and closed on the other have no
    flux, whatever the memory held that the fluxes are staged in: the mixed step
    of a patch on random terrain follows the FP64 step everywhere.  Float
    rounding of fluxes of order one over fields of order 1e-3 is 1e-4 of the
    fields' maximum; the bound is a hundred times that."""
    w = inputs.Workload("seam", 186, 98, 68, 1, terrain="grf")
    refs = w.references("sheltered")
    crefs = list(inputs.cell_reference(w.nz // 2, w.Lz)) + list(inputs.background_momentum(
        w.nz // 2, w.Lz, z_calm=w.hmax + w.Lz / w.nz, ramp=8 * w.Lz / w.nz))
    wc = inputs.Workload("coarse", w.nx // 2, w.ny // 2, w.nz // 2, 1, terrain="grf", hmax=w.hmax)
    out = {}
    for precision in ("mixed", "f64"):
        lv = amr.TwoLevel(eb, w.nx, w.ny, w.nz, w.Lx, w.Ly, w.Lz, w.heights(), 8, 76, amr.HALO_RK3,
                          precision=precision, refs_fine=refs, refs_coarse=crefs)
        Uc = to_device(wc.state("sheltered", seed=5), precision, crefs)
        Uf = lv.fill(Uc, lv.patch.empty_state())
        out[precision] = eb.step(lv.patch, Uf, w.dt(), 1, 1)
    for f in FIELDS:
        a, b = out["mixed"][f].double(), out["f64"][f]
        assert torch.isfinite(a).all(), f
        assert float((a - b).abs().max()) <= 1e-2 * float(b.abs().max()), f


@pytest.mark.parametrize("n", [(16, 16, 8), (20, 12, 8), (24, 36, 28), (50, 34, 18), (64, 32, 16), (144, 16, 16)])
def test_multigrid_reaches_the_jacobi_solution(eb, n):
    """V-cycles over grids with 4, 2 and 1 columns per thread, one or several
    levels in the single-block kernel: the same projected momenta as the Jacobi
    preconditioner.  Both solve to 1e-12, so each is within about 1e-12 times
    the condition number (a few thousand here) of the exact projection."""
    nx, ny, nz = n
    w = inputs.Workload("mg", nx, ny, nz, 1, terrain="grf", seed=7, hmax=0.15)
    refs = refs_for(nz, w.Lz)
    g = make_geometry(eb, w, w.heights(), "f64", refs)
    U = to_device(inputs.anelastic_state(w, seed=2), "f64", refs)
    out = []
    for kind in ("jacobi", "mg"):
        eb.set_preconditioner(g, kind)
        P = {f: U[f].clone() for f in U}
        it, res = eb.project(g, P, w.dt(), rtol=1e-12, maxit=3000)
        assert res <= 1e-12, (kind, it, res)
        out.append(P)
    scale = max(float(out[0][f].abs().max()) for f in ("rhou", "rhov", "rhow"))
    for f in ("rhou", "rhov", "rhow"):
        assert float((out[0][f] - out[1][f]).abs().max()) <= 1e-8 * scale, f


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("n,cols", [((8, 8, 8), (0, 8)), ((12, 10, 14), (2, 8)), ((66, 18, 10), (10, 56))])
def test_level_transfers_keep_uniform_states(eb, precision, n, cols):
    """Restriction and prolongation of a uniform full state (stored about
    different profiles per level) are that state: to 4 ulps of the stored
    value's profile in double, of the value itself in float."""
    nx, ny, nz = n
    w = inputs.Workload("lv", nx, ny, nz, 1, terrain="gaussian", hmax=0.1)
    rf, rc = refs_for(nz, w.Lz), refs_for(nz // 2, w.Lz)
    fine = make_geometry(eb, w, w.heights(), precision, rf)
    coarse = fine.coarse(*(torch.from_numpy(np.ascontiguousarray(r)).cuda() for r in rc))
    full = {"rho": 1.25, "rhotheta": 375.0, "rhou": 0.5, "rhov": -0.25, "rhow": 0.125}

    def state(g, refs):
        U = g.empty_state()
        for f, v in full.items():
            U[f].fill_(v)
            if f in ("rho", "rhotheta"):
                r = torch.from_numpy(np.ascontiguousarray(refs[f == "rhotheta"])).cuda()
                U[f].copy_((v - r)[:, None, None].expand(U[f].shape))
        return U

    Uf, Uc = state(fine, rf), state(coarse, rc)
    want_f, want_c = {f: t.clone() for f, t in Uf.items()}, {f: t.clone() for f, t in Uc.items()}
    eb.restrict(fine, coarse, Uf, Uc, 0, cols)
    eb.prolong(coarse, Uc, fine, Uf, 0, cols)
    eps = 2.0 ** -52 if precision == "f64" else 2.0 ** -23
    for f, v in full.items():
        for got, want in ((Uc[f], want_c[f]), (Uf[f], want_f[f])):
            scale = abs(v) if precision == "f64" else float(want.abs().max())
            assert float((got - want).abs().max()) <= 4 * eps * scale, f
