"""Restriction and prolongation over regular cells: the double mean of the
values plus the double difference of the levels' profiles, rounded once to the
state's precision, whatever the values are (eb_restrict: "Sums in double").
The lowest level of a flat floor holds records: its restriction weights every
fine value (other tests), so it is left out here."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

FIELDS = ("rho", "rhotheta", "rhou", "rhov", "rhow")
NX, NY, NZ = 24, 20, 16


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_11959_gb300 import eb as _eb
    _eb.load(build_if_missing=True)
    return _eb


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def profiles(nz, seed):
    """Four profiles: rho0, rho0 theta0, background rho*u and rho*v."""
    z = (np.arange(nz) + 0.5) / nz
    rng = np.random.default_rng(seed)
    return [1.2 * np.exp(-z), 360.0 * np.exp(-0.9 * z), 0.7 * z + 0.01 * rng.random(nz), np.zeros(nz)]


def levels(eb, precision):
    """A flat fine level and the coarse level merged from it."""
    pf, pc = profiles(NZ, 1), profiles(NZ // 2, 2)
    fine = eb.Geometry(NX, NY, NZ, 1.0, 1.0, 0.5, cuda(np.zeros((NY + 1, NX + 1))), precision=precision,
                       ref_rho=cuda(pf[0]), ref_rhotheta=cuda(pf[1]), ref_rhou=cuda(pf[2]), ref_rhov=cuda(pf[3]))
    coarse = fine.coarse(cuda(pc[0]), cuda(pc[1]))
    coarse.set_wind_reference(cuda(pc[2]), cuda(pc[3]))
    zf, zc = np.zeros(NZ + 1), np.zeros(NZ // 2 + 1)
    return fine, coarse, [*pf, zf], [*pc, zc]


def values(shape, kind, rng, dtype):
    """Values of one kind: smooth perturbations; magnitudes over fourteen
    decades with both signs (sums that cancel); all equal; zeros; the smallest
    numbers; the largest, with infinities and NaN among them."""
    if kind == "smooth":
        a = 1e-2 * np.sin(np.arange(int(np.prod(shape))) * 0.37).reshape(shape) + 1e-4 * rng.standard_normal(shape)
    elif kind == "spread":
        a = rng.standard_normal(shape) * 10.0 ** rng.uniform(-7, 7, shape)
    elif kind == "equal":
        a = np.full(shape, 0.1)
    elif kind == "zero":
        a = np.zeros(shape)
    elif kind == "tiny":
        a = rng.standard_normal(shape) * (1e-38 if dtype == np.float32 else 1e-308)
    else:
        big = np.finfo(dtype).max
        a = rng.choice([0.3, 0.9], shape) * (big if kind == "huge" else 1.0)
        if kind == "special":
            p = rng.random(shape)
            a = np.where(p < 0.02, np.inf, np.where(p < 0.04, -np.inf, np.where(p < 0.05, np.nan, a)))
    return a.astype(dtype)


def mean(parts):
    s = parts[0].astype(np.float64)
    for p in parts[1:]:
        s = s + p.astype(np.float64)
    return s * (1.0 / len(parts))


def restricted(f, u, pf, pc):
    """The coarse field from the fine one (the lid face of rhow left out)."""
    n = pc.size if f != "rhow" else NZ // 2
    b0, b1 = u[0:2 * n:2], u[1:2 * n:2]
    at = lambda b, y, x: b[:, y::2, x::2]
    parts = {"rho": [at(b, y, x) for b in (b0, b1) for y in (0, 1) for x in (0, 1)],
             "rhou": [at(b, y, 0) for b in (b0, b1) for y in (0, 1)],
             "rhov": [at(b, 0, x) for b in (b0, b1) for x in (0, 1)],
             "rhow": [at(b0, y, x) for y in (0, 1) for x in (0, 1)]}
    parts["rhotheta"] = parts["rho"]
    d = 0.5 * (pf[0:2 * n:2] + pf[1:2 * n:2]) - pc[:n] if f != "rhow" else np.zeros(n)
    return mean(parts[f]) + d[:, None, None]


def prolonged(f, u, pf, pc):
    """The fine field from the coarse one."""
    axis = {"rhou": 2, "rhov": 1, "rhow": 0}.get(f)
    nk = NZ + (f == "rhow")
    k, j, i = np.arange(nk), np.arange(NY), np.arange(NX)
    low = u[np.ix_(k // 2, j // 2, i // 2)]
    out = low.astype(np.float64)
    if axis is not None:
        idx = [k // 2, j // 2, i // 2]
        # (an odd rhow level always has a level above it)
        idx[axis] = np.minimum(idx[axis] + 1, u.shape[0] - 1) if axis == 0 else (idx[axis] + 1) % u.shape[axis]
        odd = ((k, j, i)[axis] % 2 == 1).reshape([-1 if a == axis else 1 for a in range(3)])
        out = np.where(odd, mean([low, u[np.ix_(*idx)]]), out)
    d = pc[np.arange(nk) // 2] - pf[:nk]
    return out + d[:, None, None]


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("kind", ["smooth", "spread", "equal", "zero", "tiny", "huge", "special"])
def test_transfers_round_the_double_means_once(eb, precision, kind):
    dtype = np.float64 if precision == "f64" else np.float32
    fine, coarse, pf, pc = levels(eb, precision)
    rng = np.random.default_rng(3)
    Uf, Uc = fine.empty_state(), coarse.empty_state()
    hf = {f: values(tuple(Uf[f].shape), kind, rng, dtype) for f in FIELDS}
    hc = {f: values(tuple(Uc[f].shape), kind, rng, dtype) for f in FIELDS}
    for f in FIELDS:
        Uf[f].copy_(torch.from_numpy(hf[f]))
        Uc[f].copy_(torch.from_numpy(hc[f]))
    R, P = {f: Uc[f].clone() for f in FIELDS}, {f: Uf[f].clone() for f in FIELDS}
    eb.restrict(fine, coarse, Uf, R)
    eb.prolong(coarse, Uc, fine, P)
    with np.errstate(all="ignore"):
        for q, f in enumerate(FIELDS):
            want = restricted(f, hf[f], pf[q], pc[q]).astype(dtype)
            assert np.array_equal(R[f].cpu().numpy()[1:NZ // 2], want[1:], equal_nan=True), f
            want = prolonged(f, hc[f], pf[q], pc[q]).astype(dtype)
            assert np.array_equal(P[f].cpu().numpy(), want, equal_nan=True), f
    fine.close()
    coarse.close()
