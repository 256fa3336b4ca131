"""Kernel variants that only larger grids reach, on grids just large enough for
them on a GPU of 152 SMs."""
import numpy as np
import pytest

from paper_2604_11959_gb300 import inputs

from _gpu_helpers import FIELDS, make_geometry, refs_for, to_device

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the sizes are for 152 SMs")
    from paper_2604_11959_gb300 import eb as _eb
    _eb.load(build_if_missing=True)
    return _eb


# sweeps of four columns per thread (from 155,648 cells, columns a multiple of
# four), with ragged blocks; of two columns, over a coarsest grid of 65x25x13 =
# 21,125 cells that runs from global memory; a second level of two columns; and
# the restriction of two coarse levels per thread (from 10 million cells)
@pytest.mark.parametrize("n", [(96, 96, 48), (100, 108, 56), (130, 50, 26), (260, 100, 52), (320, 256, 128)])
@pytest.mark.parametrize("precision", ["f64", "mixed"])
def test_multigrid_of_wide_sweeps_reaches_the_jacobi_solution(eb, n, precision):
    """Both preconditioners solve to 1e-12 of the right-hand side b.  In the
    2-norm the momenta of each are then within 1e-12 |b| L / (2 pi) of the exact
    projection (the longest wave has the smallest eigenvalue), and |b| is at most
    2 sqrt(3) / dx times the input momenta's norm: together 1.1e-12 per column
    of the domain and solve, 7e-10 at 320 columns, doubled for the terrain.  In
    float a corrected momentum is rounded once in each: one part in 2^24."""
    nx, ny, nz = n
    w = inputs.Workload("mg", nx, ny, nz, 1, terrain="grf", seed=7, hmax=0.15)
    refs = refs_for(nz, w.Lz)
    g = make_geometry(eb, w, w.heights(), precision, refs)
    U = to_device(inputs.anelastic_state(w, seed=2), precision, refs)
    mom = ("rhou", "rhov", "rhow")
    norm = sum(float(U[f].double().square().sum()) for f in mom) ** 0.5
    out = []
    for kind in ("jacobi", "mg"):
        eb.set_preconditioner(g, kind)
        P = {f: U[f].clone() for f in U}
        it, res = eb.project(g, P, w.dt(), rtol=1e-12, maxit=6000)
        assert res <= 1e-12, (kind, it, res)
        out.append((it, P))
    assert out[1][0] < out[0][0] / 4
    diff = sum(float((out[0][1][f].double() - out[1][1][f].double()).square().sum()) for f in mom) ** 0.5
    bound = 2 * 2 * 1.1e-12 * max(nx, ny) + (2.0 ** -24 if precision == "mixed" else 0.0)
    assert diff <= bound * norm, (diff / norm, bound)
    g.close()


@pytest.mark.parametrize("precision", ["f64", "mixed"])
@pytest.mark.parametrize("n", [(250, 190, 41), (256, 192, 64), (129, 300, 50)])
def test_tall_automatic_slabs_step_like_whole_columns(eb, precision, n):
    """Where tiles times slabs fill the SMs the automatic split takes slabs of
    more than eight levels: bit for bit the steps of whole columns."""
    nx, ny, nz = n
    w = inputs.Workload("split", nx, ny, nz, 1, terrain="gaussian", hmax=0.1)
    refs = refs_for(nz, w.Lz)
    g = make_geometry(eb, w, w.heights(), precision, refs)
    U = to_device(w.state("sheltered", seed=3), precision, refs)
    auto = eb.step(g, U, w.dt(), 1, 3)
    eb.set_slab_levels(g, nz)
    whole = eb.step(g, U, w.dt(), 1, 3)
    for f in FIELDS:
        assert torch.equal(auto[f], whole[f]), (precision, n, f)
    eb.sync_status(g)
    g.close()


def conv(x, layers, q, relu=True):
    W, b = layers[q]
    y = torch.nn.functional.conv3d(x, W, b, padding=W.shape[-1] // 2)
    return torch.relu(y) if relu else y


def network(x, layers):
    """The network of oracle/unet.py in torch operations, (1, 2, nz, ny, nx) in."""
    pool = lambda t: torch.nn.functional.avg_pool3d(t, 2)
    up = lambda t: torch.nn.functional.interpolate(t, scale_factor=2, mode="nearest")
    e1 = conv(conv(x, layers, 0), layers, 1)
    e2 = conv(conv(pool(e1), layers, 2), layers, 3)
    bt = conv(conv(pool(e2), layers, 4), layers, 5)
    d2 = conv(conv(torch.cat([up(bt), e2], 1), layers, 6), layers, 7)
    d1 = conv(conv(torch.cat([up(d2), e1], 1), layers, 8), layers, 9)
    return conv(d1, layers, 10, relu=False)


def test_four_level_convolution_tiles_match_torch(eb):
    """132 x 132 x 52 voxels: both finer levels of the network have the 304
    tiles of 8 x 16 x 4 voxels (two per SM) from which the convolutions of 16
    and 32 channels take four levels per tile; every edge is ragged but the
    finest level's top.  Forward pass and every layer's gradient against FP64
    torch, with the tolerances of the smaller grids' tests."""
    from oracle import unet as un
    shape = (52, 132, 132)
    rng = np.random.default_rng(6)
    p = (un.init_params(6) * 0.7 + 0.02 * rng.standard_normal(un.num_params())).astype(np.float32)
    x = torch.from_numpy(rng.standard_normal((2,) + shape)).float().cuda()
    t = torch.from_numpy(rng.standard_normal(shape)).float().cuda()
    mask = torch.from_numpy((rng.uniform(size=shape) > 0.25).astype(np.float32)).cuda()
    net = eb.UNet(shape[2], shape[1], shape[0])
    net.set_params(p)
    y = net.forward(x)
    loss, g = net.gradient(x, t, mask)
    net.sync_status()
    layers, o = [], 0
    for ci, co, k in un.LAYERS:   # BF16 weights, FP32 biases
        n = co * ci * k ** 3
        W = torch.from_numpy(p[o:o + n]).bfloat16().double().reshape(co, ci, k, k, k).cuda().requires_grad_()
        b = torch.from_numpy(p[o + n:o + n + co]).double().cuda().requires_grad_()
        layers.append((W, b))
        o += n + co
    want = network(x.double()[None], layers)[0, 0]
    ref = want.detach()
    assert float((y.double() - ref).abs().max()) <= 1e-4 * float(ref.abs().max())
    L = 0.5 * (mask.double() * (want - t.double()).square()).sum() / mask.double().sum()
    L.backward()
    assert abs(loss - L.item()) <= 1e-4 * L.item()
    got = torch.from_numpy(np.asarray(g)).double()
    parts = [q.grad.reshape(-1).cpu() for pair in layers for q in pair]
    whole = torch.cat(parts)
    assert float((got - whole).norm()) <= 1e-3 * float(whole.norm())
    for part, mine in zip(parts, torch.split(got, [q.numel() for q in parts])):
        assert float((mine - part).norm()) <= 5e-3 * float(part.norm()) + 1e-12, part.numel()
    net.close()
