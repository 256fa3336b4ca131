"""The bulk kernel's double reciprocal (prcp in csrc/eb_bulk.cuh) is the
correctly rounded quotient 1.0 / a of the host's IEEE division, bit for bit,
over every exponent."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "eb_bulk.cuh"
__global__ void k(const double *a, double *o, long long n) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < n) o[t] = bulk::prcp(make_double2(a[t], 1.0)).x;
}
extern "C" int reciprocals(const double *a, double *o, long long n) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(a, o, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def reciprocals(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2604_11959_gb300 import build
    d = tmp_path_factory.mktemp("rcp")
    src, lib = str(d / "rcp.cu"), str(d / "librcp.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", "-fmad=false", "-Xcompiler", "-fPIC", *build.ARCH, "-I",
                    build.CSRC, "-I", os.path.join(build.HERE, "..", "include"), "-shared", "-o", lib, src], check=True)
    fn = ctypes.CDLL(lib).reciprocals
    fn.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]

    def run(a):
        x = torch.from_numpy(np.ascontiguousarray(a)).cuda()
        o = torch.empty_like(x)
        torch.cuda.synchronize()
        assert fn(x.data_ptr(), o.data_ptr(), x.numel()) == 0
        return o.cpu().numpy()

    return run


def bits(sign, exponent, mantissa):
    return ((np.uint64(sign) << np.uint64(63)) | (exponent.astype(np.uint64) << np.uint64(52)) |
            mantissa.astype(np.uint64)).view(np.float64)


def check(run, a):
    with np.errstate(all="ignore"):
        want = 1.0 / a
    got = run(a)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    bad = np.flatnonzero((got.view(np.uint64) != want.view(np.uint64)) & ~nan)
    assert bad.size == 0, (bad.size, a[bad[:4]].tolist(), got[bad[:4]].tolist(), want[bad[:4]].tolist())


def test_every_exponent(reciprocals):
    """Zeros, subnormals, all 2046 normal exponents, infinities and NaN of
    both signs: random significands, the smallest ones, the largest ones (whose
    reciprocals lie closest to a rounding boundary) and single bits."""
    rng = np.random.default_rng(1)
    top = (1 << 52) - 1
    edge = np.array([0, 1, 2, 3, top, top - 1, top - 2] + [1 << b for b in range(52)] +
                    [top - (1 << b) for b in range(52)], dtype=np.uint64)
    for sign in (0, 1):
        for man in (edge, rng.integers(0, 1 << 52, 2000, dtype=np.uint64)):
            e, m = np.meshgrid(np.arange(2048, dtype=np.uint64), man, indexing="ij")
            check(reciprocals, bits(sign, e.ravel(), m.ravel()))


def test_many_significands(reciprocals):
    """Sixty-four million random significands of one binade."""
    rng = np.random.default_rng(2)
    for _ in range(8):
        m = rng.integers(0, 1 << 52, 1 << 23, dtype=np.uint64)
        check(reciprocals, bits(0, np.full_like(m, 1023), m))
