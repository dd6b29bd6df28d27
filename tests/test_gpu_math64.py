"""rcp_pos, rsqrt_pos, sqrt_pos and the integer minima and maxima of csrc/dg_math64.cuh against extended precision,
over all exponents and at the edges of their branches.

Bounds.  Reciprocal: the step leaves e0^3 < 2^-63 and one rounding of the result: 1 ulp.  Roots: x y (or the root
itself) is rounded once before the step, which halves that error, and the result is rounded once: 2 ulp.  Arguments
outside the positive normal range go to CUDA's functions (reciprocal and root correctly rounded, rsqrt within 2 ulp).
"""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_2301_11238_gb300 import build

pytestmark = pytest.mark.gpu

PROBE = """
#include "dg_math64.cuh"
using namespace dgswe;
__global__ void unary(int n, const double* x, double* y, int op) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = op == 0 ? rcp_pos(x[i]) : op == 1 ? rsqrt_pos(x[i]) : sqrt_pos(x[i]);
}
__global__ void binary(int n, const double* x, const double* z, double* y, int op) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = op == 0 ? min_f64(x[i], z[i]) : op == 1 ? max_f64(x[i], z[i]) : max_pos(x[i], z[i]);
}
extern "C" int run1(int n, const double* x, double* y, int op) {
  unary<<<(n + 127) / 128, 128>>>(n, x, y, op);
  return (int)cudaDeviceSynchronize();
}
extern "C" int run2(int n, const double* x, const double* z, double* y, int op) {
  binary<<<(n + 127) / 128, 128>>>(n, x, z, y, op);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def probe(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tmp_path_factory.mktemp("probe")
    (d / "p.cu").write_text(PROBE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", str(d / "p.cu"), "-o",
                    str(d / "p.so")], check=True)
    lib = C.CDLL(str(d / "p.so"))

    def call(op, *args):
        t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in args]
        y = torch.empty_like(t[0])
        torch.cuda.synchronize()
        f = lib.run1 if len(t) == 1 else lib.run2
        assert f(len(y), *[C.c_void_p(a.data_ptr()) for a in t], C.c_void_p(y.data_ptr()), op) == 0
        return y.cpu().numpy()

    return call


def arguments():
    """Positive normal values: random mantissas at every exponent, mantissas next to 1 and 2, powers of two."""
    rng = np.random.default_rng(0)
    e = np.arange(-1022, 1024)
    m = np.concatenate([1 + rng.random((64, e.size)), np.broadcast_to(
        np.array([1, 1 + 2.0 ** -52, 1 + 2.0 ** -24, 1 + 2.0 ** -23, 1.5, 2 - 2.0 ** -23, 2 - 2.0 ** -52])[:, None],
        (7, e.size))])
    return np.ldexp(m, e).ravel()


def exact(op, x):
    x = x.astype(np.longdouble)
    return (1 / x, 1 / np.sqrt(x), np.sqrt(x))[op]


@pytest.mark.parametrize("op,ulps", [(0, 1.0), (1, 2.0), (2, 2.0)])
def test_positive_normal(probe, op, ulps):
    x = arguments()
    y, r = probe(op, x), exact(op, x)
    ulp = np.spacing(np.abs(r).astype(np.float64)).astype(np.longdouble)
    err = np.abs(y.astype(np.longdouble) - r) / ulp
    assert err.max() <= ulps, (x[err.argmax()].hex(), float(err.max()))


@pytest.mark.parametrize("op", [0, 1, 2])
def test_other_arguments(probe, op):
    tiny = 2.0 ** -1022
    x = np.array([0.0, 5e-324, tiny / 2, tiny * (1 - 2.0 ** -52), np.inf, -1.0, -tiny, -np.inf, np.nan])
    with np.errstate(all="ignore"):
        y, r = probe(op, x), exact(op, x).astype(np.float64)
    both_nan = np.isnan(y) & np.isnan(r)
    same = (y == r) | both_nan | (np.abs(y - r) <= 2 * np.spacing(np.abs(r)))
    assert same.all(), list(zip(x, y, r))


def test_minima_and_maxima(probe):
    tiny = 5e-324
    v = np.array([-np.inf, -1e300, -2.0, -1.0 - 2.0 ** -52, -1.0, -tiny, -0.0, 0.0, tiny, 1.0, 1.0 + 2.0 ** -52, 1e300, np.inf])
    rng = np.random.default_rng(1)
    v = np.concatenate([v, np.ldexp(rng.uniform(-1, 1, 60), rng.integers(-1000, 1000, 60))])
    x, z = (a.ravel().copy() for a in np.meshgrid(v, v))
    assert np.array_equal(probe(0, x, z), np.minimum(x, z))
    assert np.array_equal(probe(1, x, z), np.maximum(x, z))
    pos = z > 0
    assert np.array_equal(probe(2, x[pos], z[pos]), np.maximum(x[pos], z[pos]))
