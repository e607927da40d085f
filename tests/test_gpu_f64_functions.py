"""The FP64 path's own reciprocal, roots, quotient and logarithm, each by
itself over its range: units in the last place against extended precision.
The bars are the roundings and the truncation of each one's last steps."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = '''
#include "qs_device.cuh"
__global__ void k(int f, const double* a, const double* b, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = f == 0 ? qs::rcp_d(a[i]) : f == 1 ? qs::rsqrt_d(a[i]) : f == 2 ? qs::div_d(a[i], b[i])
       : f == 3 ? qs::icbrt_d(a[i]) : qs::log_d(a[i]);
}
extern "C" int run(int f, const double* a, const double* b, double* y, int n) {
  k<<<(n + 255) / 256, 256>>>(f, a, b, y, n);
  return (int)cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def fn(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).eps > 2.0 ** -60:
        pytest.skip("no extended precision")
    from paper_2308_09348_gb300 import build
    d = tmp_path_factory.mktemp("f64")
    (d / "f.cu").write_text(SOURCE)
    lib = str(d / "f.so")
    subprocess.run(["nvcc", *build.ARCH, *build.FLAGS, "-I", build.INCLUDE, "-I", build.CSRC,
                    "-shared", str(d / "f.cu"), "-o", lib], check=True, capture_output=True)
    h = C.CDLL(lib)

    def run(f, a, b=None):
        a, b = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, a if b is None else b))
        y = torch.empty_like(a)
        torch.cuda.synchronize()
        assert h.run(f, *(C.c_void_p(t.data_ptr()) for t in (a, b, y)), a.numel()) == 0
        return y.cpu().numpy()

    return run


def _ulps(got, exact):
    e = exact.astype(np.longdouble)
    unit = np.spacing(np.abs(e).astype(np.float64)).astype(np.longdouble)
    return float(np.max(np.abs(got.astype(np.longdouble) - e) / unit))


def _sweep(lo, hi, seed):
    """Exponents lo..hi: random mantissas, powers of two and their neighbours."""
    rg = np.random.default_rng(seed)
    x = np.ldexp(rg.uniform(1.0, 2.0, 400000), rg.integers(lo, hi, 400000))
    p = np.ldexp(1.0, np.arange(lo, hi))
    x = np.concatenate([x, p, np.nextafter(p, np.inf), np.nextafter(2 * p, 0)])
    return x[(x >= np.ldexp(1.0, lo)) & (x < np.ldexp(1.0, hi))]


ONE = np.longdouble(1)


def test_reciprocal(fn):
    x = np.concatenate([_sweep(-1021, 1021, 1), _sweep(-2, 3, 2)])
    x = np.concatenate([x, -x])
    # the last operation's half unit, and e^3 (2^-57)
    u = _ulps(fn(0, x), ONE / x.astype(np.longdouble))
    print("rcp", u)
    assert u <= 1.0
    with np.errstate(divide="ignore"):
        s = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
        np.testing.assert_array_equal(fn(0, s), 1.0 / s)


def test_reciprocal_root(fn):
    x = np.concatenate([_sweep(-1021, 1021, 3), _sweep(-2, 3, 4)])
    # half a unit each of the last operation and (by half) of x y, 5 e^3 / 16
    u = _ulps(fn(1, x), ONE / np.sqrt(x.astype(np.longdouble)))
    print("rsqrt", u)
    assert u <= 2.0
    got = fn(1, np.array([0.0, np.inf, np.nan, -1.0]))
    assert got[0] == np.inf and got[1] == 0.0 and np.isnan(got[2:]).all()


def test_quotient(fn):
    rg = np.random.default_rng(5)
    b = _sweep(0, 500, 6)
    a = np.ldexp(rg.uniform(1.0, 2.0, b.size), rg.integers(-400, 400, b.size))
    u = _ulps(fn(2, a, b), a.astype(np.longdouble) / b.astype(np.longdouble))
    print("div", u)
    assert u <= 1.0
    np.testing.assert_array_equal(fn(2, a, np.ones_like(a)), a)       # exact
    with np.errstate(divide="ignore", invalid="ignore"):
        a = np.array([1.0, 1.0, -1.0, 0.0, np.inf, 1.0])
        b = np.array([0.0, np.inf, np.inf, 0.0, np.inf, np.nan])
        np.testing.assert_array_equal(fn(2, a, b), a / b)


@pytest.mark.parametrize("lo,hi", [(0, 1), (1, 20), (20, 127), (127, 1020)])
def test_reciprocal_cube_root(fn, lo, hi):
    x = _sweep(lo, hi, 7 + lo)
    # half a unit of the last operation, two thirds of the cube's two products,
    # 14 e^3 / 81; beyond the FP32 range CUDA's exp2(-log2(x) / 3): the rounded
    # logarithm (up to 1020 / 3, half a unit in 2^-45) times ln 2
    u = _ulps(fn(3, x), ONE / np.cbrt(x.astype(np.longdouble)))
    print("icbrt", lo, hi, u)
    assert u <= (2.5 if hi <= 127 else 512.0)
    got = fn(3, np.array([np.inf, np.nan, 1.0]))
    assert got[0] == 0.0 and np.isnan(got[1]) and got[2] == 1.0


def test_logarithm(fn):
    edges = 1.0 + np.arange(1024) / 1024.0              # the table's intervals
    x = np.concatenate([_sweep(0, 1023, 8), _sweep(0, 1, 9), edges, np.nextafter(edges, 3.0),
                        np.nextafter(edges[1:], 0.0), 1.0 + np.ldexp(1.0, -np.arange(1, 53))])
    ref = np.log(x.astype(np.longdouble))
    err = np.abs(fn(4, x).astype(np.longdouble) - ref) / np.maximum(ref, 1)
    print("log", float(err.max()) * 2.0 ** 52, "2^-52")
    assert float(err.max()) <= 2.0 ** -52
