"""The helpers of fp64_roots.cuh, compiled here into a small library of their own and run on the device:
  - Root's square root and its inverse within two units in the last place, the reciprocal's bar: the hardware's
    approximation is good to 2^-19 or better and the third-order step leaves its cube, below 2^-57; x y is rounded once,
    which the step halves, and the result once, 1.5 * 2^-53 together;
  - rounded_to_float equal to the conversion bit for bit, and split_to_floats to h = (float)x, l = (float)(x - h), on ties,
    carries into the exponent, both signs, zeros, subnormals, the edges of the range and infinities (NaN stays NaN);
  - positive_normal and at_least_2_m14 equal to the comparisons they stand for."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2605_05543_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "fp64_roots.cuh"
using namespace emppp;
__global__ void k(const double* x, long long n, double* s, double* r, float* f, float* h, float* l, int* c) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Root q(x[i]);
  s[i] = q.sqrt();
  r[i] = q.rsqrt();
  f[i] = rounded_to_float(x[i]);
  split_to_floats(x[i], h[i], l[i]);
  c[i] = (positive_normal(x[i]) ? 1 : 0) | (at_least_2_m14(x[i]) ? 2 : 0);
}
extern "C" int run(const double* x, long long n, double* s, double* r, float* f, float* h, float* l, int* c) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(x, n, s, r, f, h, l, c);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("roots")
    src, lib = str(d / "roots.cu"), str(d / "libroots.so")
    open(src, "w").write(SOURCE)
    subprocess.run([_build._nvcc(), *_build.ARCH, *_build.FLAGS, "-Xcompiler", "-fvisibility=default", "-I", _build.CSRC,
                    "-shared", src, "-o", lib], check=True, capture_output=True)
    fn = ctypes.CDLL(lib).run
    fn.argtypes = [ctypes.c_void_p, ctypes.c_longlong] + [ctypes.c_void_p] * 6

    def call(x):
        xd = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        n = xd.numel()
        out = [torch.empty(n, dtype=t, device="cuda")
               for t in (torch.float64, torch.float64, torch.float32, torch.float32, torch.float32, torch.int32)]
        torch.cuda.synchronize()
        assert fn(xd.data_ptr(), n, *[o.data_ptr() for o in out]) == 0
        return [o.cpu().numpy() for o in out]

    return call


def doubles(rng, n, lo, hi):
    """Positive doubles of random significands with exponents lo .. hi - 1."""
    return np.ldexp(1.0 + rng.random(n), rng.integers(lo, hi, n))


def test_roots_within_two_ulp(run):
    rng = np.random.default_rng(3)
    x = np.concatenate([doubles(rng, 400000, -1021, 1022), doubles(rng, 400000, -120, 120),
                        np.ldexp(1.0, np.arange(-1020, 1021)), np.nextafter(np.ldexp(1.0, np.arange(-1020, 1021)), 0.0)])
    s, r = run(x)[:2]
    xl = x.astype(np.longdouble)
    root = np.sqrt(x)  # correctly rounded
    inv = (1 / np.sqrt(xl)).astype(np.float64)
    assert np.max(np.abs(s - root) / np.spacing(root)) <= 2.0
    assert np.max(np.abs(r - inv) / np.spacing(inv)) <= 2.0


def test_roundings_equal_the_conversion(run):
    rng = np.random.default_rng(4)
    m = np.concatenate([np.arange(8), (1 << 23) - 1 - np.arange(8), rng.integers(0, 1 << 23, 4000)])  # FP32 significands
    tie = np.array([0, 1, (1 << 28) - 1, 1 << 28, (1 << 28) + 1, (1 << 29) - 1])  # what FP32 drops
    frac = (m[:, None] << 29 | tie[None]).ravel().astype(np.float64) / 2.0 ** 52
    x = [np.ldexp(1.0 + frac, e) for e in (0, 1, -1, 30, 127, 126, -75, -74, -73, -126, -127, -140, -149, -150, -160, 128, -1022)]
    x += [doubles(rng, 2000000, -200, 140), doubles(rng, 200000, -80, -68)]
    x += [np.array([0.0, np.inf, 5e-324, 2.0 ** -1030, np.finfo(np.float32).max, np.nextafter(np.finfo(np.float32).max, np.inf, dtype=np.float64),
                    (2.0 - 2.0 ** -24) * 2.0 ** 127, np.nextafter((2.0 - 2.0 ** -24) * 2.0 ** 127, 0.0)])]
    x = np.concatenate(x)
    x = np.concatenate([x, -x])
    _, _, f, h, l, _ = run(x)
    bits = lambda a: a.view(np.uint32)  # noqa: E731
    with np.errstate(over="ignore", invalid="ignore"):
        ref = x.astype(np.float32)
        low = (x - ref.astype(np.float64)).astype(np.float32)
    assert np.array_equal(bits(f), bits(ref)) and np.array_equal(bits(h), bits(ref))
    inf = np.isinf(ref)
    assert np.array_equal(l[~inf] == 0, low[~inf] == 0)
    some = ~inf & (low != 0)  # (a zero's sign means nothing)
    assert np.array_equal(bits(l[some]), bits(low[some]))
    nan = run(np.array([np.nan, -np.nan]))
    assert np.all(np.isnan(nan[2])) and np.all(np.isnan(nan[3]))


def test_comparisons(run):
    rng = np.random.default_rng(5)
    e = 2.0 ** -14
    x = np.concatenate([doubles(rng, 200000, -1021, 1023), doubles(rng, 200000, -18, -10), [e, np.nextafter(e, 0.0)],
                        [0.0, 5e-324, 2.0 ** -1022, np.nextafter(2.0 ** -1022, 0.0), np.finfo(np.float64).max]])
    x = np.concatenate([x, -x, [np.inf, -np.inf, np.nan]])
    c = run(x)[5]
    finite = np.isfinite(x)
    assert np.array_equal((c & 1) != 0, finite & (x >= 2.0 ** -1022))
    assert np.array_equal((c[finite] & 2) != 0, x[finite] >= e)
