"""div_by (csrc/rf_common.cuh), the quotient of the assembly, the inverse diagonal
blocks and the FP16 storage, against the device's division: equal to the last bit,
zeros' signs included, for operands from all of the FP64 range — exponents at
random, mantissas at random and at the ends of a binade, the neighbourhood of
exact quotients and of the places where a step would under- or overflow, zeros,
infinities and NaN."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SOURCE = r"""
#include "rf_common.cuh"
__global__ void k(long long n, const double* x, const double* h, double* got, double* want) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= n) return;
  got[t] = rf::div_by(x[t], h[t], rf::recip(h[t]));
  want[t] = __ddiv_rn(x[t], h[t]);
}
extern "C" int quotients(long long n, const double* x, const double* h, double* got, double* want) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(n, x, h, got, want);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def quotients(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2506_04763_gb300 import build as B
    d = tmp_path_factory.mktemp("quotient")
    (d / "q.cu").write_text(SOURCE)
    so = str(d / "q.so")
    subprocess.run([B.nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", B.INCLUDE, "-I", B.CSRC,
                    "-o", so, str(d / "q.cu")] + B.ARCH, check=True)
    fn = ctypes.CDLL(so).quotients
    fn.argtypes = [ctypes.c_longlong] + [ctypes.c_void_p] * 4
    torch.zeros(1, device="cuda")

    def run(x, h):
        X, H = (torch.tensor(np.asarray(t, np.float64), device="cuda") for t in (x, h))
        got, want = torch.empty_like(X), torch.empty_like(X)
        torch.cuda.synchronize()
        assert fn(X.numel(), X.data_ptr(), H.data_ptr(), got.data_ptr(), want.data_ptr()) == 0
        return got.cpu().numpy(), want.cpu().numpy()
    return run


def _same(got, want):
    return (got.view(np.int64) == want.view(np.int64)) | (np.isnan(got) & np.isnan(want))


def _numbers(rng, n, lo, hi):
    """Random signs, exponents in [lo, hi], mantissas random or next to a power of two."""
    m = 1.0 + rng.random(n)
    kind = rng.integers(0, 6, n)
    m[kind == 0] = 1.0
    m[kind == 1] = 2.0 - 2.0 ** -52
    m[kind == 2] = 1.0 + 2.0 ** -52
    with np.errstate(over="ignore", under="ignore"):
        return np.ldexp(m, rng.integers(lo, hi + 1, n)) * rng.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("xr,hr", [((-30, 30), (-30, 30)), ((-1074, 1023), (-1074, 1023)), ((-1030, -900), (-70, 70)),
                                   ((900, 1023), (-70, 70)), ((880, 980), (-1023, -900)), ((-70, 70), (900, 1023)),
                                   ((-70, 70), (-1074, -900))])
def test_quotients_equal_the_division(quotients, xr, hr):
    rng = np.random.default_rng([xr[0] + 2000, hr[0] + 2000])
    n = 1 << 20
    x, h = _numbers(rng, n, *xr), _numbers(rng, n, *hr)
    got, want = quotients(x, h)
    bad = ~_same(got, want)
    assert not bad.any(), (x[bad][:4], h[bad][:4], got[bad][:4], want[bad][:4])


def test_near_exact_quotients_and_special_values(quotients):
    rng = np.random.default_rng(3)
    n = 1 << 20
    h, q = _numbers(rng, n, -20, 20), _numbers(rng, n, -20, 20)
    x = h * q
    x = np.nextafter(x, rng.choice([-np.inf, np.inf], n))
    got, want = quotients(x, h)
    assert _same(got, want).all()
    s = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 1.0, -3.0, 5e-324, -5e-324, 2.0 ** -1022, 1.7976931348623157e308,
                  2.0 ** -959, 2.0 ** 959, 1e-200, 1e200])
    x, h = (t.ravel() for t in np.meshgrid(s, s))
    got, want = quotients(x, h)
    bad = ~_same(got, want)
    assert not bad.any(), list(zip(x[bad], h[bad], got[bad], want[bad]))
