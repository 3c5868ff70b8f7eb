"""The pivots' reciprocal (csrc/front.cuh: front_rcp) against CUDA's division, in a kernel of its own
compiled here: every value of the 20 mantissa bits that the hardware's estimate reads, every exponent
of its range, both signs.

Bounds.  The estimate truncates its argument and its result to 20 bits of mantissa: |1 - d y| <=
2 2^-20 = 2^-19.  One third-order step leaves out e^3 <= 2^-57 of the value, its two inner roundings
add less than 2^-70, its last one half an ulp; an ulp is more than 2^-53 and at most 2^-52 of the
value.  So |1 - d r| <= (1/2 + 2^-57 2^53) 2^-52 < 0.57 2^-52 (a fused multiply-add gives that residual
exactly), and r is 1 / d rounded to nearest or its neighbour."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1703_10435_gb300", "csrc")
SHIM = r'''
#include "front.cuh"
__global__ void k_check(const double* d, long long n, double* est, double* res, long long* ulp, int* ok) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double x = d[i], r = mhm::front_rcp(x);
        double y;
        asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
        est[i] = fma(-x, y, 1.0);
        res[i] = fma(-x, r, 1.0);
        ulp[i] = __double_as_longlong(r) - __double_as_longlong(1.0 / x);
        ok[i] = mhm::front_positive(x);
    }
}
extern "C" int check(const double* d, long long n, double* est, double* res, long long* ulp, int* ok) {
    k_check<<<1024, 256>>>(d, n, est, res, ulp, ok);
    return cudaDeviceSynchronize();
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1703_10435_gb300 import build
    nvcc = build._nvcc()
    if not (os.path.exists(nvcc) or shutil.which(nvcc)):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("rcp")
    (d / "shim.cu").write_text(SHIM)
    so = str(d / "librcp.so")
    subprocess.check_call([nvcc, *build.ARCH, *build.FLAGS, "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-shared", "-o",
                           so, str(d / "shim.cu")])
    return ctypes.CDLL(so)


def _check(lib, bits):
    d = torch.as_tensor(bits.view(np.float64), device="cuda")
    n = d.numel()
    est, res = torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
    ulp, ok = torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    p = lambda t: ctypes.c_void_p(t.data_ptr())
    assert lib.check(p(d), ctypes.c_longlong(n), p(est), p(res), p(ulp), p(ok)) == 0
    return est, res, ulp, ok.cpu().numpy()


def _bounds(lib, bits):
    est, res, ulp, ok = _check(lib, bits)
    assert float(est.abs().max()) <= 2.0 ** -19
    assert float(res.abs().max()) <= 0.57 * 2.0 ** -52
    assert int(ulp.abs().max()) <= 1
    assert np.array_equal(ok != 0, bits >> np.uint64(63) == 0)


@pytest.mark.parametrize("exponent", [-1022, -1, 0, 1, 1020])
@pytest.mark.parametrize("low", ["zero", "ones", "random"])
def test_every_mantissa_the_estimate_reads(lib, exponent, low):
    hi = np.arange(2 ** 20, dtype=np.uint64) << np.uint64(32)
    lo = {"zero": np.zeros(2 ** 20, np.uint64), "ones": np.full(2 ** 20, 0xffffffff, np.uint64),
          "random": np.random.default_rng(exponent + 2000).integers(0, 2 ** 32, 2 ** 20, dtype=np.uint64)}[low]
    bits = np.uint64(exponent + 1023) << np.uint64(52) | hi | lo
    _bounds(lib, bits)
    _bounds(lib, bits | np.uint64(1) << np.uint64(63))


def test_every_exponent(lib):
    rng = np.random.default_rng(1)
    e = np.repeat(np.arange(1, 2044, dtype=np.uint64), 2048)   # 2^-1022 .. 2^1020
    m = rng.integers(0, 2 ** 52, e.size, dtype=np.uint64)
    m[::2048], m[1::2048] = 0, 2 ** 52 - 1
    s = rng.integers(0, 2, e.size, dtype=np.uint64) << np.uint64(63)
    _bounds(lib, s | e << np.uint64(52) | m)


def test_accepted_pivots(lib):
    """front_positive: exactly the positive numbers of the reciprocal's range."""
    d = np.array([0.0, -0.0, 5e-324, 2.0 ** -1022 - 5e-324, 2.0 ** -1022, 1.0, -1.0, -2.0 ** -1022, np.nextafter(2.0 ** 1021, 0.0),
                  2.0 ** 1021, 1.7e308, np.inf, -np.inf, np.nan])
    want = [0, 0, 0, 0, 1, 1, 0, 0, 1, 0, 0, 0, 0, 0]
    assert _check(lib, d.view(np.uint64))[3].tolist() == want
    neg = -np.float64(np.nan)   # a NaN with its sign bit set
    assert _check(lib, np.array([neg]).view(np.uint64))[3].tolist() == [0]
