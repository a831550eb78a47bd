"""rcp_fast and sqrt_fast of the entropy expansion against correctly rounded operations, over the range and at its ends."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2403_13406_gb300 import build

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

SOURCE = """
#include "expansion.cuh"
template <class R> __global__ void k(const R *x, R *r, R *s, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        r[i] = eslbm::rcp_fast(x[i]);
        s[i] = eslbm::sqrt_fast(x[i]);
    }
}
extern "C" int f32(const void *x, void *r, void *s, int n)
{
    k<float><<<(n + 255) / 256, 256>>>((const float *)x, (float *)r, (float *)s, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int f64(const void *x, void *r, void *s, int n)
{
    k<double><<<(n + 255) / 256, 256>>>((const double *)x, (double *)r, (double *)s, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def functions(tmp_path_factory):
    d = tmp_path_factory.mktemp("fast")
    src, so = os.path.join(d, "fast.cu"), os.path.join(d, "fast.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", "-o", so, src], check=True,
                   capture_output=True)
    L = ctypes.CDLL(so)

    def call(x):
        t = torch.from_numpy(x).cuda()
        r, s = torch.empty_like(t), torch.empty_like(t)
        fn = L.f32 if x.dtype == np.float32 else L.f64
        fn.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
        assert fn(t.data_ptr(), r.data_ptr(), s.data_ptr(), x.size) == 0
        return r.cpu().numpy(), s.cpu().numpy()
    return call


@pytest.mark.parametrize("dtype,lo,hi,rcp_ulp,sqrt_ulp", [
    # the hardware's approximations: at most 1 ulp (reciprocal), a relative error of 2^-23 (square root)
    (np.float32, -126, 126, 1.5, 2.0),
    # one third-order step from a seed of 20 bits or more: the rounding of the step
    (np.float64, -1022, 1020, 1.0, 1.5),
])
def test_normal_range(functions, dtype, lo, hi, rcp_ulp, sqrt_ulp):
    rng = np.random.default_rng(1)
    x = (rng.uniform(1, 2, 1 << 20) * 2.0 ** rng.integers(lo, hi, 1 << 20)).astype(dtype)
    x = np.concatenate([x, dtype(2) ** np.arange(lo, hi + 1, dtype=dtype), rng.uniform(0.5, 2, 1 << 20).astype(dtype)])
    r, s = functions(x)
    L = np.longdouble
    for got, want, ulp in ((r, 1 / x.astype(L), rcp_ulp), (s, np.sqrt(x.astype(L)), sqrt_ulp)):
        assert (np.abs(got.astype(L) - want) <= ulp * np.spacing(want.astype(dtype)).astype(L)).all()


def test_ends_of_the_range(functions):
    """What callers must keep away from (`ordinary`): subnormal arguments count as zero, reciprocals below the normal
    range as zero; in FP64 the correction steps leave no finite value of zero, subnormal numbers and infinity."""
    sub, big = 1e-40, 3e38
    r, s = functions(np.array([0.0, -0.0, sub, -sub, np.inf, np.nan, big, -1.0], dtype=np.float32))
    assert np.array_equal(r[:5], np.float32([np.inf, -np.inf, np.inf, -np.inf, 0.0])) and np.isnan(r[5]) and r[6] == 0
    assert (s[:4] == 0).all() and np.isinf(s[4]) and np.isnan(s[5]) and np.isnan(s[7])
    r, s = functions(np.array([0.0, 1e-310, np.inf, np.nan, 1.7e308]))
    assert np.isnan(r[:4]).all() and r[4] == 0
    assert not np.isfinite(s[:4]).any()
