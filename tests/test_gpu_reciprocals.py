"""The two FP64 reciprocals of the kernels (fehmm_device.cuh), applied to arrays by a kernel compiled here, against the
correctly rounded 1 / x.  The hardware's approximation and the conversion before it are off by less than 2^-22, the
iteration cubes that, and the last operation rounds: no more than one ulp from the rounded quotient."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "fehmm_device.cuh"
__global__ void apply(const double* x, double* a, double* b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) { a[i] = fehmm::recip_d(x[i]); b[i] = fehmm::recip_fp64(x[i]); }
}
extern "C" int run(const double* x, double* a, double* b, int n) {
  apply<<<(n + 127) / 128, 128>>>(x, a, b, n);
  return (int)cudaDeviceSynchronize();
}
"""


def ulps(got, want):
    """Distance in representable numbers of two arrays of the same signs."""
    return np.abs(got.view(np.int64) - want.view(np.int64))


def test_reciprocals_within_an_ulp(tmp_path):
    import torch

    from paper_1908_08292_gb300 import build

    src, so = tmp_path / "recip.cu", tmp_path / "librecip.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(so), str(src)], check=True)
    rng = np.random.default_rng(5)
    exps = np.arange(0, 2047, dtype=np.uint64)  # 0: subnormal
    mant = np.concatenate([np.array([0, 1, 2, 1 << 28, 1 << 29, (1 << 29) - 1, 1 << 51, (1 << 52) - 1], dtype=np.uint64),
                           rng.integers(0, 1 << 52, 120, dtype=np.uint64)])
    x = ((exps[:, None] << np.uint64(52)) | mant[None, :]).reshape(-1).view(np.float64)
    x = np.concatenate([x, -x, [np.inf, -np.inf, np.nan]])
    t = [torch.tensor(x, device="cuda:0"), *(torch.zeros(x.size, dtype=torch.float64, device="cuda:0") for _ in range(2))]
    torch.cuda.synchronize()
    assert ctypes.CDLL(str(so)).run(*(ctypes.c_void_p(v.data_ptr()) for v in t), x.size) == 0
    d, j = t[1].cpu().numpy(), t[2].cpu().numpy()
    with np.errstate(divide="ignore", over="ignore"):
        want = 1.0 / x
    # recip_d: every x
    nan = np.isnan(want)
    assert np.all(np.isnan(d[nan])) and np.all(ulps(d[~nan], want[~nan]) <= 1)
    split = (x >= 2.0 ** -1022) & (x < 2.0 ** 1018)
    assert np.all(d[~split & ~nan] == want[~split & ~nan])  # the division itself
    # recip_fp64: FP32's normal range, by bits (positive) and by conversions (negative); beyond it as its comment says
    inside = ((x >= 2.0 ** -126) & (x < 2.0 ** 126)) | ((x <= -2.0 ** -125) & (x > -2.0 ** 125))
    assert np.all(ulps(j[inside], want[inside]) <= 1)
    assert not np.any(np.isfinite(j[np.abs(x) < 2.0 ** -127]))
    big = np.isfinite(x) & (np.abs(x) > 2.0 ** 127)
    assert np.all(j[big] == 0)
