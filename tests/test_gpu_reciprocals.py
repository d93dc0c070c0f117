"""recip_cubic and rsqrt_cubic (csrc/qmc_fp.cuh) over the exponent range: within their stated bounds of
the exact values where the iteration runs, CUDA's own 1/a and rsqrt(a) outside, and close to both."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = """
#include <cuda_runtime.h>
#include "qmc_fp.cuh"
__global__ void all(const double *a, int n, double *out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = qmc::recip_cubic(a[i]);
    out[n + i] = 1.0 / a[i];
    out[2 * n + i] = qmc::rsqrt_cubic(a[i]);
    out[3 * n + i] = rsqrt(a[i]);
}
extern "C" int run(const double *a, int n, double *out) {
    all<<<(n + 127) / 128, 128>>>(a, n, out);
    return (int)cudaDeviceSynchronize();
}
"""


def _evaluate(tmp_path, values):
    import torch

    from paper_1811_11720_gb300 import build as B
    src, so = os.path.join(tmp_path, "t.cu"), os.path.join(tmp_path, "t.so")
    with open(src, "w") as fh:
        fh.write(SOURCE)
    subprocess.run([B._nvcc()] + B.ARCH + ["-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-cudart", "shared",
                                          "-I", B.CSRC, "-I", B.INCLUDE, "-o", so, src], check=True)
    a = torch.from_numpy(values).cuda()
    out = torch.empty(4, len(values), dtype=torch.float64, device="cuda")
    assert ctypes.CDLL(so).run(ctypes.c_void_p(a.data_ptr()), len(values), ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy()


def test_against_the_exact_values(tmp_path):
    rng = np.random.default_rng(1)
    mant = np.concatenate([rng.uniform(1, 2, 6000), [1.0, 2 - 2.0 ** -52, 1 + 2.0 ** -52, 1.5]])
    expo = rng.integers(-1022, 1024, len(mant))
    a = np.ldexp(mant, expo)
    a = np.concatenate([a, np.ldexp([1.0, 2 - 2.0 ** -52], [[-1023], [-1022], [-1021], [-1020], [-1019], [1018], [1019], [1020], [1021], [1022]]).ravel(),
                        [5e-324, 1e-310, np.inf, 0.0, np.nan]])
    recip, cuda_recip, rsqrt, cuda_rsqrt = _evaluate(str(tmp_path), a)
    mid = (a >= 2.0 ** -1020) & (a < 2.0 ** 1020)
    assert mid.sum() > 5900 and (~mid).sum() > 10
    for got, ref in ((recip, cuda_recip), (rsqrt, cuda_rsqrt)):
        assert np.array_equal(got[~mid], ref[~mid], equal_nan=True)
    worst = [Fr(0), Fr(0)]
    for v, r, y in zip(a[mid], recip[mid], rsqrt[mid]):
        worst[0] = max(worst[0], abs(Fr(float(r)) * Fr(float(v)) - 1))
        worst[1] = max(worst[1], abs(Fr(float(y)) ** 2 * Fr(float(v)) - 1) / 2)   # to first order
    assert worst[0] <= Fr(2.0 ** -52.9) and worst[1] <= Fr(2.0 ** -52.3)
    assert np.all(np.abs(recip[mid] - cuda_recip[mid]) <= np.spacing(cuda_recip[mid]))
    assert np.all(np.abs(rsqrt[mid] - cuda_rsqrt[mid]) <= 3 * np.spacing(cuda_rsqrt[mid]))


def test_negative_arguments_of_the_reciprocal(tmp_path):
    a = -np.ldexp(np.random.default_rng(2).uniform(1, 2, 500), np.arange(-1000, 1000, 4))
    recip, cuda_recip, _, _ = _evaluate(str(tmp_path), a)
    assert np.all(np.abs(recip - cuda_recip) <= np.spacing(np.abs(cuda_recip)))
