"""The FP64 reciprocals of csrc/common.cuh against CUDA's division over the exponent range. Two Newton-Raphson
steps from an approximation within 2^-20 leave 2^-80 and the roundings of the last step: one of 2 - x r and
one of the product in rcp (2^-53 each), one in rcp_normal, whose residual 1 - x r of 2^-40 rounds at 2^-93. The
division rounds once: within 3 and 2 times 2^-53 of it."""
import ctypes
import subprocess

import pytest
import torch

from paper_1208_4830_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = """
#include "common.cuh"
__global__ void all(const double* x, double* r, double* s, double* d, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = sblm::rcp(x[i]), s[i] = sblm::rcp_normal(x[i]), d[i] = 1.0 / x[i];
}
extern "C" int run(const double* x, double* r, double* s, double* d, int n) {
    all<<<(n + 255) / 256, 256>>>(x, r, s, d, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_reciprocal_against_division(tmp_path):
    src, so = tmp_path / "reciprocal.cu", tmp_path / "reciprocal.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(so)],
                   check=True)
    g = torch.Generator().manual_seed(1)
    n = 1 << 20
    x = torch.ldexp(1.0 + torch.rand(n, generator=g, dtype=torch.float64),
                    torch.randint(-1020, 1021, (n,), generator=g).double())
    x[:4] = torch.tensor([1.0, 2.0, 2.0**-1020, 2.0**1020], dtype=torch.float64)
    x = torch.cat([x, torch.tensor([0.0, float("inf"), float("nan")], dtype=torch.float64)]).cuda()
    r, s, d = (torch.empty_like(x) for _ in range(3))
    torch.cuda.synchronize()
    assert ctypes.CDLL(str(so)).run(*(ctypes.c_void_p(a.data_ptr()) for a in (x, r, s, d)), x.numel()) == 0
    for a, most in ((r, 3), (s, 2)):
        assert ((a[:n] - d[:n]).abs() <= most * (1 + 2.0**-20) * 2.0**-53 * d[:n]).all()
    assert r[n] == float("inf") and r[n + 1] == 0 and torch.isnan(r[n + 2])
    assert torch.isnan(s[n:]).all()
