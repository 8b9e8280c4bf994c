"""The Newton-Raphson reciprocal, square root and reciprocal square root of the
FP32 terms (csrc/md.cuh) against float64, over the range of their arguments.
One step from an approximation good to 2 ulp leaves the rounding of the last
fused operation and of the intermediate products: at most 2 ulp."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "md.cuh"
__global__ void k(int n, const float *x, float *y)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        y[i] = jk::rcp_nr(x[i]);
        y[n + i] = jk::sqrt_nr(x[i]);
        y[2 * n + i] = jk::rsqrt_nr(x[i]);
    }
}
extern "C" void run(int n, const float *x, float *y) { k<<<256, 256>>>(n, x, y); cudaDeviceSynchronize(); }
"""


def test_newton_steps(tmp_path):
    from paper_2410_22278_gb300 import build as b

    src, lib = tmp_path / "ops.cu", tmp_path / "ops.so"
    src.write_text(SRC)
    subprocess.run([b.NVCC] + b.ARCH + b.FLAGS + b.FAST_F32 + ["-I" + b.CSRC, "-shared", "-o", str(lib), str(src)], check=True,
                   env=dict(os.environ))
    rng = np.random.default_rng(0)
    x = np.exp(rng.uniform(np.log(1e-12), np.log(1e12), 1 << 20)).astype(np.float32)
    xt = torch.from_numpy(x).cuda()
    y = torch.empty(3 * x.size, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    f = ctypes.CDLL(str(lib)).run
    f.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p]
    f(x.size, xt.data_ptr(), y.data_ptr())
    got = y.cpu().numpy().reshape(3, -1).astype(np.float64)
    x = x.astype(np.float64)
    for g, ref in zip(got, (1.0 / x, np.sqrt(x), 1.0 / np.sqrt(x))):
        ulp = np.spacing(ref.astype(np.float32)).astype(np.float64)
        assert np.max(np.abs(g - ref) / ulp) <= 2.0
