"""The prompt GEMM's silu (the device function itself, compiled into a small kernel) against 64 bits: the range of the division,
both its ends, values that no divisor can hold, infinities and not-a-number."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_silu(tmp_path):
    so = str(tmp_path / "libsilu.so")
    subprocess.check_call([os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"), "-gencode", "arch=compute_100a,code=sm_100a", "-O3",
                           "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I",
                           os.path.join(ROOT, "paper_2412_18910_b200", "csrc"), "-o", so, os.path.join(ROOT, "tests", "silu_kernel.cu")])
    rng = np.random.default_rng(3)
    edges = [0.0, -0.0, 1e-30, -1e-30, 79.9, 80.0, 80.1, 88.0, 88.1, 100.0, 1e6, 3e38]
    x = np.concatenate([rng.uniform(-90, 100, 1 << 18), rng.standard_normal(1 << 18), edges, np.negative(edges),
                        [np.inf, -np.inf, np.nan]]).astype(np.float32)
    dx = torch.from_numpy(x).cuda()
    dy = torch.empty_like(dx)
    lib = C.CDLL(so)
    assert lib.silu_run(C.c_void_p(dx.data_ptr()), C.c_void_p(dy.data_ptr()), C.c_int(x.size)) == 0
    y = dy.cpu().numpy().astype(np.float64)
    assert y[-3] == np.inf and np.isnan(y[-2]) and np.isnan(y[-1])
    x, y = x[:-3].astype(np.float64), y[:-3]
    want = x / (1 + np.exp(np.minimum(-x, 700)))
    # the fast exponential is off by up to 2 + 1.173 |x| units (of 2^-23 relative), the sum and the quotient by half a unit each
    bound = np.where(x < -80, 1.5e-33, np.abs(want) * (4 + 1.2 * np.abs(x) * (x < 20)) * 2.0 ** -23 + 1e-37)
    assert (np.abs(y - want) <= bound).all(), x[np.abs(y - want) > bound][:5]
