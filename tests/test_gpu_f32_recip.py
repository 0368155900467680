"""The FP32 trackers' reciprocal and reciprocal square root (f32_step.cuh) over the whole range of
floats.  The hardware's approximations are within 2 ulp, the reciprocal's Newton step brings it
within 1; subnormal arguments and results count too (their ulp is 2^-149)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from gpu_common import nphc

pytestmark = pytest.mark.gpu

SOURCE = """
#include "f32_step.cuh"
__global__ void k(const float *x, float *r, float *q, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = f32_recip(x[i]);
    q[i] = f32_rsqrt(x[i]);
}
extern "C" int run(const float *x, float *r, float *q, int n) {
    k<<<(n + 255) / 256, 256>>>(x, r, q, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_full_range(tmp_path):
    import torch
    nphc()
    from paper_1104_5497_gb300 import build as B
    src, so = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", str(src), "-o", str(so)], check=True)
    rng = np.random.default_rng(0)
    e = np.repeat(np.arange(-149, 128), 200)
    x = (np.ldexp(rng.uniform(1, 2, e.size), e)).astype(np.float32)
    x = np.concatenate([x, np.ldexp(np.float32(1), np.arange(-149, 128)).astype(np.float32)])
    xd = torch.as_tensor(x, device="cuda")
    r, q = torch.empty_like(xd), torch.empty_like(xd)
    f = ctypes.CDLL(os.fspath(so)).run
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]
    assert f(xd.data_ptr(), r.data_ptr(), q.data_ptr(), x.size) == 0
    for got, want, ulps in ((r, 1.0 / x.astype(np.float64), 1.0), (q, 1.0 / np.sqrt(x.astype(np.float64)), 2.0)):
        got = got.cpu().numpy().astype(np.float64)
        fits = want <= np.finfo(np.float32).max
        ulp = np.ldexp(1.0, np.maximum(np.floor(np.log2(want[fits])).astype(int), -126) - 23)
        assert np.all(np.abs(got[fits] - want[fits]) <= ulps * ulp)
        assert not np.isfinite(got[~fits]).any()
