"""div_by (tof_device.cuh): a / b from the rounded reciprocal of b (Markstein, IBM J. Res. Dev. 34(1), 1990) equals the
correctly rounded quotient, which is what the device's own division gives, bit for bit: random mantissas and
mantissas next to a power of two, exponents far from the ends of the range."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2605_11536_gb300 import build

pytestmark = pytest.mark.gpu

_SRC = r"""
#include "tof_device.cuh"
__global__ void compare(const float* a, const float* b, unsigned n, unsigned* differ) {
    const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (__float_as_uint(tof::div_by(a[i], b[i], 1.0f / b[i])) != __float_as_uint(a[i] / b[i])) atomicAdd(differ, 1u);
}
extern "C" int run(const float* a, const float* b, unsigned n, unsigned* differ) {
    compare<<<(n + 255u) / 256u, 256>>>(a, b, n, differ);
    return (int)cudaDeviceSynchronize();
}
"""


def test_division_by_a_shared_reciprocal(tmp_path):
    import torch
    src, so = tmp_path / "div.cu", tmp_path / "div.so"
    src.write_text(_SRC)
    r = subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-I", build.INCLUDE, "-shared", "-cudart", "shared",
                        "-o", str(so), str(src)], capture_output=True, text=True, env=dict(os.environ))
    assert r.returncode == 0, r.stderr
    run = ctypes.CDLL(str(so)).run
    run.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_uint, ctypes.c_void_p]
    rng = np.random.default_rng(1)
    n = 1 << 24

    def values():
        m = rng.integers(0, 1 << 23, size=n, dtype=np.uint32)
        edge = rng.integers(0, 64, size=n, dtype=np.uint32)
        m = np.where(rng.random(n) < 0.25, np.where(rng.random(n) < 0.5, edge, (1 << 23) - 1 - edge), m).astype(np.uint32)
        e = rng.integers(127 - 40, 127 + 41, size=n, dtype=np.uint32)
        s = rng.integers(0, 2, size=n, dtype=np.uint32)
        return torch.from_numpy(((s << 31) | (e << 23) | m).view(np.float32).copy()).cuda()

    for _ in range(4):
        a, b = values(), values()
        differ = torch.zeros(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert run(a.data_ptr(), b.data_ptr(), n, differ.data_ptr()) == 0
        assert int(differ.item()) == 0
        # against the correctly rounded quotient itself (64-bit division rounds to 32 bits correctly: 53 >= 2 * 24 + 2)
        q = (a.double() / b.double()).float()
        assert torch.equal(q, a / b)
