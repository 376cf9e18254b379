"""rsqrt_pos (the QL recurrence's FP64 reciprocal root) against the exact root: every exponent that the
recurrence gives it, odd and even, with mantissas at the ends, beside a power of two and drawn ones."""
import ctypes
import subprocess

import numpy as np
import pytest

from gpu_helpers import require_gpu, torch

pytestmark = pytest.mark.gpu

SRC = r"""
#include "rsqrt_pos.cuh"
__global__ void root(int n, const double* h, double* r) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) r[i] = otvmc::rsqrt_pos(h[i]);
}
extern "C" __attribute__((visibility("default"))) int run(int n, const double* h, double* r) {
    root<<<(n + 255) / 256, 256>>>(n, h, r);
    return (int)cudaDeviceSynchronize();
}
"""


def test_rsqrt_pos(tmp_path):
    require_gpu()
    from paper_2506_23928_gb300 import build
    src, lib = tmp_path / "root.cu", tmp_path / "libroot.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(lib), str(src)], check=True)
    g = np.random.default_rng(1)
    top = (1 << 52) - 1
    mant = np.concatenate([[0, 1, 2, 1 << 28, (1 << 29) - 1, 1 << 29, top - (1 << 29), top - 1, top],
                           g.integers(0, 1 << 52, 191)]).astype(np.int64)
    # biased exponents 65 .. 1999, the ones for which the recurrence calls it
    bits = (np.arange(65, 2000, dtype=np.int64)[:, None] << 52) | mant[None, :]
    h = bits.ravel().view(np.float64)
    h_d = torch.from_numpy(h).cuda()
    r_d = torch.zeros_like(h_d)
    torch.cuda.synchronize()
    run = ctypes.CDLL(str(lib)).run
    assert run(ctypes.c_int(h.size), ctypes.c_void_p(h_d.data_ptr()), ctypes.c_void_p(r_d.data_ptr())) == 0
    r = r_d.cpu().numpy()
    # r^2 h - 1 = 2 (relative error of r), in whole numbers scaled so that nothing is rounded: with
    # r = a 2^p and h = b 2^q (a, b of 53 bits) it is a^2 b 2^(2 p + q) - 1
    fr, er = np.frexp(r)
    fh, eh = np.frexp(h)
    a, b = np.ldexp(fr, 53).astype(np.int64).astype(object), np.ldexp(fh, 53).astype(np.int64).astype(object)
    sh = 3 * 53 - (2 * er + eh)  # a^2 b 2^-sh
    excess = np.array([float(x * x * y - (1 << int(s))) * 2.0 ** -int(s) for x, y, s in zip(a, b, sh)])
    # 1.5 2^-53, the neglected 2^-63 and 2^-60 for second-order terms
    assert np.abs(excess).max() <= 2 * (1.5 * 2.0 ** -53 + 2.0 ** -60)
