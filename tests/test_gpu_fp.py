"""The operator's own square root with its reciprocal and conversion to FP32 (csrc/vofp_fp.cuh) against CUDA's operators,
bit for bit: every exponent, both parities, powers of two and their neighbours, subnormals, the limits of the range that
takes the short way, zeros, infinities, NaN and negative values, and 2^24 random values.  (One value in some 2^36 may be
rounded the other way: 2^-11 of one in this test.)"""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SOURCE = """
#include "vofp_fp.cuh"
__global__ void both(int n, const double* d, double* r, double* rr, double* v, double* vv, float* f, float* ff) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    vofp::sqrt_and_inverse(d[i], r[i], v[i]);
    rr[i] = sqrt(d[i]);
    vv[i] = 1.0 / rr[i];
    f[i] = vofp::to_float(d[i]);
    ff[i] = (float)d[i];
}
extern "C" int run(int n, const double* d, double* r, double* rr, double* v, double* vv, float* f, float* ff) {
    both<<<(n + 255) / 256, 256>>>(n, d, r, rr, v, vv, f, ff);
    return (int)cudaDeviceSynchronize();
}
"""


def _values():
    rng = np.random.default_rng(12)
    low = np.array([0, 1, 2, 3, 1 << 28, (1 << 28) + 1, (1 << 29) - 1, 1 << 29, (1 << 51) - 1, 1 << 51, (1 << 52) - 2, (1 << 52) - 1],
                   dtype=np.uint64)
    e = np.arange(2047, dtype=np.uint64)[:, None] << np.uint64(52)
    mantissa = np.concatenate([np.broadcast_to(low, (2047, low.size)), rng.integers(0, 1 << 52, (2047, 64), dtype=np.uint64)], 1)
    grid = (e | mantissa).ravel().view(np.float64)
    exponent = rng.integers(190, 1810, 1 << 24, dtype=np.uint64) << np.uint64(52)
    random = (exponent | rng.integers(0, 1 << 52, 1 << 24, dtype=np.uint64)).view(np.float64)
    return np.concatenate([grid, -grid, [np.inf, -np.inf, np.nan, 0.0, -0.0], random])


def test_square_root_reciprocal_and_conversion_match_cuda(tmp_path):
    from paper_1410_1937_gb300 import build as B
    (tmp_path / "fp.cu").write_text(SOURCE)
    lib = str(tmp_path / "fp.so")
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", lib, str(tmp_path / "fp.cu")], check=True)
    d = torch.from_numpy(_values()).cuda()
    out = [torch.empty_like(d) for _ in range(4)] + [torch.empty_like(d, dtype=torch.float32) for _ in range(2)]
    torch.cuda.synchronize()
    assert ctypes.CDLL(lib).run(d.numel(), *(ctypes.c_void_p(t.data_ptr()) for t in (d, *out))) == 0
    for got, want in zip(out[::2], out[1::2]):
        word = torch.int64 if got.dtype == torch.float64 else torch.int32
        differ = (got.view(word) != want.view(word)) & ~(got.isnan() & want.isnan())
        assert int(differ.sum()) == 0, d[differ][:8].tolist()
