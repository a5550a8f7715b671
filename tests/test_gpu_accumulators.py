"""The premise of the products in digits: mma.sync adds integers exactly in its FP32
accumulators up to 2^24, the most that 4 x 256 (one column) or 8 x 128 (eight
columns) products of digits in [-128, 127] can reach."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1601_03432_gb300", "csrc")
SOURCE = r"""
#include "smpm_digits.cuh"
// one warp: acc = sum over `tiles` 16 x 16 by 16 x 8 products of biased digits
__global__ void k_sum(const uint2* a, const uint2* b, int tiles, float* out) {
  float acc[4] = {0, 0, 0, 0};
  for (int t = 0; t < tiles; ++t) {
    const uint2 w = a[t * 32 + threadIdx.x], v = b[t * 32 + threadIdx.x];
    uint32_t r[4], s[4];
    digit_a(w.x, w.y, r);
    digit_a(v.x, v.y, s);
    mma_16816(acc, r, s[0], s[2]);
  }
  for (int v = 0; v < 4; ++v) out[threadIdx.x * 4 + v] = acc[v];
}
extern "C" int sum_tiles(const void* a, const void* b, int tiles, void* out) {
  k_sum<<<1, 32>>>((const uint2*)a, (const uint2*)b, tiles, (float*)out);
  return cudaGetLastError() || cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1601_03432_gb300.build import ARCH, COMMON
    d = tmp_path_factory.mktemp("digits")
    src, so = d / "sum.cu", d / "sum.so"
    src.write_text(SOURCE)
    nvcc = "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-shared", *ARCH, *COMMON, "-I", CSRC, "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def tile_words(D):
    """Digits of 16 x 16 tiles (tiles, row, column) as the fragments of pack_digits."""
    lane = np.arange(32)
    g, q = lane // 4, lane % 4
    w = np.zeros((D.shape[0], 32, 2), np.uint32)
    for h in range(2):
        for b in range(4):
            d = D[:, g + 8 * (b // 2), 2 * q + (b % 2) + 8 * h]
            w[:, :, h] |= ((d + 128).astype(np.uint32) & 255) << np.uint32(8 * b)
    return w


@pytest.mark.parametrize("kind", ["lowest", "odd", "highest", "random", "cancelling"])
@pytest.mark.parametrize("tiles", [64, 63, 1])
def test_sums_of_digit_products_are_exact(lib, kind, tiles):
    rng = np.random.default_rng(tiles)
    A = np.full((tiles, 16, 16), -128, np.int64)
    X = np.full((tiles, 8, 16), -128, np.int64)  # (tile, column, k)
    if kind == "odd":  # 2^24 - 255 with 64 tiles
        A[-1, :, 3], X[-1, :, 3] = 127, 127
    elif kind == "highest":
        A[:] = X[:] = 127
    elif kind == "random":
        A, X = rng.integers(-128, 128, A.shape), rng.integers(-128, 128, X.shape)
    elif kind == "cancelling":  # up to half of the range and back, an odd rest
        A[tiles // 2:] = 127
        A[0, :, 0] = 1
    X16 = np.zeros((tiles, 16, 16), np.int64)  # columns as rows g of a tile
    X16[:, :8] = X
    a, b = (torch.as_tensor(tile_words(m).view(np.int32), device="cuda") for m in (A, X16))
    out = torch.empty(32, 4, device="cuda")
    torch.cuda.synchronize()
    assert lib.sum_tiles(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), tiles,
                         ctypes.c_void_p(out.data_ptr())) == 0
    want = np.einsum("trk,tck->rc", A, X)
    assert np.abs(want).max() <= 1 << 24
    lane = np.arange(32)
    got = out.cpu().numpy().astype(np.int64)
    for v in range(4):
        assert np.array_equal(got[:, v], want[lane // 4 + 8 * (v // 2), 2 * (lane % 4) + v % 2]), kind
