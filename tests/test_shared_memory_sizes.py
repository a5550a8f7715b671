"""The largest grids that the solve kernels have taken stay within their shared
memory (one group per CTA, w in global memory: the least they need).  Host code
only: the size functions of the kernels' headers, compiled with nvcc."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_03432_gb300", "csrc")
NVCC = "/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else shutil.which("nvcc")
SOURCE = r"""
#include "smpm_device.cuh"
#include "smpm_digits.cuh"
#include <cstdio>
#include <cstdlib>
namespace {
#include "smpm_gmres.cuh"
#include "smpm_prepost.cuh"
}
int main(int argc, char** argv) {
  for (int i = 1; i + 3 < argc; i += 4) {
    const long long mx = std::atoi(argv[i]), my = std::atoi(argv[i + 1]);
    const int n = std::atoi(argv[i + 2]), m = std::atoi(argv[i + 3]), M = 4 * n;
    const long long nb = (mx * my + 1) / 2, d = (mx - 1) * my + mx * (my - 1);
    const int ES = 2 * M * (int)((nb + 151) / 152);
    std::printf("%zu %zu\n", prepost_smem_bytes(m, M, n, ES, 8, 8, d, true),
                gmres_smem_bytes<double>(m, M, n, ES, 8, 0, d, true));
  }
}
"""

# elements, order, restart: the last sizes of a square and of an eight times longer
# grid that fitted the kernels with FP64 products (w and w2 in shared memory)
GRIDS = [(114, 114, 2, 50), (40, 320, 2, 50), (112, 112, 2, 200), (39, 312, 2, 200), (111, 111, 4, 50),
         (105, 105, 8, 50), (100, 100, 12, 50), (95, 95, 16, 50), (86, 86, 24, 50), (79, 79, 32, 50),
         (77, 77, 32, 200), (28, 224, 32, 50)]


@pytest.mark.skipif(NVCC is None, reason="nvcc not found")
def test_largest_grids_fit(tmp_path):
    from paper_1601_03432_gb300.build import ARCH, COMMON
    src, exe = tmp_path / "sizes.cu", tmp_path / "sizes"
    src.write_text(SOURCE)
    subprocess.run([NVCC, *ARCH, *COMMON, "-O0", "-I", CSRC, "-o", str(exe), str(src), "-lgomp"], check=True)
    out = subprocess.run([str(exe), *(str(v) for g in GRIDS for v in g)], check=True, capture_output=True, text=True)
    budget = 232448 - 2048  # opt-in shared memory of a CTA less the staged arguments
    for g, line in zip(GRIDS, out.stdout.split("\n")):
        assert max(int(v) for v in line.split()) <= budget, (g, line)
