"""A launch the runtime refuses is returned as an error and leaves none behind: whoever asks
CUDA for the last error next (a framework after a launch of its own) does not find it."""
import ctypes
import os
import subprocess

import pytest

from paper_1411_2860_gb300 import _build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "pdl.cuh"
__global__ void nothing(int) {}
extern "C" int refused(int pdl) {
  (void)cudaGetLastError();
  const dim3 grid(1);   // 4096 threads a block: refused on the host
  const cudaError_t e = pdl ? pj::launch_pdl(nothing, grid, 4096, 0, 0, 1, 0) : pj::launch_plain(nothing, grid, 4096, 0, 0, 0);
  return static_cast<int>(e);
}
extern "C" int left_behind() { return static_cast<int>(cudaPeekAtLastError()); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("launch")
    src, so = str(d / "refused.cu"), str(d / "refused.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([_build.nvcc(), "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                    "-I", os.path.join(_build.HERE, "csrc"), src, "-o", so], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("pdl", [0, 1])
def test_refused_launch_leaves_no_error_behind(lib, pdl):
    assert lib.refused(pdl) != 0
    assert lib.left_behind() == 0
