"""Index arithmetic of the kernels that walk a whole lattice
(csrc/lbm_index.cuh), compiled by g++ and run on the shapes where 32-bit
indices can overflow: a lattice may hold up to 2^31 - 1 nodes in any shape."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOP = 2 ** 31 - 1


@pytest.fixture(scope="module")
def walks(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("needs g++")
    so = str(tmp_path_factory.mktemp("index_walks") / "libwalks.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-fsanitize=undefined", "-fno-sanitize-recover",
                           "-static-libubsan", "-I", os.path.join(ROOT, "paper_1412_5170_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "host_arithmetic", "index_walks.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    lib.walk_nodes.restype = ctypes.c_longlong
    lib.walk_nodes.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.c_uint]
    return lib


@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 97), (97, 1), (8, 16384), (4096, 4096), (46341, 46340), (3, TOP // 3), (TOP // 3, 3),
                                   (1, TOP), (TOP, 1), (TOP - 100, 1), (TOP // 2, 2), (2, TOP // 2)])
def test_nodes(walks, nx, ny):
    """Every node once, with its column and row, whatever the grid."""
    n = nx * ny
    for ctas in (1, 64, 152 * 32, min((n + 255) // 256, 2 ** 22)):
        step = 256 * ctas
        for first in {0, 1, step // 2, step - 1}:
            if n // step > 3 * 10 ** 6:
                continue   # one CTA over the largest lattices: too many steps to look at each
            assert walks.walk_nodes(nx, ny, step, first) == max(0, -(-(n - first) // step)), (nx, ny, step, first)
