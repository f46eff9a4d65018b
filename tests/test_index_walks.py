"""Index arithmetic of the kernels that walk a whole lattice
(csrc/lbm_index.cuh, and the cuts of csrc/lbm_host.cpp), compiled by g++ and
run on the shapes where 32-bit indices can overflow: a lattice may hold up to
2^31 - 1 nodes in any shape."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOP = 2 ** 31 - 1


@pytest.fixture(scope="module")
def walks(tmp_path_factory):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    csrc = os.path.join(ROOT, "paper_1412_5170_gb300", "csrc")
    so = str(tmp_path_factory.mktemp("index_walks") / "libwalks.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-fsanitize=undefined", "-fno-sanitize-recover",
                           "-static-libubsan", "-I", csrc, "-I", os.path.join(ROOT, "include"), "-I", cuda,
                           os.path.join(ROOT, "tests", "host_arithmetic", "index_walks.cpp"),
                           os.path.join(csrc, "lbm_host.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    for fn, args in ((lib.walk_nodes, [ctypes.c_int, ctypes.c_int, ctypes.c_uint, ctypes.c_uint]),
                     (lib.walk_chunk, [ctypes.c_int, ctypes.c_int, ctypes.c_uint])):
        fn.restype, fn.argtypes = ctypes.c_longlong, args
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


@pytest.mark.parametrize("ctas", [2, 4])
@pytest.mark.parametrize("nx,ny", [(1, 1), (1, 9), (33, 4231), (1023, 1021), (8, 1 << 20), (4096, 4), (1, TOP), (1, TOP - 7), (1, TOP - 8),
                                   (1, TOP - 16), (2, TOP // 2), (TOP, 1), (TOP - 20, 1)])
def test_walks_of_tiles(walks, nx, ny, ctas):
    """The plan's strips and chunks cover the lattice, and every chunk its rows."""
    out = (ctypes.c_int * 3)()
    walks.walk_plan(nx, ny, 152, ctas, out)
    sx, sy, rows = out
    assert 32 * (sx - 1) < nx <= 32 * sx and 1 <= sy <= 65535 and rows % 8 == 0
    assert rows * (sy - 1) < ny <= rows * sy
    for b in {0, sy // 2, sy - 1}:
        assert walks.walk_chunk(ny, rows, b) == min(rows, ny - b * rows)
