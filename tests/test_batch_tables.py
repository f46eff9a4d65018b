"""The growing device tables of a batch (work items, tiles) when an
allocation fails: the table stays as it was, usable, with nothing leaked or
given back early.  Host code (lbm_host.h) under g++, the allocator a fake."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def tab(tmp_path_factory):
    cuda = "/usr/local/cuda/include"
    if not shutil.which("g++") or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("tables") / "libtables.so")
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1412_5170_gb300", "csrc"), "-I", cuda,
                           os.path.join(ROOT, "tests", "host_arithmetic", "tables.cpp"), "-o", so])
    lib = ctypes.CDLL(so)
    lib.write_read.restype = ctypes.c_longlong
    return lib


def test_a_failed_allocation_leaves_the_table(tab):
    assert not tab.reserve(10, 1) and tab.capacity() == 0 and tab.buffers() == 0
    assert tab.reserve(10, 0) and tab.capacity() == 10 and tab.write_read(10) == 10
    assert not tab.reserve(11, 1) and tab.capacity() == 10 and tab.buffers() == 1
    assert tab.write_read(10) == 10              # still the old buffer
    assert tab.reserve(7, 1) and tab.capacity() == 10   # no allocation needed
    assert tab.reserve(11, 0) and tab.capacity() == 11 and tab.buffers() == 1
    assert tab.early_frees() == 0


def test_the_batch_grows_its_tables_through_it():
    """Both tables, and the tiled step is taken only once its table is in place."""
    src = open(os.path.join(ROOT, "paper_1412_5170_gb300", "csrc", "lbm_batch.cu")).read()
    assert src.count("table_reserve(b->items") == 1 and src.count("table_reserve(b->stiles") == 1
    body = src[src.index("int build_tiles("):src.index("int build_items(")]
    assert body.index("b->use_tiles = false") < body.index("table_reserve") < body.index("b->use_tiles = true")
