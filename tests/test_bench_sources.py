"""bench.py's kernel captures (DRAM traffic, FP64 instructions) are keyed by a
hash of the sources that make the single lattice's step kernels: every file of
csrc/ that those sources include must be in it, and the planner that cuts their
tiles."""
import importlib
import os
import re
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1412_5170_gb300", "csrc")


def closure(names):
    todo, seen = list(names), set()
    while todo:
        n = todo.pop()
        if n in seen or not os.path.exists(os.path.join(CSRC, n)):
            continue
        seen.add(n)
        todo += re.findall(r'#include "([^"]+)"', open(os.path.join(CSRC, n)).read())
    return seen


def test_hash_covers_the_step_kernels():
    sys.path.insert(0, ROOT)
    bench = importlib.import_module("bench")
    hashed = {os.path.basename(s) for s in bench.KERNEL_SOURCES}
    assert all(os.path.exists(os.path.join(ROOT, s)) for s in bench.KERNEL_SOURCES)
    assert closure(["lbm_strip_f32.cu", "lbm_kernels.cuh", "lbm_tilewalk.cuh", "lbm_host.cpp"]) <= hashed
