"""bench.py reports a captured DRAM figure only while the step kernel's sources
are those it was captured on: the hash covers every file the kernel is made of."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2205_00686_gb300", "csrc")


def test_the_source_hash_covers_the_step_kernel():
    import bench
    need, todo = set(), ["lbm_step.cu"]
    while todo:
        name = todo.pop()
        if name in need:
            continue
        need.add(name)
        with open(os.path.join(CSRC, name)) as f:
            todo += [n for n in re.findall(r'#include "([^"]+)"', f.read()) if os.path.exists(os.path.join(CSRC, n))]
    assert need == {os.path.basename(p) for p in bench.STEP_SOURCES}
