"""Segment height of an untuned batch (csrc/lbm_rules.h), compiled for the host:
a launch takes no longer than with 64 rows (to a tenth) however uneven the
members are, and ordinary mixes take the height of the shortest rounds."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = """
#include "lbm_rules.h"
extern "C" int rows(const int* nx, const int* ny, int n, int threads, long long slots) {
    return lbm::batch_rows(nx, ny, (size_t)n, threads, slots);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, so = str(d / "rules.cpp"), str(d / "rules.so")
    with open(src, "w") as f:
        f.write(SRC)
    csrc = os.path.join(ROOT, "paper_2205_00686_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + csrc, src, "-o", so], check=True)
    L = ctypes.CDLL(so)

    def rows(members, threads, slots):
        nx = (ctypes.c_int * len(members))(*[m[0] for m in members])
        ny = (ctypes.c_int * len(members))(*[m[1] for m in members])
        return L.rows(nx, ny, len(members), threads, ctypes.c_longlong(slots))
    return rows


def iterations(members, threads, slots, R):
    """Row iterations of a launch: the segments (even within a domain) go,
    longest first, to the CTA that is free first."""
    import heapq
    seg = []
    for nx, ny in members:
        n = -(-ny // R)
        h = -(-ny // n)
        seg += [min(h, ny - y) + 8 for y in range(0, ny, h)] * -(-nx // (threads - 8))
    free = [0] * slots
    for s in sorted(seg, reverse=True):
        heapq.heapreplace(free, free[0] + s)
    return max(free)


@pytest.mark.parametrize("members", [
    [(64, 64)] * 10000 + [(64, 4096)],
    [(64, 64)] * 4000 + [(1024, 1024)],
    [(64, 64)] * 8000 + [(1024, 2048)],
    [(64, 64)] * 3000 + [(64, 4096)] * 300,
    [(200, 2)] * 5000 + [(120, 3000)],
], ids=["10000+64x4096", "4000+1024x1024", "8000+1024x2048", "3000+300x64x4096", "5000x2rows"])
@pytest.mark.parametrize("threads,slots", [(128, 608), (224, 304), (128, 152)])
def test_many_short_members_with_a_tall_one(rule, members, threads, slots):
    R = rule(members, threads, slots)
    assert 1 <= R <= max(ny for _, ny in members)
    assert iterations(members, threads, slots, R) <= 1.1 * iterations(members, threads, slots, 64)


def shortest_by_rounds(members, threads, slots):
    """The height in [8, tallest] of the launch w (R + 8) over round counts w
    from the least that could hold all rows."""
    W = threads - 8
    strips = [(-(-nx // W), ny) for nx, ny in members]
    most = max(ny for _, ny in strips)
    w0 = max(1, -(-sum(k * ny for k, ny in strips) // (slots * most)))
    best = None
    for w in range(w0, w0 + 12):
        for R in range(min(8, most), most + 1):
            if sum(k * -(-ny // R) for k, ny in strips) <= w * slots:
                if best is None or w * (R + 8) < best[0]:
                    best = (w * (R + 8), R)
                break
    return best[1]


@pytest.mark.parametrize("threads,slots", [(128, 608), (224, 304)])
def test_ordinary_mixes_take_the_shortest_rounds(rule, threads, slots):
    rng = random.Random(3)
    for n, lo, hi in [(1, 64, 512), (8, 64, 200), (20, 64, 300), (64, 64, 512), (200, 64, 512)]:
        members = [(rng.randint(lo, hi), rng.randint(lo, hi)) for _ in range(n)]
        assert rule(members, threads, slots) == shortest_by_rounds(members, threads, slots)
