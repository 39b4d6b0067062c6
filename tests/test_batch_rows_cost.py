"""The segment-height rule runs at every attach and detach: it takes few passes
over the members, and gives the answer of the search without short cuts."""
import ctypes
import os
import random
import subprocess

import pytest

import test_batch_rows as T

COUNT = T.SRC + """
extern "C" int passes(const int* nx, const int* ny, int n, int threads, long long slots, int* rows) {
    int p = 0;
    *rows = lbm::batch_rows(nx, ny, (size_t)n, threads, slots, &p);
    return p;
}
"""


def plain(members, threads, slots):
    """64 rows or, of 12 round counts w from the fewest that can hold all rows and
    the uncut strips, the shortest w (R + 8) with the least R that fits."""
    W = threads - 8
    strips = [(-(-nx // W), ny) for nx, ny in members]
    most = max(ny for _, ny in strips)

    def segments(R):
        return sum(k * -(-ny // R) for k, ny in strips)

    rows = min(64, most)
    best = max(1, -(-segments(rows) // slots)) * (rows + 8)
    w0 = max(1, -(-segments(most) // slots), -(-sum(k * ny for k, ny in strips) // (slots * most)))
    for w in range(w0, w0 + 12):
        R = min(8, most)
        while segments(R) > w * slots:
            R += 1
        if w * (R + 8) < best:
            best, rows = w * (R + 8), R
    return rows


@pytest.mark.parametrize("threads,slots", [(128, 608), (224, 304), (128, 152)])
def test_few_passes_over_the_members(tmp_path, threads, slots):
    src, so = str(tmp_path / "rules.cpp"), str(tmp_path / "rules.so")
    with open(src, "w") as f:
        f.write(COUNT)
    csrc = os.path.join(T.ROOT, "paper_2205_00686_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + csrc, src, "-o", so], check=True)
    L = ctypes.CDLL(so)
    rng = random.Random(9)
    for n, lo, hi in [(1, 2, 700), (5, 64, 200), (20, 64, 300), (82, 64, 512), (512, 64, 512), (300, 1, 2000)]:
        m = [(rng.randint(lo, hi), rng.randint(lo, hi)) for _ in range(n)]
        nx, ny = ((ctypes.c_int * n)(*[v[k] for v in m]) for k in (0, 1))
        rows = ctypes.c_int()
        p = L.passes(nx, ny, n, threads, ctypes.c_longlong(slots), ctypes.byref(rows))
        assert p <= 40
        assert rows.value == plain(m, threads, slots)
