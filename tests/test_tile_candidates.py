"""CPU checks of the tiles the small-domain form really takes
(csrc/lbm_tile.cu): the index model of test_tile_schedule.py on those it leaves
out, and the threads that take the nodes around a tile."""
import pytest

from test_tile_schedule import OPEN, PERIODIC, WALL
from test_tile_schedule import test_tile_step_reads_what_was_written_and_writes_once as model

# (tx, ty, the surrounding nodes have threads of their own)
TILES = [(8, 8, 1), (32, 8, 0), (32, 10, 0), (32, 12, 0), (8, 4, 1), (16, 8, 0), (20, 14, 0)]


@pytest.mark.parametrize("tx,ty", [(8, 8), (16, 8), (32, 10), (32, 12)])
@pytest.mark.parametrize("fx", [PERIODIC, OPEN])
@pytest.mark.parametrize("fy", [(PERIODIC, PERIODIC), (WALL, WALL), (WALL, OPEN), (OPEN, OPEN)])
@pytest.mark.parametrize("nx,ny", [(33, 13), (2, 2), (9, 25)])
def test_index_model(tx, ty, fx, fy, nx, ny):
    model(tx, ty, fx, fy, nx, ny)


@pytest.mark.parametrize("tx,ty,sep", TILES)
def test_threads_cover_the_nodes_around(tx, ty, sep):
    n1 = 2 * (tx + ty) + 4
    n = n1 + 2 * (tx + ty) + 12
    own_w, ring_w = -(-tx * ty // 32), -(-n // 32)
    ring0 = own_w * 32 if sep else 0
    threads = (own_w + ring_w) * 32 if sep else max(own_w * 32, -(-n1 // 32) * 32)
    assert tx * ty <= threads <= 512
    for tw in range(1, tx + 1):
        for th in range(1, ty + 1):
            m1 = 2 * (tw + th) + 4
            m = m1 + 2 * (tw + th) + 12
            taken = []
            for t in range(threads):
                k = t - ring0 if t >= ring0 else t - ring0 + threads
                if k < m:
                    taken.append(k)          # set up once, force formed when k < m1
                taken += range(k + threads, m, threads)
            assert sorted(taken) == list(range(m))
            # the first ring, whose velocity stage B forms, has a thread each
            assert m1 <= threads
