"""CPU model of the small-domain step's index arithmetic (csrc/lbm_tile.cu):
for domains of ragged sizes, every boundary kind and several tiles, each value
a stage reads has been written by the stage before, shared-memory indices stay
inside their arrays, and every population of the next state is written exactly
once, from the node that the pull form of the step names as its source."""
import itertools

import pytest

PERIODIC, WALL, OPEN = 0, 1, 2
C9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def ring(tw, th):
    """Local coordinates of the nodes around a tw x th tile, first ring first."""
    out = []
    for d in (1, 2):
        w, h = tw + 2 * d, th + 2 * (d - 1)
        out += [(k - d, -d) for k in range(w)]
        out += [(k - d, th + d - 1) for k in range(w)]
        out += [(-d, k - (d - 1)) for k in range(h)]
        out += [(tw + d - 1, k - (d - 1)) for k in range(h)]
    return out


def pull_source(x, y, i, nx, ny, flow):
    """(source node, direction) of f_i(x, y, t+1): Eq. 6 with halfway
    bounce-back walls and zero-gradient open edges (flow: W, E, S, N)."""
    sx, sy = x - C9[i][0], y - C9[i][1]
    if not 0 <= sy < ny and flow[2 if sy < 0 else 3] == WALL:
        return (x, y), OPP[i]
    if not 0 <= sx < nx:
        sx = sx % nx if flow[0] == PERIODIC else x
    if not 0 <= sy < ny:
        sy = sy % ny if flow[2] == PERIODIC else y
    return (sx, sy), i


@pytest.mark.parametrize("tx,ty", [(32, 8), (8, 4), (4, 4), (16, 5), (20, 14)])
@pytest.mark.parametrize("fx", [PERIODIC, OPEN])
@pytest.mark.parametrize("fy", [(PERIODIC, PERIODIC), (WALL, WALL), (WALL, OPEN), (OPEN, OPEN)])
@pytest.mark.parametrize("nx,ny", [(33, 9), (2, 2), (7, 23), (40, 16), (21, 15)])
def test_tile_step_reads_what_was_written_and_writes_once(tx, ty, fx, fy, nx, ny):
    perx, pery = fx == PERIODIC, fy[0] == PERIODIC
    flow = (fx, fx, fy[0], fy[1])
    W2, W1 = tx + 4, tx + 2
    N2, N1 = W2 * (ty + 4), W1 * (ty + 2)
    threads = (max(tx * ty, 2 * (tx + ty) + 4) + 31) // 32 * 32
    writes = {}

    def put(x, y, i, src):
        assert 0 <= x < nx and 0 <= y < ny
        assert (x, y, i) not in writes
        writes[(x, y, i)] = src

    for y0, x0 in itertools.product(range(0, ny, ty), range(0, nx, tx)):
        tw, th = min(tx, nx - x0), min(ty, ny - y0)
        r = ring(tw, th)
        n1 = 2 * (tw + th) + 4
        assert n1 <= threads and len(set(r)) == len(r) == n1 + 2 * (tw + th) + 12
        psi, near = {}, {}
        nodes = [(lx, ly, True) for ly in range(th) for lx in range(tw)]
        nodes += [(lx, ly, k < n1) for k, (lx, ly) in enumerate(r)]
        for lx, ly, first_ring in nodes:
            x, y = x0 + lx, y0 + ly
            x = x % nx if perx else x
            y = y % ny if pery else y
            i2 = (ly + 2) * W2 + lx + 2
            if not 0 <= x < nx:
                continue
            if not 0 <= y < ny:
                if (y == -1 and fy[0] == WALL) or (y == ny and fy[1] == WALL):
                    assert 0 <= i2 < N2
                    psi[i2] = ("ghost", x, y)
                continue
            assert 0 <= i2 < N2 and i2 not in psi
            psi[i2] = (x, y)
            if first_ring:
                i1 = (ly + 1) * W1 + lx + 1
                assert 0 <= i1 < N1 and i1 not in near
                near[i1] = (x, y)

        def beyond(x, y):
            """The node whose psi stands for (x, y)."""
            x = x % nx if perx else min(max(x, 0), nx - 1)
            if 0 <= y < ny:
                return (x, y)
            kind = fy[0] if y < 0 else fy[1]
            if kind == WALL:
                return ("ghost", x, y)
            return (x, y % ny if kind == PERIODIC else min(max(y, 0), ny - 1))

        for lx, ly, first_ring in nodes:
            i1, i2 = (ly + 1) * W1 + lx + 1, (ly + 2) * W2 + lx + 2
            if not first_ring or i1 not in near:
                continue
            x, y = near[i1]
            dw, de = (0 if not perx and x == 0 else -1), (0 if not perx and x == nx - 1 else 1)
            ds = 0 if fy[0] == OPEN and y == 0 else -W2
            dn = 0 if fy[1] == OPEN and y == ny - 1 else W2
            for (ox, cx), (oy, cy) in itertools.product(((dw, -1), (0, 0), (de, 1)),
                                                        ((ds, -1), (0, 0), (dn, 1))):
                assert psi[i2 + ox + oy] == beyond(x + cx, y + cy)
        for ly, lx in itertools.product(range(th), range(tw)):
            c1 = (ly + 1) * W1 + lx + 1
            x, y = x0 + lx, y0 + ly
            eW, eE, eS, eN = x == 0, x == nx - 1, y == 0, y == ny - 1
            # velocities and destinations of the thermal blend
            vd, vu = pery or not eS, pery or not eN
            rows = [0]
            if vd or fy[0] != WALL:
                rows.append(-W1 if vd else 0)
            if vu or fy[1] != WALL:
                rows.append(W1 if vu else 0)
            for row in rows:
                for col in ((0 if not perx and eW else -1), 0, (0 if not perx and eE else 1)):
                    assert c1 + row + col in near
            # the pushes
            oW, oE = (nx - 1 if eW else -1), (1 - nx if eE else 1)
            oS, oN = (ny - 1 if eS else -1), (1 - ny if eN else 1)
            for i, (cx, cy) in enumerate(C9):
                hasW, hasE = perx or not eW, perx or not eE
                hasS, hasN = pery or not eS, pery or not eN
                out_y = (not hasN) if cy > 0 else ((not hasS) if cy < 0 else False)
                if out_y and (fy[1] if cy > 0 else fy[0]) == WALL:
                    put(x, y, OPP[i], ((x, y), i))
                    continue
                xs, ys = [], []
                if cx == 0 or (hasE if cx > 0 else hasW):
                    xs.append(x + (0 if cx == 0 else (oE if cx > 0 else oW)))
                if cx != 0 and not perx and (eW if cx > 0 else eE):
                    xs.append(x)
                if not out_y:
                    ys.append(y + (0 if cy == 0 else (oN if cy > 0 else oS)))
                if (cy > 0 and eS and fy[0] == OPEN) or (cy < 0 and eN and fy[1] == OPEN):
                    ys.append(y)
                for px, py in itertools.product(xs, ys):
                    put(px, py, i, ((x, y), i))
    assert len(writes) == 9 * nx * ny
    for (x, y, i), src in writes.items():
        assert src == pull_source(x, y, i, nx, ny, flow)
