"""The plane schedule of the marching 3-D step (csrc/lbm3d.cu, no GPU): for
segments, walls and periodic domains, every ring read finds the plane it wants
(no slot was overwritten first), no slot is written in the phase in which
another plane's value is read from it, and every plane of a segment is collided
and blended exactly once.  A ring one slot smaller is caught."""
import itertools

import pytest

RING = {"psi": 3, "u": 3, "ic": 3}


def schedule(z0, z1, nz, walls):
    """(iteration, phase, op, array, plane) of one unit; planes unwrapped."""
    beyond = lambda z: walls and (z < 0 or z >= nz)
    for k in range(z0 - 2, z1 + 3):
        if k <= z1 + 1 and (not beyond(k) or k in (-1, nz)):
            yield k, 1, "w", "psi", k
        q = k - 3
        if z0 <= q < z1:
            for dz in (-1, 0, 1):
                if not beyond(q + dz):
                    yield k, 1, "r", "u", q + dz
                    yield k, 1, "r", "ic", q + dz
            yield k, 1, "g", None, q
        p = k - 1
        if z0 - 1 <= p <= z1 and not beyond(p):
            for dz in (-1, 0, 1):
                yield k, 2, "r", "psi", p + dz
            yield k, 2, "w", "u", p
            yield k, 2, "w", "ic", p
            if z0 <= p < z1:
                yield k, 2, "f", None, p


def check(z0, z1, nz, walls):
    held, done = {a: {} for a in RING}, {"f": [], "g": []}
    for _, group in itertools.groupby(schedule(z0, z1, nz, walls), key=lambda e: e[:2]):
        group = list(group)
        writes = {(a, z % RING[a]): z for _, _, op, a, z in group if op == "w"}
        for _, _, op, a, z in group:
            if op == "r":
                assert held[a].get(z % RING[a]) == z, (a, z)
                assert writes.get((a, z % RING[a]), z) == z, (a, z)
            elif op in done:
                done[op].append(z)
        for (a, slot), z in writes.items():
            held[a][slot] = z
    assert done["f"] == done["g"] == list(range(z0, z1))


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("nz,zseg", [(1, 1), (2, 1), (2, 2), (7, 3), (61, 5), (70, 32), (256, 32)])
def test_every_read_finds_its_plane(nz, zseg, walls):
    if walls and nz < 2:
        pytest.skip("walls need two planes")
    for z0 in range(0, nz, zseg):
        check(z0, min(nz, z0 + zseg), nz, walls)


@pytest.mark.parametrize("ring", sorted(RING))
def test_a_smaller_ring_is_caught(ring, monkeypatch):
    monkeypatch.setitem(RING, ring, RING[ring] - 1)
    with pytest.raises(AssertionError):
        check(0, 16, 16, False)
