"""CPU model of the ring exchange of lattices kept on the chip (csrc/lbm_resident.cuh).

Each tile receives its ring through an inbox whose entries the tiles around it send.  For
random cuts of random lattices under every non-periodic boundary set: each entry a tile
expects is sent exactly once, by the tile that holds the value, and together with the
tile's own nodes and ghosts the entries cover every value that its pulls and its ring's
moments read.
"""
import random

import pytest

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1, 1, 0, -1, 0)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1, 0, 1, 0, -1)
FLAT, UP, DOWN = (1, 3, 9, 11), (2, 5, 6, 10), (4, 7, 8, 12)
WEST, EAST = (5, 8, 1, 9, 2, 4, 5, 8), (6, 7, 3, 11, 2, 4, 6, 7)
CORNERS, SEND_MAX = 32, 96


class Tile:
    def __init__(self, nx, nr, ns, nb, t):
        self.ts, self.tb = t % ns, t // ns
        self.x0, self.j0 = nx * self.ts // ns, nr * self.tb // nb
        self.w, self.h = nx * (self.ts + 1) // ns - self.x0, nr * (self.tb + 1) // nb - self.j0
        self.below, self.above = self.j0 > 0, self.j0 + self.h < nr
        self.left, self.right = self.x0 > 0, self.x0 + self.w < nx

    def has(self, i, j):
        return self.x0 <= i < self.x0 + self.w and self.j0 <= j < self.j0 + self.h


def corner(a, e):
    """Entry e of the corners: (population, row, column), or None if unused (res_corner)."""
    if e < 24:
        m, east, north = e % 6, (e // 6) & 1, e >= 12
        side, end = a.right if east else a.left, a.above if north else a.below
        r = a.h + (m == 5) if north else -1 - (m == 5)
        c = a.w + (m == 4) if east else -1 - (m == 4)
        q = {1: 4 if north else 2, 2: 3 if east else 1, 3: 11 if east else 9}.get(
            m, (7 if east else 8) if north else (6 if east else 5))
        used = side or end if m == 0 else (side if m in (1, 4) else end)
        return (q, r, c) if used else None
    m = e - 24
    if m >= 6:
        return None
    q = (6, 5, 7, 8, 7, 6)[m]
    if m < 4:
        used = (a.right if m & 1 else a.left) and not (a.below if m < 2 else a.above)
        return (q, -1 if m < 2 else a.h, a.w - 1 if m & 1 else 0) if used else None
    used = not a.right and (a.below if m == 4 else a.above)
    return (q, 0 if m == 4 else a.h - 1, a.w) if used else None


def writer(bc, nx, nr, q, i, j):
    """The node whose collision or boundary rule writes population q of cell (i, j) (res_writer)."""
    wi, wj = i, j
    if j < 0 and bc["bottom"] == "wall":
        wi += {5: 1, 6: -1}.get(q, 0)
    if j >= nr and bc["top"] == "wall":
        wi += {7: -1, 8: 1}.get(q, 0)
    if i >= nx and bc["out"] == "wall":
        wj += {6: 1, 7: -1}.get(q, 0)
    return min(max(wi, 0), nx - 1), min(max(wj, 0), nr - 1)


def sends(tiles, n, nx, nr, ns, nb, bc, W, TH):
    """(tile, entry, population, cell) of everything tile n sends (res_send, res_lists)."""
    a, cols = tiles[n], 24 * W
    for r in range(a.h):
        down, up = a.below and r <= 1, a.above and r >= a.h - 2
        flat_down, flat_up = a.below and r == 0, a.above and r == a.h - 1
        for c in range(a.w):
            cell = (a.x0 + c, a.j0 + r)
            for k in range(4):
                if flat_down or flat_up:
                    yield n - ns if flat_down else n + ns, (12 * W if flat_down else 0) + c + k * W, FLAT[k], cell
                if down:
                    yield n - ns, (16 if r == 0 else 20) * W + c + k * W, DOWN[k], cell
                if up:
                    yield n + ns, (4 if r == a.h - 1 else 8) * W + c + k * W, UP[k], cell
        for k in range(8):
            if a.left:
                yield n - 1, cols + (8 + k) * TH + r, EAST[k], (a.x0 + (k >= 6), a.j0 + r)
            if a.right:
                yield n + 1, cols + k * TH + r, WEST[k], (a.x0 + a.w - 1 - (k >= 6), a.j0 + r)
    count = 0
    for d in range(9):
        s, b = a.ts + d % 3 - 1, a.tb + d // 3 - 1
        if d == 4 or not (0 <= s < ns and 0 <= b < nb):
            continue
        o = tiles[b * ns + s]
        for e in range(CORNERS):
            x = corner(o, e)
            if x and a.has(*writer(bc, nx, nr, x[0], o.x0 + x[2], o.j0 + x[1])):
                cell = (o.x0 + x[2], o.j0 + x[1])
                assert -1 <= cell[0] - a.x0 <= a.w and -1 <= cell[1] - a.j0 <= a.h  # in the sender's ring
                count += 1
                yield b * ns + s, cols + 16 * TH + e, x[0], cell
    assert count <= SEND_MAX


def receives(a, nx, nr, bc, W, TH):
    """(entry, population, row, column) of everything the tile expects (res_lists)."""
    for n in range(24):
        u = n >> 2
        q = (FLAT if u in (0, 3) else (UP if u < 3 else DOWN))[n & 3]
        r = (-2 if u == 2 else -1) if u < 3 else (a.h + 1 if u == 5 else a.h)
        if a.below if u < 3 else a.above:
            for c in range(a.w):
                yield n * W + c, q, r, c
    for n in range(16):
        c = (-1 if n < 6 else -2) if n < 8 else (a.w if n < 14 else a.w + 1)
        if a.left if n < 8 else a.right:
            for r in range(a.h):
                yield 24 * W + n * TH + r, (WEST + EAST)[n], r, c
    for e in range(CORNERS):
        x = corner(a, e)
        if x and not a.has(*writer(bc, nx, nr, x[0], a.x0 + x[2], a.j0 + x[1])):
            yield 24 * W + 16 * TH + e, *x


@pytest.mark.parametrize("out", ["outflow", "wall"])
@pytest.mark.parametrize("top", ["wall", "open"])
@pytest.mark.parametrize("bottom", ["axis", "wall"])
def test_every_ring_value_is_sent_once_by_its_holder(bottom, top, out):
    rng = random.Random(f"{bottom} {top} {out}")
    bc = dict(bottom=bottom, top=top, out=out)
    for _ in range(10):
        W, TH = rng.choice([(8, 8), (8, 16), (6, 16)])
        ns, nb = rng.randint(1, 4), rng.randint(1, 4)
        nx = rng.randint(2 * ns if ns > 1 else 1, W * ns)
        nr = rng.randint(2 * nb if nb > 1 else 1, min(TH, 9) * nb)
        tiles = [Tile(nx, nr, ns, nb, t) for t in range(ns * nb)]
        inbox = {}
        for n in range(len(tiles)):
            for t, e, q, cell in sends(tiles, n, nx, nr, ns, nb, bc, W, TH):
                assert (t, e) not in inbox
                inbox[t, e] = (q, cell)
        for n, a in enumerate(tiles):
            got = set()
            for e, q, r, c in receives(a, nx, nr, bc, W, TH):
                assert inbox.pop((n, e)) == (q, (a.x0 + c, a.j0 + r))
                got.add((q, r, c))

            def pulls(r, c, qs):
                for q in qs:
                    rr, cc = r - EY[q], c - EX[q]
                    if not (0 <= rr < a.h and 0 <= cc < a.w):
                        own = a.has(*writer(bc, nx, nr, q, a.x0 + cc, a.j0 + rr))
                        assert own or (q, rr, cc) in got, (nx, nr, ns, nb, n, r, c, q)

            for r in range(a.h):
                for c in range(a.w):
                    pulls(r, c, range(13))
                for c, beside in ((-1, a.left), (a.w, a.right)):  # rho u_r beside the tile
                    if beside:
                        pulls(r, c, (2, 4, 5, 6, 7, 8))
            for r, beside in ((-1, a.below), (a.h, a.above)):  # the moments of the rows beside it
                if beside:
                    for c in range(a.w):
                        pulls(r, c, range(1, 13))
        assert not inbox  # nothing is sent that no tile expects
